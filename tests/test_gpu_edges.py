"""Edges of the phase-space and unweighting kernels and of the binding's stream:
outputs that are not 16-byte aligned, tiles and groups of tiles that end between
events, dense and sparse tiles, the current stream inside a graph capture.

Every comparison is exact: the same arithmetic in another place (phase space,
stream), or whole numbers (unweighting, against torch's own comparison)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2303_18244_gb300 import mg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n", [1, 127, 128, 129, 1000])
@pytest.mark.parametrize("proc,sqrts", [("e+ e- > mu+ mu-", 500.0), ("g g > t t~", 1000.0), ("g g > t t~ g", 1200.0),
                                        ("g g > t t~ g g", 1500.0), ("g g > t t~ g g g", 2000.0)])
def test_phase_space_at_any_alignment(proc, sqrts, n):
    h = mg.Process(proc)
    npar = h.info.npar
    want = torch.empty((n, npar, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, sqrts, 7, 11, want)
    buf = torch.full((n * npar * 4 + 2,), -1.0, dtype=torch.float64, device="cuda")
    got = buf[1:-1].view(n, npar, 4)  # 8 bytes past a 16-byte boundary
    mg.rambo(h, sqrts, 7, 11, got)
    assert torch.equal(got, want)
    assert float(buf[0]) == -1.0 and float(buf[-1]) == -1.0


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 16 * 4096 - 1, 16 * 4096, 16 * 4096 + 1, 33 * 4096 + 77])
@pytest.mark.parametrize("kept", [0.0, 0.01, 0.124, 0.126, 0.7, 1.0])
def test_unweighting_around_tiles(n, kept):
    """A tile of 4096 events writes its indices lane by lane up to 512 kept ones
    and word by word beyond; a block writes 16 tiles."""
    g = torch.Generator(device="cuda").manual_seed(n)
    r = torch.rand((n,), dtype=torch.float64, device="cuda", generator=g)
    w = torch.full((n,), kept, dtype=torch.float64, device="cuda")
    idx = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    mg.unweight(w, r, 1.0, idx, cnt)
    want = torch.nonzero(r < w).flatten()
    assert int(cnt) == want.numel()
    assert torch.equal(idx[:want.numel()], want)
    assert bool((idx[want.numel():] == -1).all())


@pytest.mark.parametrize("proc,sqrts", [("g g > t t~", 1000.0), ("g g > t t~ g g", 1500.0)])
def test_current_stream_is_used_inside_a_capture(proc, sqrts):
    h = mg.Process(proc, precision=mg.MG_MIXED)
    mom = torch.empty((300, h.info.npar, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, sqrts, 5, 0, mom)
    want = torch.empty(300, dtype=torch.float64, device="cuda")
    mg.sigma(h, mom, want)
    got = torch.zeros_like(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mg.sigma(h, mom, got)  # on the capturing stream: recorded, not run
    torch.cuda.synchronize()
    assert bool((got == 0).all())
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, want)

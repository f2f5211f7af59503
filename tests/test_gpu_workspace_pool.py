"""The memory that the two-phase path keeps between calls: one workspace per
device, however many handles, given back with the last of them."""
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_2303_18244_gb300 import mg  # noqa: E402

pytestmark = pytest.mark.gpu

PROC, N = "g g > t t~ g g g", 8704  # a full workspace: 1 GiB
GIB, SLACK = 1 << 30, 128 << 20     # slack: granularity of the pools, the contexts' own growth


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_handles_keep_one_workspace_and_give_it_back():
    hs = [mg.Process(PROC, precision=mg.MG_MIXED, alpha_s=0.1 + 0.01 * k) for k in range(3)]
    mom = torch.empty((N, 7, 4), dtype=torch.float64, device="cuda")
    mg.rambo(hs[0], 2000.0, 3, 0, mom)
    out = torch.empty(N, dtype=torch.float64, device="cuda")
    mg.sigma(hs[0], mom, out, nevt=1)  # modules are loaded
    before = _free()
    for h in hs:
        mg.sigma(h, mom, out)
        _free()
    assert before - _free() <= GIB + SLACK
    for h in hs[1:]:
        h.close()
    want = out.clone()
    mg.sigma(hs[0], mom, want)  # the pool outlives its other handles
    assert bool(torch.isfinite(want).all())
    hs[0].close()
    assert before - _free() <= SLACK
    h = mg.Process(PROC, precision=mg.MG_MIXED, alpha_s=0.1)  # and is made anew
    mg.sigma(h, mom, out)
    assert torch.equal(out, want)


def test_threads_and_streams_share_the_pool():
    """Calls of two handles from two threads on streams of their own, handles
    made and destroyed meanwhile: each call's values are those of a call alone."""
    n = 1500
    mom = torch.empty((n, 7, 4), dtype=torch.float64, device="cuda")
    alone = []
    for k in range(2):
        h = mg.Process(PROC, precision=mg.MG_MIXED, alpha_s=0.1 + 0.05 * k)
        mg.rambo(h, 2000.0, 3, 0, mom)
        alone.append(torch.empty(n, dtype=torch.float64, device="cuda"))
        mg.sigma(h, mom, alone[-1])
        torch.cuda.synchronize()
        h.close()
    ok = [False, False]

    def work(k):
        s = torch.cuda.Stream()
        good = True
        for _ in range(4):
            h = mg.Process(PROC, precision=mg.MG_MIXED, alpha_s=0.1 + 0.05 * k)
            got = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(5)]
            torch.cuda.current_stream().synchronize()
            for g in got:
                mg.sigma(h, mom, g, stream=s)
            s.synchronize()
            good &= all(torch.equal(g, alone[k]) for g in got)
            h.close()
        ok[k] = good

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert ok == [True, True]

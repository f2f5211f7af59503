"""A kernel that may start before its predecessor has finished (programmatic
stream serialisation) reads what that kernel writes only after
griddepcontrol.wait, through pointers that do not promise read-only memory."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2303_18244_gb300" / "csrc"


def _early_kernels():
    """(file, parameter list, body) of every __global__ function with a griddepcontrol.wait."""
    for f in sorted(CSRC.glob("*.cu*")):
        text = re.sub(r"//[^\n]*", "", f.read_text())
        starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
        for a, b in zip(starts, starts[1:]):
            fn = text[a:b]
            if "griddepcontrol.wait" in fn:
                m = re.search(r"\w+_kernel\((.*?)\)\s*\{", fn, re.S)
                yield f.name, m.group(1), fn[m.end():]


def test_early_kernels_promise_no_read_only_inputs():
    found = list(_early_kernels())
    assert found
    for name, params, body in found:
        for p in params.split(","):
            assert not ("*" in p and "const" in p and "__restrict__" in p), (name, p.strip())
        assert "__ldg(" not in body and "__ldcs(" not in body, name


@pytest.mark.gpu
def test_back_to_back_calls_read_their_own_pass():
    """Calls in a row on one stream reuse one workspace, whose former contents
    are another call's bits and counts; each call's kept set is exact."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_18244_gb300 import mg
    g = torch.Generator(device="cuda").manual_seed(5)
    calls = []
    for q in range(24):
        n = (1 << 20) + 4096 * (q % 3) + 17 * q
        r = torch.rand((n,), dtype=torch.float64, device="cuda", generator=g)
        w = torch.full((n,), (0.02, 0.9, 0.3)[q % 3], dtype=torch.float64, device="cuda")
        idx = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        cnt = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        calls.append((w, r, idx, cnt))
    torch.cuda.synchronize()
    for w, r, idx, cnt in calls:
        mg.unweight(w, r, 1.0, idx, cnt)
    torch.cuda.synchronize()
    for w, r, idx, cnt in calls:
        want = torch.nonzero(r < w).flatten()
        assert int(cnt) == want.numel()
        assert torch.equal(idx[:want.numel()], want)
        assert bool((idx[want.numel():] == -1).all())


@pytest.mark.gpu
def test_unweighting_in_a_captured_graph():
    """The early launch and the stream-ordered workspace inside a CUDA graph:
    replays on other inputs in the same buffers give their own kept sets."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2303_18244_gb300 import mg
    n = 40 * 4096 + 77
    g = torch.Generator(device="cuda").manual_seed(8)
    r = torch.rand((n,), dtype=torch.float64, device="cuda", generator=g)
    w = torch.full((n,), 0.5, dtype=torch.float64, device="cuda")
    idx = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    mg.unweight(w, r, 1.0, idx, cnt)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mg.unweight(w, r, 1.0, idx, cnt)
    for kept in (0.02, 0.9, 0.3):
        w.fill_(kept)
        idx.fill_(-1)
        graph.replay()
        want = torch.nonzero(r < w).flatten()
        assert int(cnt) == want.numel()
        assert torch.equal(idx[:want.numel()], want)
        assert bool((idx[want.numel():] == -1).all())

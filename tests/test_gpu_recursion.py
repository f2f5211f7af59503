"""Tiles of the recursion kernels: a CTA works on up to EV events side by side
(and on fewer per tile when the batch does not fill the SMs), so the sizes
around a tile, one event, and batches of several waves of tiles with a ragged
end can go wrong.

Every thread does the same arithmetic for an event wherever it sits in a batch,
so each value must be bit-identical to the one in a larger batch (tolerance
0), and that batch is checked against the oracle (1e-12 in FP64 by the parity
tests' rule, the mixed bounds in FP32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_2303_18244_gb300 import mg  # noqa: E402
from paper_2303_18244_gb300.inputs import process_momenta  # noqa: E402
from mixed_bounds import check_mixed  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [("g g > t t~", 1000.0, mg.MG_FP64, 3000), ("g g > t t~ g", 1200.0, mg.MG_FP64, 3000),
         ("g g > t t~ g", 1200.0, mg.MG_MIXED, 6000), ("g g > t t~ g g", 1500.0, mg.MG_FP64, 1500),
         ("g g > t t~ g g", 1500.0, mg.MG_MIXED, 4000), ("g g > t t~ g g g", 2000.0, mg.MG_FP64, 330),
         ("g g > t t~ g g g", 2000.0, mg.MG_MIXED, 700)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _me(h, mom, n, first=0):
    out = torch.full((n + 2,), -1.0, dtype=torch.float64, device="cuda")
    mg.sigma(h, mom[first:first + n].contiguous(), out, nevt=n)
    torch.cuda.synchronize()
    assert mg.process_status(h) == 0
    assert bool((out[n:] == -1.0).all())  # nothing written past the batch
    return out[:n]


@pytest.mark.parametrize("proc,sqrts,precision,n", CASES,
                         ids=["ggtt-fp64", "ggttg-fp64", "ggttg-mixed", "ggttgg-fp64", "ggttgg-mixed", "ggttggg-fp64",
                              "ggttggg-mixed"])
def test_every_batch_size_gives_the_same_values(proc, sqrts, precision, n):
    p = process_momenta(proc, sqrts, n, 67)
    mom = torch.from_numpy(p).cuda()
    h = mg.Process(proc, precision=precision)
    full = _me(h, mom, n)
    k = 24 if "g g g" in proc else 64
    pick = np.unique(np.concatenate([[0, n - 1], np.random.default_rng(5).integers(0, n, k)]))
    ref = O.me(proc, p[pick])
    r = np.abs(full[torch.from_numpy(pick).cuda()].cpu().numpy() / ref - 1)
    if precision == mg.MG_FP64:
        bad = np.nonzero(r > 1e-12)[0]
        if bad.size:
            got = full[torch.from_numpy(pick[bad]).cuda()].cpu().numpy()
            r[bad] = np.abs(got / O.me(proc, p[pick[bad]], extended=True) - 1)
        assert r.max() <= 1e-12
    else:
        check_mixed(proc, r)
    for m, first in [(1, 7), (2, 0), (3, 5), (4, 11), (5, 2), (11, 1), (12, 3), (13, 0), (25, 9), (153, 20), (305, 13)]:
        assert torch.equal(_me(h, mom, m, first), full[first:first + m]), (m, first)

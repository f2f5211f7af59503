"""A helicity list that leaves out states which matter: every mode sums, and
chooses from, exactly the listed ones.

The list comes from calibration events at 1e14 GeV, where the top is massless
and its helicity-flip states vanish; the calls are at ordinary energies, where
those states contribute.  Bounds are those of the modes' parity tests, relative
to the sum over all helicities, whose terms the same amplitudes give: 1e-12 in
FP64, the mixed bounds, the paper and float modes' bounds.  Batches of other
sizes repeat the same arithmetic event by event: bit-identical."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2303_18244_gb300 import mg  # noqa: E402
from mixed_bounds import check_mixed  # noqa: E402

pytestmark = pytest.mark.gpu

PROCS = [("g g > t t~", 1000.0), ("g g > t t~ g", 1200.0), ("g g > t t~ g g", 1500.0), ("g g > t t~ g g g", 2000.0),
         ("u u~ > t t~ g", 1200.0)]
IDS = ["ggtt", "ggttg", "ggttgg", "ggttggg", "uuttg"]
N = 613


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _momenta(h, sqrts, n, seed):
    mom = torch.empty((n, h.info.npar, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, sqrts, seed, 0, mom)
    return mom


def _handle(proc, precision):
    h = mg.Process(proc, precision=precision)
    listed, mask = mg.good_helicities(h, _momenta(h, 1e14, 512, 31))
    assert 0 < listed < 0.8 * h.info.n_hel
    return h, torch.from_numpy(mask).cuda().bool()


def _sigma(h, mom):
    out = torch.empty(mom.shape[0], dtype=torch.float64, device="cuda")
    mg.sigma(h, mom, out)
    return out


def _per_helicity(h, mom):
    per = torch.empty((mom.shape[0], h.info.n_hel), dtype=torch.float64, device="cuda")
    mg.sigma_helicities(h, mom, per)
    return per


@pytest.mark.parametrize("precision", [mg.MG_FP64, mg.MG_MIXED, mg.MG_FLOAT, mg.MG_MIXED_PAPER],
                         ids=["fp64", "mixed", "float", "paper"])
@pytest.mark.parametrize("proc,sqrts", PROCS, ids=IDS)
def test_sum_over_the_list(proc, sqrts, precision):
    h, mask = _handle(proc, precision)
    mom = _momenta(h, sqrts, N, 41)
    per = _per_helicity(h, mom)
    want, full = per[:, mask].sum(1), per.sum(1)
    assert float((1 - want / full).median()) > 0.01  # what the list leaves out is seen
    got = _sigma(h, mom)
    r = ((got - want).abs() / full).cpu().numpy()
    if precision == mg.MG_FP64:
        assert r.max() <= 1e-12
    elif precision == mg.MG_MIXED:
        check_mixed(proc, r)
    elif precision == mg.MG_FLOAT:
        assert np.median(r) <= 1e-5 and np.quantile(r, 0.99) <= 1e-3 and r.max() <= 5e-2
    else:
        assert np.median(r) <= 1e-6 and r.max() <= 1e-4
    for n, first in ((1, 0), (3, 7), (12, 1), (13, 100), (305, 300)):
        part = mom[first:first + n].contiguous()
        assert torch.equal(_sigma(h, part), got[first:first + n])
        assert torch.equal(_per_helicity(h, part), per[first:first + n])
    assert mg.process_status(h) == 0


@pytest.mark.parametrize("proc,sqrts", PROCS, ids=IDS)
def test_choice_from_the_list(proc, sqrts):
    h, mask = _handle(proc, mg.MG_FP64)
    mom = _momenta(h, sqrts, N, 43)
    rnd = torch.rand((N, 2), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))

    def select(h, mom, rnd):
        n = mom.shape[0]
        me = torch.empty(n, dtype=torch.float64, device="cuda")
        hel, col = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
        w = torch.empty((n, h.info.n_col), dtype=torch.float64, device="cuda")
        mg.sigma_select(h, mom, rnd, me, hel, col, w)
        return me, hel, col, w

    me, hel, col, w = select(h, mom, rnd)
    per = _per_helicity(h, mom)
    listed = per[:, mask]
    assert float(((me - listed.sum(1)).abs() / per.sum(1)).max()) <= 1e-12
    for weights, index, chosen, r in ((listed, torch.nonzero(mask).flatten(), hel, rnd[:, 0]),
                                      (w, torch.arange(w.shape[1], device="cuda"), col, rnd[:, 1])):
        cum = weights.cumsum(1)
        th = (r * cum[:, -1])[:, None]
        want = index[((cum > th) & (weights > 0)).int().argmax(1)]
        clear = (cum - th).abs().min(1).values > 1e-12 * cum[:, -1]
        assert int(clear.sum()) > 0.9 * N
        assert torch.equal(chosen.long()[clear], want[clear])
    # the flow weights of the FP32 selection, another program (per helicity):
    # FP32 amplitudes, 1e-3 as the largest of the mixed bounds
    hm, _ = _handle(proc, mg.MG_MIXED)
    wm = select(hm, mom, rnd)[3]
    scale = w.sum(1, keepdim=True)
    assert float(((wm / wm.sum(1, keepdim=True) - w / scale).abs()).max()) <= 1e-3
    for n, first in ((1, 0), (3, 7), (13, 100), (305, 300)):
        part = select(h, mom[first:first + n].contiguous(), rnd[first:first + n].contiguous())
        for a, b in zip(part, (me, hel, col, w)):
            assert torch.equal(a, b[first:first + n])

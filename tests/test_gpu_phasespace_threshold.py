"""Phase space close to the production threshold of the top pair, where sqrt_s
and the masses cancel to a few digits (mg_rambo)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2303_18244_gb300 import mg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _events(proc, sqrts, n=4000):
    h = mg.Process(proc)
    mom = torch.empty((n, h.info.npar, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, sqrts, 19, 0, mom)
    return mom.cpu()


@pytest.mark.parametrize("above", [1e-10, 1e-12])
@pytest.mark.parametrize("proc", ["g g > t t~ g", "g g > t t~ g g", "g g > t t~ g g g"], ids=["1g", "2g", "3g"])
def test_gluons_take_the_energy_above_threshold(proc, above):
    """sqrt_s = 2 m_t (1 + d) leaves T = 346 d GeV (exact: sqrt_s - 346) to the
    tops' kinetic energies and the gluons.  Where the kinetic part is at most
    1e-9 T = 3e-17 GeV it is far below the spacing of doubles at m_t: the
    computed energies of the tops are m_t, the residual of the mass-shell
    equation is exact, and the gluons' energies add up to T but for that 1e-9
    and the rounding of the map (1e-15); bound 1e-8."""
    sqrts = 346.0 * (1.0 + above)
    gap = sqrts - 346.0
    p = _events(proc, sqrts)
    assert bool((p[:, 4:, 0] > 0).all())
    kinetic = (p[:, 2:4, 1:] ** 2).sum((1, 2)) / 346.0
    at_rest = kinetic <= 1e-9 * gap
    assert int(at_rest.sum()) >= 1000
    assert float((p[at_rest, 4:, 0].sum(1) / gap - 1).abs().max()) <= 1e-8


@pytest.mark.parametrize("proc,sqrts", [("e+ e- > mu+ mu-", 500.1), ("g g > t t~", 346.0 * (1 + 1e-9)),
                                        ("g g > t t~", 1000.3), ("u u~ > t t~", 1e10)])
def test_two_equal_masses_share_the_energy(proc, sqrts):
    p = _events(proc, sqrts)
    assert bool((p[:, 2:, 0] == 0.5 * sqrts).all())


@pytest.mark.parametrize("sqrts", [1e-200, 1e-40, 1e40, 1e200])
def test_any_scale_of_energies(sqrts):
    """The map only scales with sqrt_s for massless final states: the momenta at
    sqrt_s 2^k are those at sqrt_s times 2^k, bit for bit."""
    import math
    e = 2.0 ** round(math.log2(sqrts / 500.0))
    assert torch.equal(_events("e+ e- > mu+ mu-", 500.0 * e), _events("e+ e- > mu+ mu-", 500.0) * e)

"""The workspace of the two-phase mixed g g > t t~ g g g path is counted in
events: the same for every helicity list, bounded for every batch."""
import pytest

torch = pytest.importorskip("torch")

from paper_2303_18244_gb300 import mg  # noqa: E402

pytestmark = pytest.mark.gpu

PROC = "g g > t t~ g g g"


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_workspace_does_not_follow_the_helicity_list():
    """At 1e14 GeV the top is massless to FP64 accuracy and most helicity
    states drop out of the list; a call keeps its workspace and its slices."""
    h = mg.Process(PROC, precision=mg.MG_MIXED)
    sizes = (1, 128, 129, 8704, 8705, 20000, 1 << 20, 2_000_000, 10_000_000)
    want = [mg.sigma_workspace_bytes(h, n) for n in sizes]
    mom = torch.empty((1024, 7, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, 1e14, 3, 0, mom)
    listed, _ = mg.good_helicities(h, mom)
    assert 0 < listed < 100
    assert [mg.sigma_workspace_bytes(h, n) for n in sizes] == want
    row = 120 * 128 * 8
    for n, b in zip(sizes, want):
        assert b % row == 0 and row <= b <= 1 << 30
        assert b == min((n + 127) // 128 * 128, (1 << 30) // (128 * row) * 128) * row
    mg.rambo(h, 2000.0, 3, 0, mom)
    out = torch.empty(1024, dtype=torch.float64, device="cuda")
    assert mg.diag_sigma_phases(h, mom, out)[2] == 1


def test_slices_give_the_values_of_one_slice():
    """Values around the first slice's end are those of a batch of their own."""
    h = mg.Process(PROC, precision=mg.MG_MIXED)
    n = 2 * 8704 + 5
    mom = torch.empty((n, 7, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, 2000.0, 5, 0, mom)
    got, own = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(40, dtype=torch.float64, device="cuda")
    assert mg.diag_sigma_phases(h, mom, got)[2] == 3
    for a in (0, 8704 - 20, 2 * 8704 - 35):
        mg.sigma(h, mom[a:a + 40], own)
        assert torch.equal(own, got[a:a + 40])

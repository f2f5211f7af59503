"""The mixed mode adds the FP32 |M|^2 of the helicities in FP64: a sum beyond
the FP32 range, of terms inside it, is finite and right."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2303_18244_gb300 import mg  # noqa: E402
from paper_2303_18244_gb300.generator.colour import colour_matrix_exact, common_denominator  # noqa: E402

pytestmark = pytest.mark.gpu

FP32_MAX = float(np.finfo(np.float32).max)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("proc,sqrts,ngluon,part", [("g g > t t~", 1000.0, 2, 4), ("g g > t t~ g", 1200.0, 3, 8),
                                                    ("g g > t t~ g g", 1500.0, 4, 8)], ids=["ggtt", "ggttg", "ggttgg"])
def test_sum_beyond_the_fp32_range(proc, sqrts, ngluon, part):
    """|M|^2 grows as alpha_s^n for n gluons; alpha_s puts the largest term of
    the event whose terms are the most even at 1 / part of the FP32 range."""
    h = mg.Process(proc)
    n = 4096
    mom = torch.empty((n, h.info.npar, 4), dtype=torch.float64, device="cuda")
    mg.rambo(h, sqrts, 23, 0, mom)
    hel = torch.empty((n, h.info.n_hel), dtype=torch.float64, device="cuda")
    mg.sigma_helicities(h, mom, hel)
    hel *= h.info.iden * common_denominator(colour_matrix_exact(ngluon))[0]  # the kernels' terms
    even = hel.sum(1) / hel.max(1).values
    i = int(even.argmax())
    assert float(even[i]) > part + 0.5  # the sum is beyond the range then
    scale = FP32_MAX / part / float(hel[i].max())
    over = {"alpha_s": h.params.alpha_s * scale ** (1.0 / ngluon)}
    event = mom[i:i + 1].contiguous()
    want, got = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
    mg.sigma(mg.Process(proc, **over), event, want)
    mg.sigma(mg.Process(proc, precision=mg.MG_MIXED, **over), event, got)
    assert bool(torch.isfinite(got).all())
    assert float((got / want - 1).abs()) <= 1e-4

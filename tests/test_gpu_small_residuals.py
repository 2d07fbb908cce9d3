"""The structural term of residuals so small that the loss of one sample,
R^2 / (2 eps), is a float32 subnormal while an A-scan's sum is not (GPU only).

Float32 bounds relative to the sum, 1e-5 together: the subnormal grid (two
roundings of at most 2^-150 per sample, mean loss 4e-40 at the smallest
amplitude: 4e-6), the approximate square root, reciprocal and product (5 ulp:
3e-7) and the sums over the depth (at most 25 roundings per lane: 1.5e-6)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 1e-3


@pytest.mark.parametrize("amplitude", [1e-21, 3e-21, 3e-20, 1e-18])
@pytest.mark.parametrize("w,h,d", [(9, 7, 512), (5, 6, 465)])
def test_subnormal_losses_are_summed(w, h, d, amplitude):
    import paper_2010_06931_gb300 as octmc
    rng = np.random.default_rng(w + d)
    s = (amplitude * rng.rayleigh(1.0, (2, h, w, d))).astype(np.float32)
    t = np.arange(w * h, dtype=np.float64).reshape(h, w)
    P = octmc.Problem(s[0], s[1], t, t, eps_h=EPS)
    R = (s[0] - s[1]).astype(np.float64)  # the kernel's float32 residual at zero displacement
    want = (R * R / EPS / (1.0 + np.sqrt(1.0 + (R / EPS) ** 2))).sum()
    # general kernel, then the column kernel of the axial prealignment (its tilt term is 0 here)
    got = P.eval_terms(0, P.zeros(0))[0]
    assert abs(got - want) <= 1e-5 * want, (got, want)
    got = P.prealign_eval(0, torch.zeros(P.prealign_size(0), dtype=torch.float64, device="cuda"))
    assert abs(got - want) <= 1e-5 * want, (got, want)

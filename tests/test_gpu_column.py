"""The prealignment's one-column data kernel against the general data kernel
on the same field (GPU only): without transverse displacement the general
interpolant is the column itself, so the objective is the same float
arithmetic in the same order and must agree bitwise; the parameter gradient
is the general gradient's axial planes summed per B-scan (float64 sums of at
most 40 terms in another order: 1e-12 of the largest magnitude sum)."""
import numpy as np
import pytest

from octsynth import make_pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,d,storage,loss,shift", [
    (9, 7, 1, 0, 0, 0.4), (12, 5, 61, 1, 0, 2.0), (8, 13, 116, 0, 1, 3.0), (17, 9, 117, 2, 0, 140.0),
    (16, 16, 128, 0, 0, 30.0), (23, 11, 233, 1, 1, 0.0), (11, 40, 256, 0, 0, 5.0)])
def test_column_kernel_equals_general_kernel(w, h, d, storage, loss, shift):
    import paper_2010_06931_gb300 as octmc
    p = make_pair(w, h, d, n_layers=4, n_slabs=2, n_saccades=1, max_saccade=2.0, drift_sigma=0.02, seed=w + d)
    kw = dict(storage=storage, loss=loss, delta0=0.0)
    G = octmc.Problem(p["sx"], p["sy"], p["tx"], p["ty"], p["ax"], p["ay"], p["vx"], p["vy"], **kw)
    rng = np.random.default_rng(d)
    prm = np.zeros(2 * (w + h))
    prm[:h] = rng.normal(0.0, 1.0, h) * shift
    prm[2 * h:2 * h + w] = rng.normal(0.0, 1.0, w) * shift
    prm_t = torch.from_numpy(prm).cuda()
    D = G.prealign_disp(0, prm_t)
    gp = torch.zeros_like(prm_t)
    f = G.prealign_eval(0, prm_t, gp)
    grad = torch.empty_like(D)
    assert G.eval_objective_grad(0, D, grad) == f  # no tilts: T = 0
    g = grad.cpu().numpy()
    want = np.concatenate([g[0, 2].sum(1), (g[0, 2] * (np.arange(w) - 0.5 * (w - 1))).sum(1),
                           g[1, 2].sum(0), (g[1, 2] * (np.arange(h) - 0.5 * (h - 1))[:, None]).sum(0)])
    bar = 1e-12 * max(np.abs(g[0, 2]).sum(1).max(), np.abs(g[1, 2]).sum(0).max()) * max(w, h)
    assert np.abs(gp.cpu().numpy() - want).max() <= bar

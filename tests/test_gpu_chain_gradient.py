"""Both directions of the acquisition chains of a new problem (GPU only),
read back through the gradient of the temporal regulariser: an A-scan's
gradient takes its previous and its next neighbour and both weights.  With
empty volumes the data term and its gradient are exactly 0.

Float32 bound per component: two pairs of about 8 ulp each (difference,
quotient, approximate square root, weight, sum) times alpha d, then one ulp of
the whole with its mean term: 1e-6 (2 alpha d + |2 mu S|)."""
import numpy as np
import pytest

from .test_gpu_create import maps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ALPHA, EPS = 0.5, 1e-2


def gradient(D, tx, ty, d):
    _, _, h, w = D.shape
    S = D.sum(axis=(0, 2, 3))
    G = np.zeros(D.shape) + (S / (w * h))[None, :, None, None]  # 2 mu S, mu = 1 / (2 w h)
    for V, t in enumerate((tx, ty)):
        t = t.reshape(-1)
        o = np.lexsort((np.arange(t.size), t))
        dt = np.diff(t[o])
        om = dt[dt > 0].min() / np.maximum(dt, dt[dt > 0].min()) if (dt > 0).any() else np.ones(dt.size)
        for c in range(3):
            x = np.diff(D[V, c].reshape(-1)[o]) / EPS
            dl = ALPHA * d * om * x / np.sqrt(1.0 + x * x)
            g = G[V, c].reshape(-1)
            g[o[1:]] += dl
            g[o[:-1]] -= dl
    return G, np.abs(S / (w * h)).max()


@pytest.mark.parametrize("kind", ["raster", "swapped", "ties", "constant", "reversed", "random"])
@pytest.mark.parametrize("w,h", [(1, 1), (1, 9), (13, 1), (11, 14), (70, 33)])
def test_gradient_of_the_regulariser(kind, w, h):
    import paper_2010_06931_gb300 as octmc
    rng = np.random.default_rng(w * 31 + h)
    d = 4
    tx, ty = maps(kind, w, h, rng)
    s = np.zeros((h, w, d), np.float32)
    P = octmc.Problem(s, s, tx, ty, levels=2, alpha=ALPHA, eps_r=EPS)
    for l in range(2):
        if l:
            pad = lambda t: np.pad(t, [(0, t.shape[0] % 2), (0, t.shape[1] % 2)], mode="edge")
            tx, ty = ((p[0::2, 0::2] + p[0::2, 1::2] + p[1::2, 0::2] + p[1::2, 1::2]) / 4.0 for p in (pad(tx), pad(ty)))
        D = rng.normal(0.0, 0.3, P.disp_shape(l))
        G = torch.full(P.disp_shape(l), 7.0, dtype=torch.float64, device="cuda")
        P.eval_terms(l, torch.from_numpy(D).cuda(), G)
        dl = P.level_shape(l)[2]
        want, mean = gradient(D, tx, ty, dl)
        assert np.abs(G.cpu().numpy() - want).max() <= 1e-6 * (2.0 * ALPHA * dl + mean)

"""The persistent level kernel with several A-scans per warp (GPU only): each
warp fills its interpolation table again for every A-scan, so a field whose
neighbouring A-scans differ everywhere must give the gradient of the kernels
that take one A-scan per warp.

Both solvers run one iteration from the same field.  The gradients are the
same float32 values but for the mean term, whose float64 sums differ in order
(one float32 ulp of it, 1e-9); the first step follows -g with a factor of at
most 1, so the fields agree to 1e-8 px.  A table of another A-scan would move
that A-scan by about its own step (1e-3 px and more)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1, 2])  # f32, bf16, f16
@pytest.mark.parametrize("w,h,d", [(128, 120, 40), (97, 101, 117), (211, 150, 8)])
def test_one_iteration_equals_the_graph_loop(w, h, d, storage):
    import paper_2010_06931_gb300 as octmc
    rng = np.random.default_rng(w + d)
    k = np.arange(d)
    base = 0.2 + 0.6 / (1.0 + np.exp(-(k - 0.5 * d) / 2.0))
    s = (base * (0.5 + rng.random((2, h, w, d)))).astype(np.float32)
    j, i = np.meshgrid(np.arange(h, dtype=np.float64), np.arange(w, dtype=np.float64), indexing="ij")
    img = rng.random((2, h, w)).astype(np.float32)
    D0 = torch.from_numpy(rng.normal(0.0, 1.0, (2, 3, h, w))).cuda()
    out = []
    for ascans in (0, 1 << 20):
        P = octmc.Problem(s[0], s[1], j * w + i, i * h + j, img[0], img[1], storage=storage, max_iter=1,
                          persistent_ascans=ascans)
        D = D0.clone()
        st = P.solve_level(0, D)
        out.append((D, st))
    (Da, a), (Db, b) = out
    assert a["evals"] == b["evals"] and a["iters"] == b["iters"] == 1
    assert abs(a["f"] - b["f"]) <= 1e-9 * abs(a["f"])
    assert float((Da - D0).abs().max()) > 1e-3
    assert float((Da - Db).abs().max()) <= 1e-8

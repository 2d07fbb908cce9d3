"""The projection's filters, sums and selection at the edges of their tiles
(15-sample rank segments, 10-column median strips, 4- and 16-sample loads,
32-depth blocks) against the oracle, with the bounds of the other projection
tests; and the caller-workspace entry point against the allocating one (GPU
only)."""
import ctypes as C

import numpy as np
import pytest

from .test_gpu_octa import check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def scan(h, w, d, fast_axis, kind="plain"):
    rng = np.random.default_rng(h * 7919 + w * 101 + d)
    A, S = rng.random((h, w, d)), rng.random((h, w, d))
    if kind == "ties":  # few distinct values: long runs, equal order statistics
        A, S = np.round(A * 3) / 3, np.round(S * 5) / 5
    elif kind == "wide":  # both signs, magnitudes over 60 binary orders, zeros
        A = np.ldexp(A, rng.integers(-30, 30, A.shape)) * rng.choice([-1.0, 0.0, 1.0], A.shape)
    return dict(A=A.astype(np.float32), S=S.astype(np.float32), fast_axis=fast_axis)


@pytest.mark.parametrize("h,w,d,kind", [
    (14, 15, 31, "plain"), (16, 29, 32, "ties"), (30, 31, 33, "wide"), (7, 81, 20, "plain"), (45, 10, 48, "wide"),
    (9, 11, 130, "ties"), (3, 160, 17, "plain"), (61, 4, 257, "wide")])
@pytest.mark.parametrize("fast_axis", [0, 1])
def test_projection_at_tile_edges(h, w, d, kind, fast_axis):
    v = np.ones(h if fast_axis == 0 else w, np.float32)
    v[:: 3] = 0.0
    # with quantiles that fall in different leading digits the selection follows up to four prefixes
    check(scan(h, w, d, fast_axis, kind), v=v, q_lo=0.02, q_hi=0.97)


def test_validity_means_are_as_exact_as_float64_sums():
    import paper_2010_06931_gb300 as octmc
    sc = scan(12, 70, 512, 0)
    v, m = octmc.saccade_validity(torch.from_numpy(sc["A"]).cuda(), 0)
    want = sc["A"].astype(np.longdouble).mean(axis=(1, 2))
    assert np.abs(m.cpu().numpy() - want).max() <= 4 * 2.0 ** -53 * float(want.max())


def test_caller_workspace_equals_the_allocating_entry_point():
    import paper_2010_06931_gb300 as octmc
    from paper_2010_06931_gb300 import _native as N
    sc = scan(20, 33, 64, 0)
    A, S = torch.from_numpy(sc["A"]).cuda(), torch.from_numpy(sc["S"]).cuda()
    v = torch.ones(20, device="cuda")
    v[4] = 0.0
    E, info = octmc.enface(A, S, 0, v)
    E2 = torch.empty_like(E)
    i2 = (C.c_double * 4)()
    p = lambda t: C.c_void_p(t.data_ptr())
    L = N.lib()
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    args = [p(A), p(S), 33, 20, 64, 0, p(v), 0.05, 0.95, 0.1, float("nan"), p(E2), None, i2]
    assert L.octmc_enface(*args, st) == 0
    assert torch.equal(E, E2)
    assert [info["p_lo"], info["p_hi"], info["t_oct"], info["kept"]] == list(i2)
    need = L.octmc_enface_workspace(33, 20, 64, 0)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    assert L.octmc_enface_ws(*args, p(ws), need - 1, st) == -1
    assert L.octmc_enface_ws(*args, None, need, st) == -1
    assert L.octmc_enface_workspace(0, 20, 64, 0) == -1

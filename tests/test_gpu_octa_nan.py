"""The rank-filtered volume of scans with NaN voxels (GPU only).  A minimum or
maximum of a NaN and a number is the number, so the values depend on the order
of the exchanges; the order is that of the sequential forms below, and the
comparison is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def exchange(a, i, j):
    a[i], a[j] = np.fmin(a[i], a[j]), np.fmax(a[i], a[j])


def shifted(v, o, axis):
    return np.take(v, np.clip(np.arange(v.shape[axis]) + o, 0, v.shape[axis] - 1), axis=axis)


def median(v):
    lo, mid, hi = [], [], []
    for dj in (-1, 0, 1):
        for di in (-1, 0, 1):
            col = shifted(shifted(v, dj, 0), di, 1)
            s = [shifted(col, dk, 2) for dk in (-1, 0, 1)]
            for i, j in ((0, 1), (1, 2), (0, 1)):
                exchange(s, i, j)
            for part, x in zip((lo, mid, hi), s):
                part.append(x)
    for e in (8, 7, 6, 5):
        for i in range(e):
            exchange(lo, i, e)
    for b in range(4):
        for i in range(b + 1, 9):
            exchange(hi, b, i)
    for q in range(2):
        exchange(mid, q, 8 - q)
        for i in range(q + 1, 8 - q):
            exchange(mid, q, i)
            exchange(mid, i, 8 - q)
    a = lo[5:] + mid[2:6]
    for first, new in enumerate([mid[6]] + hi[:4]):
        exchange(a, first, 7)
        for i in range(first + 1, 7):
            exchange(a, first, i)
            exchange(a, i, 7)
        a[7] = new
    x, y, z = a[5:]
    return np.fmax(np.fmin(x, y), np.fmin(np.fmax(x, y), z))


def third_smallest(v, axis):
    a = [np.full_like(v, np.inf) for _ in range(3)]
    for o in range(-7, 8):
        x = shifted(v, o, axis)
        for q in range(3):
            a[q], x = np.fmin(a[q], x), np.fmax(a[q], x)
    return a[2]


def put(A, kind, rng):
    h, w, d = A.shape
    if kind == "block":
        A[h // 4:h // 2 + 1, w // 4:w // 2 + 1, d // 4:d // 2 + 1] = np.nan
    elif kind == "columns":
        A[rng.random((h, w)) < 0.3] = np.nan
    elif kind == "half":
        A[rng.random(A.shape) < 0.5] = np.nan
    elif kind == "sparse":
        A[rng.random(A.shape) < 0.03] = np.nan
    elif kind == "deep":
        A[:, :, d // 2:] = np.nan
    elif kind == "all":
        A[:] = np.nan
    elif kind == "infinite":  # both signs and NaN
        A[rng.random(A.shape) < 0.2] = np.inf
        A[rng.random(A.shape) < 0.2] = -np.inf
        A[rng.random(A.shape) < 0.1] = np.nan
    return A


@pytest.mark.parametrize("kind", ["block", "columns", "half", "sparse", "deep", "all", "infinite", "none"])
@pytest.mark.parametrize("h,w,d", [(1, 1, 1), (3, 2, 5), (16, 15, 33), (31, 41, 64)])
@pytest.mark.parametrize("fast_axis", [0, 1])
def test_filtered_volume(h, w, d, kind, fast_axis):
    import paper_2010_06931_gb300 as octmc
    rng = np.random.default_rng(h + d)
    A = put(rng.random((h, w, d)).astype(np.float32), kind, rng)
    S = rng.rayleigh(0.5, (h, w, d)).astype(np.float32)
    v = np.ones(h if fast_axis == 0 else w, np.float32)
    F = torch.zeros((h, w, d), dtype=torch.float32, device="cuda")
    octmc.enface(A, S, fast_axis, v, filtered=F)
    want = median(A)
    for axis in ((1, 0) if fast_axis == 0 else (0, 1)):
        want = third_smallest(want, axis)
    np.testing.assert_array_equal(F.cpu().numpy(), want)

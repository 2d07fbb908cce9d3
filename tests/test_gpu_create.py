"""Creation of a problem (GPU only): the pyramid against float64 box means
rounded once (bit-exact), and the acquisition chains of time maps in and out
of raster order, read back through the regulariser R (float32 terms summed in
float64: 1e-5 relative, as every term of the objective)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def down(v):
    """Box mean over pairs per axis, the edge repeated, in the kernel's order of addition."""
    v = v.astype(np.float64)
    for ax in range(3):
        if v.shape[ax] % 2:
            v = np.concatenate([v, np.take(v, [-1], axis=ax)], axis=ax)
    s = 0.0
    for b in range(2):
        for a in range(2):
            s = s + (v[b::2, a::2, 0::2] + v[b::2, a::2, 1::2])
    return (s * 0.125).astype(np.float32)


def values(rng, shape, kind):
    v = rng.rayleigh(0.5, shape).astype(np.float32)
    if kind == "wide":  # magnitudes over 80 binary orders, either sign, zeros
        v = (np.ldexp(v, rng.integers(-40, 40, shape)) * rng.choice([-1.0, 0.0, 1.0], shape)).astype(np.float32)
    elif kind == "halfway":  # sums whose last bits sit on rounding boundaries
        v = (rng.integers(0, 1 << 24, shape).astype(np.float32) * np.exp2(rng.integers(-14, 3, shape))).astype(np.float32)
    elif kind == "special":
        v.reshape(-1)[::7] = np.inf
        v.reshape(-1)[3::11] = 3e38
        v.reshape(-1)[5::13] = 1e-42
    return v


@pytest.mark.parametrize("w,h,d,kind", [
    (1, 1, 2, "plain"), (2, 3, 1, "plain"), (7, 5, 5, "wide"), (9, 16, 6, "halfway"), (17, 3, 8, "special"),
    (16, 10, 61, "wide"), (33, 9, 130, "halfway"), (12, 21, 512, "plain"), (8, 8, 515, "special")])
def test_pyramid_is_the_float64_mean_rounded_once(w, h, d, kind):
    import paper_2010_06931_gb300 as octmc
    rng = np.random.default_rng(w * 1000 + d)
    sx, sy = values(rng, (h, w, d), kind), values(rng, (h, w, d), kind)
    t = np.arange(w * h, dtype=np.float64).reshape(h, w)
    P = octmc.Problem(sx, sy, t, t, levels=3)
    for l in (1, 2):
        with np.errstate(all="ignore"):
            sx, sy = down(sx), down(sy)
        got = P.level_data(l)
        np.testing.assert_array_equal(got["sx"].cpu().numpy(), sx)
        np.testing.assert_array_equal(got["sy"].cpu().numpy(), sy)


def regulariser(D, tx, ty, d, eps=1e-2):
    R = 0.0
    for V, t in enumerate((tx, ty)):
        t = t.reshape(-1)
        o = np.lexsort((np.arange(t.size), t))
        dt = np.diff(t[o])
        om = dt[dt > 0].min() / np.maximum(dt, dt[dt > 0].min()) if (dt > 0).any() else np.ones(dt.size)
        for c in range(3):
            x = np.diff(D[V, c].reshape(-1)[o])
            R += d * (om * (x * x / eps) / (1 + np.sqrt(1 + (x / eps) ** 2))).sum()
    return R


def maps(kind, w, h, rng):
    j, i = np.meshgrid(np.arange(h, dtype=np.float64), np.arange(w, dtype=np.float64), indexing="ij")
    row, col = j * (w + 3) + i, i * (h + 2) + j
    if kind == "raster":
        return row, col
    if kind == "swapped":
        return col, row
    if kind == "ties":  # equal times order by index, along rows but not along columns
        return np.floor(row / 5), np.floor(col / 5)
    if kind == "constant":
        return np.zeros((h, w)), np.full((h, w), 2.5)
    if kind == "reversed":
        return -row, -col
    return rng.permutation(w * h).reshape(h, w) * 0.37, rng.normal(size=(h, w))


@pytest.mark.parametrize("kind", ["raster", "swapped", "ties", "constant", "reversed", "random"])
@pytest.mark.parametrize("w,h", [(1, 1), (1, 9), (13, 1), (11, 14), (70, 33)])
@pytest.mark.parametrize("on_device", [False, True])
def test_chains_of_any_time_map(kind, w, h, on_device):
    import paper_2010_06931_gb300 as octmc
    rng = np.random.default_rng(w * 31 + h)
    d = 4
    s = rng.random((2, h, w, d)).astype(np.float32)
    tx, ty = maps(kind, w, h, rng)
    args = [s[0], s[1], tx, ty]
    if on_device:
        args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in args]
    P = octmc.Problem(*args, levels=2)
    for l in range(2):
        if l:
            pad = lambda t: np.pad(t, [(0, t.shape[0] % 2), (0, t.shape[1] % 2)], mode="edge")
            tx, ty = ((p[0::2, 0::2] + p[0::2, 1::2] + p[1::2, 0::2] + p[1::2, 1::2]) / 4.0 for p in (pad(tx), pad(ty)))
        D = rng.normal(0.0, 0.3, P.disp_shape(l))
        R = P.eval_terms(l, torch.from_numpy(D).cuda())[2]
        want = regulariser(D, tx, ty, P.level_shape(l)[2])
        assert abs(R - want) <= 1e-5 * max(want, 1e-30)


@pytest.mark.parametrize("on_device", [False, True])
def test_times_that_are_not_finite_are_refused(on_device):
    import paper_2010_06931_gb300 as octmc
    s = np.ones((5, 6, 8), np.float32)
    t = np.arange(30, dtype=np.float64).reshape(5, 6)
    bad = t.copy()
    bad[3, 2] = np.inf
    for pair in ((t, bad), (bad, t)):
        args = [s, s, *pair]
        if on_device:
            args = [torch.from_numpy(a).cuda() for a in args]
        with pytest.raises(octmc.OctmcError):
            octmc.Problem(*args)

"""Performance cases of the registration framework: what its users have it do,
each through the package's public entry points.

A pair stands for two orthogonal raster scans of one retina: layered bands on
a bowl with a drusen-like bump, unit-mean Rayleigh speckle drawn per scan, a
vessel pattern with noise as the en-face angiography, and per scan an eye
motion (random-walk drift, saccades, a 1 Hz axial sinusoid) whose B-scans
around a saccade are invalid.  Sizes are those of the package's own workloads
(64^3, 128 x 128 x 256, 300 x 300 x 512, 600 x 600 x 800), the 465-sample
depth of a clinical scan, and odd ones.

Kinds:
  eval      objective + gradient at a displacement field (one solver trial
            point, or one call of a user's own optimiser)
  batch     the objectives of several pairs through autograd, forward and
            backward
  solve     the coarse-to-fine L-BFGS solve, with a cap on its iterations
  prealign  the rough axial prealignment, with a cap on its iterations
  merge     the final resampling and merging of both scans
  enface    saccade validity and en-face projection of one OCTA scan
  create    the upload and pyramid of a new pair
  lbfgs     one direction of the stand-alone L-BFGS
"""
import math

import torch

import paper_2010_06931_gb300 as octmc
from paper_2010_06931_gb300 import autograd

STORAGE = {"f32": octmc.F32, "bf16": octmc.BF16, "f16": octmc.F16}
LOSS = {"huber": octmc.LOSS_PSEUDO_HUBER, "ssd": octmc.LOSS_SSD}
BYTES = {"f32": 4, "bf16": 2, "f16": 2}
ALPHA, DELTA0, EPS_H, EPS_R, ETA = 0.1, 0.5, 1e-3, 1e-2, 0.7


def listed():
    return [
        # the smallest pair in use: launches and latency count
        dict(name="eval_64_f32", kind="eval", w=64, h=64, d=64, storage="f32", loss="huber", angio=True, noise=0.5),
        # the clinical-size evaluation that a solve and the benchmark repeat
        dict(name="eval_300x512_f32", kind="eval", w=300, h=300, d=512, storage="f32", loss="huber", angio=True,
             noise=0.5),
        # odd sizes, the clinical depth, squared differences without angiography, on a field without noise
        dict(name="eval_237x301x465_f16_ssd", kind="eval", w=237, h=301, d=465, storage="f16", loss="ssd",
             angio=False, noise=0.0),
        # the wide-field pair in 16-bit storage: the largest evaluation
        dict(name="eval_600x800_bf16", kind="eval", w=600, h=600, d=800, storage="bf16", loss="huber", angio=True,
             noise=0.1),
        # several small pairs in one differentiable call, forward and backward
        dict(name="batch8_128x256_autograd", kind="batch", pairs=8, w=128, h=128, d=256, storage="f32", noise=0.5),
        # the solve of a small pair: short kernels, one after another
        dict(name="solve_64_3lv", kind="solve", w=64, h=64, d=64, storage="f32", levels=3, iters=20),
        # the clinical-size solve, a fixed budget of iterations on each of the three levels
        dict(name="solve_300x512_3lv", kind="solve", w=300, h=300, d=512, storage="f32", levels=3, iters=10),
        # stage 1 of the same pair
        dict(name="prealign_300x512_3lv", kind="prealign", w=300, h=300, d=512, storage="f32", levels=3, iters=8),
        # the last step of a registration: both scans resampled and merged
        dict(name="merge_300x512_f32", kind="merge", w=300, h=300, d=512, storage="f32", corrected=False),
        # angiography preprocessing of one scan
        dict(name="enface_300x512", kind="enface", w=300, h=300, d=512, fast=0),
        # a new pair: upload from device arrays, pyramid, acquisition chains
        dict(name="create_300x512_3lv", kind="create", w=300, h=300, d=512, storage="f32", levels=3),
        # a direction of the stand-alone optimiser at the clinical field's size
        dict(name="lbfgs_540000_m8", kind="lbfgs", n=540000, m=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, most, lo=(24, 24, 40), hi=(420, 420, 640)):
    """w, h, d spread over their logarithms with at most `most` voxels."""
    while True:
        w, h, d = (_log_int(rng, a, b) for a, b in zip(lo, hi))
        if w * h * d <= most:
            return w, h, d


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "batch", "solve", "solve", "prealign", "merge", "enface", "create",
                       "lbfgs"])
    storage = rng.choice(["f32", "f32", "bf16", "f16"])
    if kind == "eval":
        w, h, d = _grid(rng, 100_000_000, hi=(600, 600, 800))
        return dict(kind=kind, w=w, h=h, d=d, storage=storage, loss=rng.choice(["huber", "huber", "ssd"]),
                    angio=rng.random() < 0.8, noise=rng.choice([0.0, 0.1, 0.5]))
    if kind == "batch":
        w, h, d = _grid(rng, 4_200_000, hi=(128, 128, 256))
        return dict(kind=kind, pairs=rng.randint(2, 16), w=w, h=h, d=d, storage=storage, noise=rng.choice([0.0, 0.5]))
    if kind in ("solve", "prealign"):
        levels = rng.randint(1, 3)
        w, h, d = _grid(rng, 46_000_000)
        return dict(kind=kind, w=w, h=h, d=d, storage=storage, levels=levels,
                    iters=rng.randint(4, 10) if kind == "solve" else rng.randint(3, 8))
    if kind == "merge":
        w, h, d = _grid(rng, 46_000_000)
        return dict(kind=kind, w=w, h=h, d=d, storage=storage, corrected=rng.random() < 0.4)
    if kind == "enface":
        w, h, d = _grid(rng, 46_000_000)
        return dict(kind=kind, w=w, h=h, d=d, fast=rng.randint(0, 1))
    if kind == "create":
        w, h, d = _grid(rng, 46_000_000)
        return dict(kind=kind, w=w, h=h, d=d, storage=storage, levels=rng.randint(2, 3))
    return dict(kind=kind, n=_log_int(rng, 5_000, 1_000_000), m=rng.randint(2, 12))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rand(g, *shape, dtype=torch.float32):
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype)


def _normal(g, *shape, dtype=torch.float64):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _ij(w, h):
    return torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float64),
                          torch.arange(w, device="cuda", dtype=torch.float64), indexing="ij")


def _times(w, h):
    """Sampling-time maps: raster order with a flyback of a quarter B-scan."""
    j, i = _ij(w, h)
    return j * (w + round(0.25 * w)) + i, i * (h + round(0.25 * h)) + j


def _motion(g, w, h):
    """Eye position [3][h][w] of each scan's A-scans and its B-scan validity."""
    out = []
    for scan in range(2):
        nf, nb = (w, h) if scan == 0 else (h, w)
        per = nf + round(0.25 * nf)
        n = per * nb
        m = torch.cumsum(0.03 * math.sqrt(90000.0 / n) * _normal(g, 3, n), dim=1)
        at = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * n
        jump = 2.0 * _normal(g, 2, 3)
        s = torch.arange(n, device="cuda", dtype=torch.float64)
        m[:2] += (jump[:, :, None] * (s[None, None, :] >= at[None, :, None])).sum(1)
        m[2] += 2.0 * torch.sin(2.0 * math.pi * 3.9 * s / n + 6.28 * _rand(g, 1, dtype=torch.float64))
        m = m.view(3, nb, per)[:, :, :nf]
        if scan == 1:
            m = m.transpose(1, 2)
        b = torch.arange(nb, device="cuda", dtype=torch.float64)
        v = ((b[:, None] - torch.floor(at / per)[None, :]).abs() > 2.0).all(1).float()
        out.append(((m - m.mean(dim=(1, 2), keepdim=True)).contiguous(), v))
    return out


def _retina(seed, w, h, d, m, speckle):
    """[h][w][d] float32 structural volume of one scan acquired with motion m."""
    g = _gen(seed)
    j, i = _ij(w, h)
    x, y = (i + m[0]) / w - 0.5, (j + m[1]) / h - 0.5
    bowl = 0.12 * d * (x * x + y * y)
    bump = 6.0 * torch.exp(-((x - 0.1) ** 2 + (y + 0.15) ** 2) / 0.02)
    k = torch.arange(d, device="cuda", dtype=torch.float32)
    n_layers = 9
    amp = [0.55, -0.3, 0.35, -0.25, 0.4, -0.45, 0.5, 0.2, -0.6]
    out = torch.empty((h, w, d), dtype=torch.float32, device="cuda")
    rows = max(1, (1 << 25) // (w * d))
    for j0 in range(0, h, rows):
        sl = slice(j0, min(h, j0 + rows))
        vol = torch.full((sl.stop - sl.start, w, d), 0.08, dtype=torch.float32, device="cuda")
        for q in range(n_layers):
            surf = (d * (0.25 + 0.05 * q) + bowl[sl] + bump[sl] * (q + 1) / n_layers - m[2][sl]).float()
            vol += amp[q] * torch.sigmoid((k - surf[..., None]) / 0.7)
        vol.clamp_(min=0.02)
        if speckle:
            u = torch.rand(vol.shape, generator=g, device="cuda").clamp_(min=1e-7)
            vol *= torch.sqrt(u.log_().mul_(-2.0)) * math.sqrt(2.0 / math.pi)
        out[sl] = vol
    return out


def _vessels(g, w, h, m):
    """[h][w] float32 en-face angiography seen with motion m."""
    j, i = _ij(w, h)
    x, y = i + m[0], j + m[1]
    img = torch.zeros_like(x)
    for q in range(5):
        a = 0.4 + 1.1 * q
        s = math.cos(a) * x + math.sin(a) * y + 4.0 * torch.sin(0.07 * (math.cos(a) * y - math.sin(a) * x) + q)
        img += 0.3 * torch.exp(-((torch.remainder(s + 9.0 * q, 37.0) - 18.5) / 1.6) ** 2)
    return (img + 0.01 * _normal(g, h, w)).float()


def _pair(c, seed):
    """Inputs of one pair: volumes, time maps, angiography, validity, field."""
    w, h, d = c["w"], c["h"], c["d"]
    g = _gen(seed * 7919 + 13)
    (mx, vx), (my, vy) = _motion(g, w, h)
    tx, ty = _times(w, h)
    p = dict(sx=_retina(seed * 7919 + 1, w, h, d, mx, True), sy=_retina(seed * 7919 + 2, w, h, d, my, True),
             tx=tx, ty=ty, ax=None, ay=None, vx=None, vy=None)
    if c.get("angio", True):
        p.update(ax=_vessels(g, w, h, mx), ay=_vessels(g, w, h, my), vx=vx, vy=vy)
    D = -torch.stack([mx, my])
    D += c.get("noise", 0.0) * _normal(g, 2, 3, h, w)
    return p, D.contiguous()


def _problem(c, p, **kw):
    return octmc.Problem(p["sx"], p["sy"], p["tx"], p["ty"], p["ax"], p["ay"], p["vx"], p["vy"],
                         storage=STORAGE[c["storage"]], alpha=ALPHA, delta0=DELTA0, eps_h=EPS_H, eps_r=EPS_R, **kw)


def _octa_scan(c, seed):
    """One scan's OCTA (decorrelation) and OCT volumes; two saturated B-scans."""
    w, h, d = c["w"], c["h"], c["d"]
    g = _gen(seed * 7919 + 3)
    m = torch.zeros((3, h, w), device="cuda", dtype=torch.float64)
    S = _retina(seed * 7919 + 4, w, h, d, m, True)
    dec = _retina(0, w, h, d, m, False).mul_(-8.0).exp_().mul_(0.85).add_(0.05)
    ves = _vessels(g, w, h, m)
    k = torch.arange(d, device="cuda", dtype=torch.float32)
    dec += 0.7 * ves[..., None] * torch.exp(-((k - 0.42 * d) / (0.06 * d)) ** 2)
    dec += 0.03 * torch.randn(dec.shape, generator=g, device="cuda")
    nb = h if c["fast"] == 0 else w
    for b in torch.randint(0, nb, (2,), generator=g, device="cuda").tolist():
        sat = 0.9 + 0.03 * torch.randn((w if c["fast"] == 0 else h, d), generator=g, device="cuda")
        if c["fast"] == 0:
            dec[b] = sat
        else:
            dec[:, b] = sat
    return dec.clamp_(0.0, 1.0).contiguous(), S


def _history(c, seed):
    """m curvature pairs of a quadratic with a spread spectrum, and a gradient."""
    g = _gen(seed * 7919 + 5)
    n = c["n"]
    diag = torch.exp(3.0 * _normal(g, n) / 3.0)
    S = [0.1 * _normal(g, n) for _ in range(c["m"])]
    return S, [diag * s for s in S], _normal(g, n)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        P, D = [], []
        for k in range(c["pairs"]):
            p, f = _pair(c, seed * 31 + k)
            P.append(_problem(c, p))
            P[-1].set_eta(0, ETA)
            D.append(f.requires_grad_())
        return dict(kind=kind, P=P, D=D)
    if kind == "lbfgs":
        S, Y, grad = _history(c, seed)
        opt = octmc.Lbfgs(c["n"], c["m"])
        for s, y in zip(S, Y):
            opt.push(s, y)
        return dict(kind=kind, opt=opt, g=grad)
    if kind == "enface":
        A, S = _octa_scan(c, seed)
        return dict(kind=kind, A=A, S=S, fast=c["fast"])
    p, D = _pair(c, seed)
    if kind == "create":
        return dict(kind=kind, case=c, p=p)
    kw = {}
    if kind in ("solve", "prealign"):
        kw = dict(levels=c["levels"], max_iter=c["iters"])
    if kind == "eval":
        kw = dict(loss=LOSS[c["loss"]])
    P = _problem(c, p, **kw)
    if kind == "eval":
        P.set_eta(0, ETA)
        return dict(kind=kind, P=P, D=D, G=torch.empty_like(D),
                    T=torch.empty(6, dtype=torch.float64, device="cuda"))
    if kind == "merge":
        outs = ("merged", "weights", "angio") + (("corrected_x", "corrected_y") if c["corrected"] else ())
        return dict(kind=kind, P=P, D=D, outs=outs)
    return dict(kind=kind, P=P)


# ---------------------------------------------------------------- one pass
def run(state):
    kind = state["kind"]
    if kind == "eval":
        state["P"].eval_objective_grad_async(0, state["D"], state["G"], state["T"])
        return dict(grad=state["G"], terms=state["T"])
    if kind == "batch":
        for D in state["D"]:
            D.grad = None
        f = autograd.batch_objective(state["P"], 0, state["D"], mode="save")
        f.backward()
        return dict(f=f.detach(), grads=[D.grad for D in state["D"]])
    if kind == "solve":
        D, stats = state["P"].solve_full()
        return dict(field=D, f=[s["f"] for s in stats], eta=[s["eta"] for s in stats],
                    evals=[s["evals"] for s in stats])
    if kind == "prealign":
        prm, D, stats = state["P"].prealign_full()
        return dict(prm=prm, field=D, f=[s["f"] for s in stats], evals=[s["evals"] for s in stats])
    if kind == "merge":
        return state["P"].merge(state["D"], outputs=state["outs"])
    if kind == "enface":
        v, means = octmc.saccade_validity(state["A"], state["fast"])
        E, info = octmc.enface(state["A"], state["S"], state["fast"], v)
        return dict(v=v, means=means, image=E, **info)
    if kind == "create":
        c = state["case"]
        P = _problem(c, state["p"], levels=c["levels"])
        out = [P.level_data(l) for l in range(1, c["levels"])]
        P.destroy_problem()
        return out
    d, gtd = state["opt"].direction(state["g"])
    return dict(dir=d, gtd=gtd)


# ---------------------------------------------------------------- work
def _eval_work(w, h, d, s):
    """Both volumes, both images, the field and the gradient once; per voxel
    and scan 44 multiply-adds of the separable interpolant with its adjoint
    gradient, per voxel pair 8 flops of loss."""
    return w * h * (2.0 * d * s + 8 + 48 + 48), w * h * d * 184.0


def work(case):
    c, kind = case, case["kind"]
    if kind == "lbfgs":  # the pairs are read for the products and for the combination
        n, m = float(c["n"]), c["m"]
        return dict(bytes=n * 8 * (2 * m + 2), flops=n * (8 * m + 2))
    w, h, d = c["w"], c["h"], c["d"]
    n, s = float(w) * h, BYTES.get(c.get("storage", "f32"), 4)
    if kind == "eval":
        b, f = _eval_work(w, h, d, s)
    elif kind == "batch":
        b, f = (c["pairs"] * v for v in _eval_work(w, h, d, s))
    elif kind in ("solve", "prealign"):
        b = f = 0.0
        for _ in range(c["levels"]):
            eb, ef = _eval_work(w, h, d, s)
            if kind == "prealign":  # integer transverse positions: the axial filter alone
                ef = w * h * d * (2 * 8 * 2 + 8.0)
            b, f = b + (c["iters"] + 1) * eb, f + (c["iters"] + 1) * ef
            w, h, d = (w + 1) // 2, (h + 1) // 2, (d + 1) // 2
    elif kind == "merge":
        outs = 3 if c["corrected"] else 1
        b, f = n * (2.0 * d * s + outs * d * 4.0 + 48 + 8 + 8 + 4), n * d * (2 * 24 * 2 + 3.0)
    elif kind == "enface":  # both volumes once; median and rank filters as compare-exchanges
        b, f = n * (2.0 * d * 4 + 4), n * d * (2 * 100 + 2 * 14 * 5.0)
    else:  # create: the volumes read, every level written
        b = n * 2.0 * d * 4
        f = 0.0
        for _ in range(c["levels"]):
            b += 2.0 * w * h * d * s + w * h * (8 + 32.0)
            w, h, d = (w + 1) // 2, (h + 1) // 2, (d + 1) // 2
            f += 2.0 * w * h * d * 8
    return dict(bytes=float(b), flops=float(f))


# ---------------------------------------------------------------- 64-bit values
def _keys(t):
    """Catmull-Rom weights (and their derivatives) of the samples n-1..n+2."""
    w = [t * (-0.5 + t * (1 - 0.5 * t)), 1 + t * t * (1.5 * t - 2.5), t * (0.5 + t * (2 - 1.5 * t)),
         t * t * (0.5 * t - 0.5)]
    dw = [-0.5 + t * (2 - 1.5 * t), t * (4.5 * t - 5), 0.5 + t * (4 - 4.5 * t), t * (1.5 * t - 1)]
    return w, dw


def _stored(c, vol):
    return vol if c["storage"] == "f32" else vol.to(torch.bfloat16 if c["storage"] == "bf16" else torch.float16)


def _resample(vol, i, j, D, grad):
    """[n][d] values of one volume at A-scans (i, j) displaced by D [3][n],
    and with `grad` their derivatives with respect to the displacement."""
    h, w, d = vol.shape
    bx, by, bz = (torch.floor(v) for v in (i + D[0], j + D[1], D[2]))
    wx, dwx = _keys(i + D[0] - bx)
    wy, dwy = _keys(j + D[1] - by)
    wz, dwz = _keys(D[2] - bz)
    T = Tx = Ty = 0.0
    for b in range(4):
        jj = (by.long() - 1 + b).clamp(0, h - 1)
        for a in range(4):
            s = vol[jj, (bx.long() - 1 + a).clamp(0, w - 1)].double()
            T = T + (wx[a] * wy[b])[:, None] * s
            if grad:
                Tx = Tx + (dwx[a] * wy[b])[:, None] * s
                Ty = Ty + (wx[a] * dwy[b])[:, None] * s
    k = torch.arange(d, device="cuda")
    I, Iz, Ix, Iy = 0.0, 0.0, 0.0, 0.0
    for c in range(4):
        at = (k[None, :] + bz.long()[:, None] - 1 + c).clamp(0, d - 1)
        e = T.gather(1, at)
        I = I + wz[c][:, None] * e
        if grad:
            Iz = Iz + dwz[c][:, None] * e
            Ix = Ix + wz[c][:, None] * Tx.gather(1, at)
            Iy = Iy + wz[c][:, None] * Ty.gather(1, at)
    return (I, Ix, Iy, Iz) if grad else I


def _image(img, i, j, D):
    """Values and x, y derivatives of an en-face image at displaced positions."""
    h, w = img.shape
    bx, by = torch.floor(i + D[0]), torch.floor(j + D[1])
    wx, dwx = _keys(i + D[0] - bx)
    wy, dwy = _keys(j + D[1] - by)
    v = vx = vy = 0.0
    for b in range(4):
        for a in range(4):
            s = img[(by.long() - 1 + b).clamp(0, h - 1), (bx.long() - 1 + a).clamp(0, w - 1)].double()
            v, vx, vy = v + wx[a] * wy[b] * s, vx + dwx[a] * wy[b] * s, vy + wx[a] * dwy[b] * s
    return v, vx, vy


def _line(v, u):
    """Validity by the zero-tangent Hermite interpolant, and its derivative."""
    b = torch.floor(u)
    t, n = u - b, v.numel()
    p0, p1 = (v[(b.long() + q).clamp(0, n - 1)].double() for q in (0, 1))
    return p0 + (p1 - p0) * t * t * (3 - 2 * t), (p1 - p0) * 6 * t * (1 - t)


def _loss(x, eps, kind):
    if kind == "ssd":
        return x * x, 2 * x
    q = torch.sqrt(1 + (x / eps) ** 2)
    return x * x / eps / (1 + q), x / eps / q


def _exact_eval(c, seed, loss="huber"):
    """Gradient [2][3][h][w] and terms of the objective."""
    p, D = _pair(c, seed)
    w, h, d = c["w"], c["h"], c["d"]
    jj, ii = (v.reshape(-1) for v in _ij(w, h))
    Df = D.view(2, 3, -1)
    sx, sy = _stored(c, p["sx"]), _stored(c, p["sy"])
    n = w * h
    G = torch.zeros((2, 3, n), dtype=torch.float64, device="cuda")
    S = torch.zeros((), dtype=torch.float64, device="cuda")
    A = torch.zeros_like(S)
    step = max(1, (1 << 24) // d)
    for a in range(0, n, step):
        sl = slice(a, min(n, a + step))
        i, j, X, Y = ii[sl], jj[sl], Df[0][:, sl], Df[1][:, sl]
        IX, XX, XY, XZ = _resample(sx, i, j, X, True)
        IY, YX, YY, YZ = _resample(sy, i, j, Y, True)
        L, dL = _loss(IX - IY, EPS_H, loss)
        Ls = L.sum(1)
        gs = [(dL * v).sum(1) for v in (XX, XY, XZ)] + [-(dL * v).sum(1) for v in (YX, YY, YZ)]
        if p["ax"] is None:
            S += Ls.sum()
            G.view(6, n)[:, sl] = ETA * torch.stack(gs)
            continue
        vx, dvx = _line(p["vx"], j + X[1])
        vy, dvy = _line(p["vy"], i + Y[0])
        dl = DELTA0 * vx * vy
        ax, axx, axy = _image(p["ax"], i, j, X)
        ay, ayx, ayy = _image(p["ay"], i, j, Y)
        La, dLa = _loss(ax - ay, EPS_H, loss)
        S += ((1 - dl) * Ls).sum()
        A += (dl * d * La).sum()
        gs = [ETA * (1 - dl) * v for v in gs]
        ca, dd = dl * d / ETA * dLa, -ETA * Ls + d * La / ETA
        gs[0] = gs[0] + ca * axx
        gs[1] = gs[1] + ca * axy + dd * DELTA0 * dvx * vy
        gs[3] = gs[3] - ca * ayx + dd * DELTA0 * vx * dvy
        gs[4] = gs[4] - ca * ayy
        G.view(6, n)[:, sl] = torch.stack(gs)
    R = torch.zeros_like(S)
    for V, t in enumerate((p["tx"], p["ty"])):
        o = torch.argsort(t.reshape(-1))
        dt = t.reshape(-1)[o].diff()
        om = dt.min() / dt
        for q in range(3):
            L, dL = _loss(Df[V, q][o].diff(), EPS_R, "huber")
            R += d * (om * L).sum()
            G[V, q].index_add_(0, o[1:], ALPHA * d * om * dL)
            G[V, q].index_add_(0, o[:-1], -ALPHA * d * om * dL)
    mu = 1.0 / (2.0 * n)
    Sc = Df.sum(dim=(0, 2))
    G += (2 * mu * Sc)[None, :, None]
    M = mu * (Sc ** 2).sum()
    f = ETA * S + A / ETA + ALPHA * R + M
    return G.view(2, 3, h, w), torch.stack([S, A, R, M, f, torch.full_like(S, ETA)])


def _exact_merge(c, seed, beta=2.0, tau=0.05):
    p, D = _pair(c, seed)
    w, h, d = c["w"], c["h"], c["d"]
    n = w * h
    jj, ii = (v.reshape(-1) for v in _ij(w, h))
    Df = D.view(2, 3, -1)
    raw = []
    for V in range(2):
        u, v = (ii + Df[V, 0]).clamp(0, w - 1), (jj + Df[V, 1]).clamp(0, h - 1)
        x0, y0 = torch.floor(u), torch.floor(v)
        fx, fy = u - x0, v - y0
        x0, y0 = x0.long(), y0.long()
        x1, y1 = (x0 + 1).clamp(max=w - 1), (y0 + 1).clamp(max=h - 1)
        foot = [(y0 * w + x0, (1 - fx) * (1 - fy)), (y0 * w + x1, fx * (1 - fy)), (y1 * w + x0, (1 - fx) * fy),
                (y1 * w + x1, fx * fy)]
        dens = torch.zeros(n, dtype=torch.float64, device="cuda")
        for at, wt in foot:
            dens.index_add_(0, at, wt)
        rho = sum(wt * dens[at] for at, wt in foot)
        raw.append(torch.exp(-beta * (rho - 1).clamp(min=0)))
    cl = [torch.where(r >= tau, r, torch.zeros_like(r)) for r in raw]
    none = (cl[0] == 0) & (cl[1] == 0)
    cl[0] = torch.where(none & (raw[0] >= raw[1]), torch.ones_like(raw[0]), cl[0])
    cl[1] = torch.where(none & (raw[0] < raw[1]), torch.ones_like(raw[1]), cl[1])
    wx, wy = cl[0] / (cl[0] + cl[1]), cl[1] / (cl[0] + cl[1])
    va = _line(p["vx"], jj + Df[0, 1])[0], _line(p["vy"], ii + Df[1, 0])[0]
    a = [(cl[V] * va[V]).clamp(min=0) for V in range(2)]
    im = _image(p["ax"], ii, jj, Df[0])[0], _image(p["ay"], ii, jj, Df[1])[0]
    tot = a[0] + a[1]
    ang = torch.where(tot > 0, (a[0] * im[0] + a[1] * im[1]) / tot.clamp(min=1e-300), torch.zeros_like(tot))
    sx, sy = _stored(c, p["sx"]), _stored(c, p["sy"])
    out = dict(weights=torch.stack([wx, wy]).view(2, h, w), angio=ang.view(h, w))
    vols = {k: torch.empty((n, d), dtype=torch.float64, device="cuda")
            for k in ("merged",) + (("corrected_x", "corrected_y") if c["corrected"] else ())}
    step = max(1, (1 << 24) // d)
    for b in range(0, n, step):
        sl = slice(b, min(n, b + step))
        IX = _resample(sx, ii[sl], jj[sl], Df[0][:, sl], False)
        IY = _resample(sy, ii[sl], jj[sl], Df[1][:, sl], False)
        vols["merged"][sl] = wx[sl, None] * IX + wy[sl, None] * IY
        if c["corrected"]:
            vols["corrected_x"][sl], vols["corrected_y"][sl] = IX, IY
    out.update({k: v.view(h, w, d) for k, v in vols.items()})
    return out


def _shift(v, o, dim):
    """v at index + o along dim, edges replicated."""
    n = v.shape[dim]
    return v.index_select(dim, (torch.arange(n, device="cuda") + o).clamp(0, n - 1))


def _exact_enface(c, seed):
    A, S = _octa_scan(c, seed)
    w, h, d, fast = c["w"], c["h"], c["d"], c["fast"]
    nb, bdim = (h, 0) if fast == 0 else (w, 1)
    red = (1, 2) if fast == 0 else (0, 2)
    means = A.double().mean(dim=red)
    lim = means.mean() + 3 * means.std(unbiased=False)
    sat = means > lim
    bad = torch.zeros_like(sat)
    for b in torch.nonzero(sat).flatten().tolist():
        bad[max(0, b - 2):b + 3] = True
    v = (~bad).float()
    F = torch.empty_like(A)
    rows = max(1, (1 << 23) // (w * d))
    for j0 in range(0, h, rows):
        at = (torch.arange(j0 - 1, min(h, j0 + rows) + 1, device="cuda")).clamp(0, h - 1)
        slab = A.index_select(0, at)
        m = slab.shape[0] - 2
        nine = [_shift(_shift(slab[b:b + m], di, 1), dk, 2) for b in range(3) for di in (-1, 0, 1) for dk in (-1, 0, 1)]
        F[j0:j0 + m] = torch.stack(nine, -1).median(dim=-1).values
    for dim in ((1, 0) if fast == 0 else (0, 1)):
        a1 = torch.full_like(F, math.inf)
        a2, a3 = a1.clone(), a1.clone()
        for o in range(-7, 8):
            x = _shift(F, o, dim)
            a1, x = torch.minimum(a1, x), torch.maximum(a1, x)
            a2, x = torch.minimum(a2, x), torch.maximum(a2, x)
            a3 = torch.minimum(a3, x)
        F = a3
    keep = v > 0 if bool((v > 0).any()) else torch.ones_like(v, dtype=torch.bool)
    sel = F.index_select(bdim, torch.nonzero(keep).flatten()).reshape(-1).sort().values
    qs = []
    for q in (0.05, 0.95):
        pos = q * (sel.numel() - 1)
        lo = int(math.floor(pos))
        x0, x1 = float(sel[lo]), float(sel[min(lo + 1, sel.numel() - 1)])
        qs.append(x0 + (pos - lo) * (x1 - x0))
    del sel
    cut = qs[0] + 0.1 * (qs[1] - qs[0])
    t_oct = float(S.index_select(bdim, torch.nonzero(keep).flatten()).double().mean())
    mask = (F.double() < cut) & (S.double() > t_oct)
    cnt = mask.sum(2)
    E = (A.double() * mask).sum(2) / cnt.clamp(min=1)
    Eb = E if fast == 0 else E.t()
    so = Eb.sort(dim=1).values
    nf = so.shape[1]
    Eb = Eb - 0.5 * (so[:, (nf - 1) // 2] + so[:, nf // 2])[:, None]
    ok = torch.nonzero(v > 0).flatten().tolist()
    src = [b if not ok or v[b] > 0 else min(ok, key=lambda q: (abs(q - b), q)) for b in range(nb)]
    Eb = Eb[src]
    E = Eb if fast == 0 else Eb.t()
    return dict(v=v.double(), means=means, image=E.contiguous(), p_lo=qs[0], p_hi=qs[1], t_oct=t_oct, kept=None)


def _exact_create(c, seed):
    p, _ = _pair(c, seed)

    def down(v, dims):
        v = v.double()
        for k in dims:
            if v.shape[k] % 2:
                v = torch.cat([v, v.narrow(k, v.shape[k] - 1, 1)], k)
        for k in dims:
            n = v.shape[k] // 2
            even = torch.arange(n, device="cuda") * 2
            v = v.index_select(k, even) + v.index_select(k, even + 1)
        return (v / 2 ** len(dims)).float()

    out = []
    lv = dict(p)
    for _ in range(1, c["levels"]):
        lv = dict(sx=down(lv["sx"], (0, 1, 2)), sy=down(lv["sy"], (0, 1, 2)), ax=down(lv["ax"], (0, 1)),
                  ay=down(lv["ay"], (0, 1)), vx=down(lv["vx"], (0,)), vy=down(lv["vy"], (0,)))
        out.append({k: (_stored(c, t) if k in ("sx", "sy") else t).double() for k, t in lv.items()})
    return out


def _exact_lbfgs(c, seed):
    """Two-loop recursion with H0 = (s'y / y'y) of the newest pair."""
    S, Y, g = _history(c, seed)
    q, al = g.clone(), []
    for s, y in zip(reversed(S), reversed(Y)):
        al.append(torch.dot(s, q) / torch.dot(s, y))
        q = q - al[-1] * y
    q = q * (torch.dot(S[-1], Y[-1]) / torch.dot(Y[-1], Y[-1]))
    for s, y, a in zip(S, Y, reversed(al)):
        q = q + s * (a - torch.dot(y, q) / torch.dot(s, y))
    return dict(dir=-q, gtd=float(-torch.dot(g, q)))


def exact(case, seed):
    """The outputs of run() in 64 bits.  The capped solves have none: their
    iterates depend on every line search before them."""
    c, kind = case, case["kind"]
    if kind == "eval":
        G, T = _exact_eval(c, seed, c["loss"])
        return dict(grad=G, terms=T)
    if kind == "batch":
        got = [_exact_eval(c, seed * 31 + k) for k in range(c["pairs"])]
        return dict(f=sum(T[4] for _, T in got), grads=[G for G, _ in got])
    if kind == "merge":
        return _exact_merge(c, seed)
    if kind == "enface":
        return _exact_enface(c, seed)
    if kind == "create":
        return _exact_create(c, seed)
    if kind == "lbfgs":
        return _exact_lbfgs(c, seed)
    return None

"""The work users of this library have it do, as cases that can be timed and compared.

Every case goes through the public Python entry points (``paper_1605_02060_gb300.lddmm``,
``autograd``, ``surrogate`` and ``warm64``) on inputs that already lie on the GPU.  ``kind`` says
which part of a registration it is:

  step        one or a few gradient-descent iterations from a velocity field in hand (a resumed
              checkpoint or a warm start), the loop every registration consists of
  register    a whole multiscale schedule from v = 0
  apply       applying a stored registration: label transfer and warps in both directions
  grad        energy and exact gradient through torch.autograd
  preprocess  mask generation and histogram matching of a raw target
  evaluate    surface distances and Dice of a result
  train       one training step of the warm-start network
  predict     the network's initial velocity on a registration grid

Grids are (nx, ny, nz); 264x160x228 is the 50 um brain box, 132x80x114 the 100 um one, 32^3 the
single-ellipsoid problem, 64^3 the network's grid and 128^3 the gradient's.
"""
import math

import numpy as np
import torch

from paper_1605_02060_gb300 import autograd as AG
from paper_1605_02060_gb300 import lddmm as L
from paper_1605_02060_gb300 import surrogate as SG
from paper_1605_02060_gb300 import warm64 as W64

DEV = "cuda" if torch.cuda.is_available() else "cpu"
FULL = (264, 160, 228)
N_FULL = 264 * 160 * 228


def _step(name, dims, iters=1, T=10, k_mode=1, storage=0, rk4=False, h=(1.0, 1.0, 1.0)):
    return {"name": name, "kind": "step", "nx": dims[0], "ny": dims[1], "nz": dims[2], "T": T,
            "iters": iters, "k_mode": k_mode, "storage": storage, "rk4": rk4, "hx": h[0],
            "hy": h[1], "hz": h[2]}


def _dims(kind, name, dims, **kw):
    return dict({"name": name, "kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2]}, **kw)


def listed():
    return [
        # one iteration of the smallest problem with its energy read back, as an optimiser loop
        # that checks the energy does it: default parameters (FP32 products for K)
        _step("step_32", (32, 32, 32), k_mode=0),
        # the 4x/2x/1x schedule on the 100 um brain box, the default 20 iterations per level; its
        # coarse levels are 33x20x29 and 66x40x57
        _dims("register", "register_132", (132, 80, 114), T=10, iterations=20, k_mode=1),
        # a box cropped from a scan: no axis is a round number
        _step("step_odd", (141, 97, 109)),
        # the 100 um box with default parameters (plain fp32 throughout)
        _step("step_132_fp32", (132, 80, 114), iters=2, k_mode=0),
        # a stretch of the headline loop at 50 um
        _step("step_264", FULL, iters=3),
        # the precision form: velocity and images stored bf16
        _step("step_264_bf16", FULL, storage=1),
        # a stored 50 um registration applied to an atlas and both images
        _dims("apply", "apply_264", FULL, T=10, k_mode=1),
        # one pair of a batch of 128^3 pairs, maps recomputed from checkpoints
        _dims("grad", "grad_128", (128, 128, 128), T=10, checkpoint=True),
        # a raw 50 um target: threshold, opening, closing, then the template's grey levels matched
        _dims("preprocess", "preprocess_264", FULL, r_open=1, r_close=3, bins=32, points=8),
        # scoring a 50 um result
        _dims("evaluate", "evaluate_264", FULL),
        # one Adam step of the shipped network's architecture at its training batch
        {"name": "train_64", "kind": "train", "n": 64, "batch": 8},
        # the learned warm start's network for a 50 um pair
        _dims("predict", "predict_264", FULL),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi, most):
    """Three sizes spread over their logarithm, odd ones among them, of at most `most` voxels."""
    while True:
        d = tuple(_size(rng, lo, hi) for _ in range(3))
        if d[0] * d[1] * d[2] <= most:
            return d


def draw(rng):
    kind = rng.choice(["step", "step", "step", "register", "apply", "grad", "preprocess",
                       "evaluate", "train", "predict"])
    if kind == "step":
        k_mode = rng.choice([0, 1, 1, 1, 2])
        # FP32 products up to the 100 um box, tensor-core products up to the 50 um box and a
        # little past 256 along an axis
        d = _box(rng, 20, 300, 132 * 80 * 114 if k_mode == 0 else N_FULL)
        rk4 = rng.random() < 0.2
        h = tuple(rng.choice([1.0, 1.0, 0.5, 1.25]) for _ in range(3))
        c = _step("", d, iters=rng.choice([1, 2]), T=4 if rk4 else rng.choice([5, 8, 10]),
                  k_mode=k_mode, storage=rng.choice([0, 0, 1]), rk4=rk4, h=h)
    elif kind == "register":
        d = _box(rng, 24, 160, 132 * 80 * 114)
        c = _dims(kind, "", d, T=rng.choice([5, 10]), iterations=rng.choice([5, 10, 20]),
                  k_mode=rng.choice([1, 1, 2]))
    elif kind == "apply":
        c = _dims(kind, "", _box(rng, 24, 264, N_FULL), T=rng.choice([4, 10]), k_mode=1)
    elif kind == "grad":
        c = _dims(kind, "", _box(rng, 16, 160, 128 ** 3), T=rng.choice([4, 10]),
                  checkpoint=rng.random() < 0.5)
    elif kind == "preprocess":
        c = _dims(kind, "", _box(rng, 32, 264, N_FULL), r_open=rng.randint(0, 2),
                  r_close=rng.randint(1, 3), bins=rng.choice([32, 64, 100]),
                  points=rng.choice([4, 8, 15]))
    elif kind == "evaluate":
        c = _dims(kind, "", _box(rng, 32, 264, N_FULL))
    elif kind == "train":
        c = {"kind": kind, "n": rng.choice([16, 24, 32, 40, 48, 56, 64]), "batch": rng.randint(1, 8)}
    else:
        c = _dims(kind, "", _box(rng, 40, 264, N_FULL))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------------------
# inputs: smooth random fields from Gaussian blobs, ellipsoid-union masks pulled through them

def _gen(seed):
    return torch.Generator().manual_seed(int(seed))


def _blobs(shape, n, width, g, lo=0.0, hi=1.0):
    """n separable Gaussians of the given width (voxels) with centres in the box, [n][z][y][x]."""
    ax = []
    for d in shape:
        c = (lo + (hi - lo) * torch.rand(n, generator=g)) * d
        x = torch.arange(d, dtype=torch.float32)
        ax.append(torch.exp(-0.5 * ((x[None] - c[:, None]) / width) ** 2).to(DEV))
    return ax[0][:, :, None, None] * ax[1][:, None, :, None] * ax[2][:, None, None, :]


def _smooth(shape, ncomp, amplitude, g, n=12):
    """ncomp smooth fields scaled to a common maximum of `amplitude`, [ncomp][z][y][x]."""
    b = _blobs(shape, n, 0.18 * min(shape), g)
    w = torch.randn(ncomp, n, generator=g).to(DEV)
    f = (w @ b.reshape(n, -1)).reshape((ncomp,) + tuple(shape))
    return f * (amplitude / f.abs().amax())


def _pull(a, u):
    """a at the nearest voxel of x + u(x) (edges clamped), u in voxels as (x, y, z)."""
    Z, Y, X = a.shape
    z, y, x = torch.meshgrid(*(torch.arange(d, device=DEV, dtype=torch.float32) for d in (Z, Y, X)),
                             indexing="ij")
    i = [torch.floor(q + s + 0.5).long().clamp_(0, d - 1)
         for q, s, d in ((z, u[2], Z), (y, u[1], Y), (x, u[0], X))]
    return a[i[0], i[1], i[2]]


def _ellipsoids(shape, g):
    """Union of three overlapping ellipsoids (the brain's outline), bool."""
    m = torch.zeros(shape, dtype=torch.bool, device=DEV)
    base = [(0.5, 0.5, 0.5, 0.36, 0.33, 0.33), (0.38, 0.5, 0.55, 0.2, 0.24, 0.24),
            (0.62, 0.5, 0.55, 0.2, 0.24, 0.24)]
    for e in base:
        j = (torch.rand(6, generator=g) - 0.5) * 0.06
        p = [v + float(d) for v, d in zip(e, j)]
        q = 0.0
        for k, d in enumerate(shape):              # axes z, y, x of the array
            c, a = p[2 - k] * d, p[5 - k] * d
            r = ((torch.arange(d, device=DEV, dtype=torch.float32) - c) / a) ** 2
            q = q + r.reshape([-1 if i == k else 1 for i in range(3)])
        m |= q <= 1.0
    return m


def _dilate(m, r):
    f = m.to(torch.float32)[None, None]
    return torch.nn.functional.max_pool3d(f, 2 * r + 1, 1, r)[0, 0]


def _pair(shape, g):
    """Binary template and target masks and the weight mask (float32), and the warp between."""
    u = _smooth(shape, 3, max(3.0, 0.05 * min(shape)), g)
    m0 = _ellipsoids(shape, g)
    m1 = _pull(m0, u)
    return m0.float(), m1.float(), _dilate(m0 | m1, 2), u


def _labels(m0, g, n=50):
    """Regions 1..n of the mask (nearest of n seeds), as int16 bit patterns of uint16 labels."""
    Z, Y, X = m0.shape
    s = torch.rand(n, 3, generator=g)
    best = torch.full(m0.shape, 3e38, device=DEV)
    lab = torch.zeros(m0.shape, dtype=torch.int16, device=DEV)
    ax = [torch.arange(d, device=DEV, dtype=torch.float32) for d in (Z, Y, X)]
    for k in range(n):
        c = [0.15 + 0.7 * float(s[k, i]) for i in range(3)]
        d2 = ((ax[0] - c[0] * Z) ** 2)[:, None, None] + ((ax[1] - c[1] * Y) ** 2)[None, :, None] + \
             ((ax[2] - c[2] * X) ** 2)[None, None, :]
        near = d2 < best
        best = torch.where(near, d2, best)
        lab.masked_fill_(near, k + 1)
    return torch.where(m0 > 0.5, lab, torch.zeros_like(lab))


def _velocity(shape, T, h, g):
    """A mid-registration velocity field [T][3][z][y][x] in physical units: smooth in space,
    changing slowly over time, moving voxels by up to 4% of the smallest side plus a drift."""
    amp = 0.04 * min(shape)
    a, b = _smooth(shape, 3, amp, g), _smooth(shape, 3, 0.3 * amp, g)
    drift = (0.37 * (2 * torch.rand(3, generator=g) - 1)).to(DEV)[:, None, None, None]
    hh = torch.tensor(h, dtype=torch.float32, device=DEV)[:, None, None, None]
    v = torch.empty((T, 3) + tuple(shape), device=DEV)
    for t in range(T):
        v[t] = (a + ((t + 0.5) / T - 0.5) * 2.0 * b + drift) * hh
    return v


def _raw_target(m, g):
    """A sparsely labelled scan: 0.05 inside with 1% bright log-normal voxels, noise everywhere,
    smoothed by a one-voxel Gaussian (the image that is thresholded)."""
    dg = torch.Generator(device=DEV).manual_seed(int(torch.randint(1 << 30, (1,), generator=g)))
    r = torch.rand(m.shape, generator=dg, device=DEV)
    ln = torch.exp(torch.randn(m.shape, generator=dg, device=DEV))
    img = torch.where(r < 0.01, ln, torch.zeros_like(ln)) + 0.05
    img = torch.where(m > 0.5, img, torch.zeros_like(img))
    img = img + 0.02 * torch.randn(m.shape, generator=dg, device=DEV)
    k = torch.exp(-0.5 * torch.arange(-3, 4, dtype=torch.float32) ** 2)
    k = (k / k.sum()).tolist()
    sm = img
    for ax in range(3):
        acc = torch.zeros_like(sm)
        for i, c in enumerate(k):
            acc += c * torch.roll(sm, i - 3, ax)
        sm = acc
    return img, sm


# ------------------------------------------------------------------------------------------

def _shape(c):
    return (c["nz"], c["ny"], c["nx"])


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    g = _gen(seed)
    k = case["kind"]
    s = {}
    if k == "train":
        n, B = case["n"], case["batch"]
        x, y = [], []
        for _ in range(B):
            m0, m1, _, u = _pair((n, n, n), g)
            x.append(torch.stack([m0, m1]))
            y.append(_smooth((n, n, n), 3, 1.0, g) * (u.abs().amax(0) > 0.02 * n) * 2.5)
        s["x"], s["y"] = torch.stack(x), torch.stack(y)
        return s
    shape = _shape(case)
    s["I0"], s["I1"], s["M"], u = _pair(shape, g)
    if k in ("step", "apply", "grad"):
        h = (case.get("hx", 1.0), case.get("hy", 1.0), case.get("hz", 1.0))
        s["v"] = _velocity(shape, case["T"], h, g)
        if case.get("storage"):
            s["v"] = s["v"].bfloat16().float()
    if k == "apply":
        s["L0"] = _labels(s["I0"], g)
        b = _smooth(shape, 1, 0.5, g)[0]
        s["G0"], s["G1"] = s["I0"] * (0.5 + b), s["I1"] * (0.5 + _pull(b, u))
    if k == "evaluate":
        lab = _labels(s["I0"], g)
        s["LA"], s["LB"] = _pull(lab, 0.9 * u), _pull(lab, u)
        s["A"], s["B"] = (s["LA"] > 0).to(torch.uint8), (s["LB"] > 0).to(torch.uint8)
    if k == "preprocess":
        s["raw"], s["smooth"] = _raw_target(s["I1"], g)
        lab = _labels(s["I0"], g).long()
        grey = (0.5 + 0.15 * torch.randn(51, generator=g)).to(DEV)
        grey[0] = 0.0
        s["atlas"] = grey[lab]
    return s


def prepare(case, seed):
    k = case["kind"]
    s = _inputs(case, seed)
    s["case"] = case
    if k == "train":
        n, B = case["n"], case["batch"]
        # a run in progress: weights, Adam's second moments of some 2000 steps, a decayed rate
        net = SG.UNet3D(chans=W64.CHANS, cin=2, cout=3, n=n, batch=B, seed=int(seed) % 1000)
        net.step_count = 2000
        for m in net.vw + net.vb:
            m.fill_(1e-4)
        s["net"] = net
        return s
    if k == "predict":
        s["net"] = W64.load_net(W64.WEIGHTS)
        return s
    if k == "preprocess":
        return s
    shape = _shape(case)
    kw = {"k_mode": case.get("k_mode", 1), "T": case.get("T", 10)}
    if k == "step":
        kw.update(storage=case["storage"], flags=4 if case["rk4"] else 0, hx=case["hx"],
                  hy=case["hy"], hz=case["hz"])
    if k == "grad":
        kw["flags"] = 2 if case["checkpoint"] else 0
    if k == "register":
        kw.update(iterations=case["iterations"], level_factor=[4, 2, 1])
    p = L.default_params(case["nx"], case["ny"], case["nz"], **kw)
    s["ctx"] = L.Lddmm(p, s["I0"], s["I1"], s["M"])
    if k in ("step", "register"):
        s["out"] = torch.empty((kw["T"], 3) + shape, device=DEV)
    if k == "register":
        c = (lambda n: (n + 3) // 4)
        s["zero"] = torch.zeros((kw["T"], 3) + tuple(c(d) for d in shape), device=DEV)
        s["J0"] = torch.empty(shape, device=DEV)
    if k == "apply":
        s["lab"] = torch.empty(shape, dtype=torch.int16, device=DEV)
        s["w0"], s["w1"] = torch.empty(shape, device=DEV), torch.empty(shape, device=DEV)
    return s


# the energies are sums of FP32 terms: a log keeps them as float32
def _energy32(e):
    return np.array([e["total"], e["reg"], e["data"], e["min_det"]], np.float32)


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "step":
        ctx = s["ctx"]
        ctx.set_velocity(s["v"])
        for _ in range(c["iters"] - 1):
            ctx.step(want_energy=False)
        e = ctx.step()
        v = ctx.get_velocity(s["out"])
        # a field stored bf16 is kept in that type
        return {"v": v.bfloat16() if c["storage"] else v, "energy": _energy32(e)}
    if k == "register":
        ctx = s["ctx"]
        ctx.set_level(0)
        ctx.set_velocity(s["zero"])
        trace = ctx.register()
        return {"v": ctx.get_velocity(s["out"]), "J0": ctx.get_field(L.LDDMM_FIELD_J0, s["J0"]),
                "energies": np.array([t["total"] for t in trace], np.float32)}
    if k == "apply":
        ctx = s["ctx"]
        ctx.set_velocity(s["v"])
        return {"labels": ctx.transfer_labels(s["L0"], s["lab"]),
                "moved": ctx.warp(s["G0"], 0, s["w0"]), "back": ctx.warp(s["G1"], 1, s["w1"])}
    if k == "grad":
        v = s["v"].detach().requires_grad_(True)
        E = AG.energy(v, s["ctx"])
        E.backward()
        return {"grad": v.grad, "energy": E.detach().float()}
    if k == "preprocess":
        mask = L.mask_morphology(s["smooth"], 0.025, c["r_open"], c["r_close"])
        matched = L.histogram_match(s["atlas"], s["I0"], s["raw"], mask.float(), bins=c["bins"],
                                    points=c["points"])
        return {"mask": mask, "matched": matched}
    if k == "evaluate":
        ctx = s["ctx"]
        hd, md, na, nb = ctx.surface_distance(s["A"], s["B"])
        return {"hausdorff": hd, "median": md, "voxels": [na, nb], "dice": ctx.dice(s["LA"], s["LB"])}
    if k == "train":
        net = s["net"]
        loss = net.train_step(s["x"], s["y"], 1e-4)
        return {"loss": loss.float(), "y": net.y, "dw": list(net.dw), "db": list(net.db)}
    return {"v0": W64.predict_v0(s["net"], s["I0"], s["I1"], _shape(c))}


# ------------------------------------------------------------------------------------------
# what a pass cannot do without

def _net_flops(n, B, cout=3):
    f, Lv = 0.0, len(W64.CHANS)
    for i, (co, ci, k) in enumerate(SG.conv_shapes(W64.CHANS, 2, cout)):
        lv = i // 2 if i < 2 * Lv else (Lv - 2 - (i - 2 * Lv) // 2 if i < 4 * Lv - 2 else 0)
        f += 2.0 * co * ci * k ** 3 * (n >> lv) ** 3
    return f * B


def _iteration(N, T, eb, rk4):
    """(bytes, flops) of one gradient-descent iteration: v read and written, the three images
    read; a trilinear lookup is 21 operations per value (two lookups of three values per step for
    the maps, nine of one value for the images and the residual; RK4 adds 9 values per map), the
    stencils and the update about 70, K two real FFTs per component, the regulariser 30."""
    fl = 21.0 * (6 + 9 + (18 if rk4 else 0)) + 70 + 30 + 3 * 2 * 2.5 * math.log2(N)
    return T * 3 * 2 * eb * N + 3 * eb * N, T * N * fl


def work(case):
    k = case["kind"]
    if k == "train":
        n, B = case["n"], case["batch"]
        nw = sum(co * (ci * kk ** 3 + 1) for co, ci, kk in SG.conv_shapes(W64.CHANS, 2, 3))
        return {"bytes": 4.0 * B * 5 * n ** 3 + 4.0 * B * 3 * n ** 3 + 7 * 4.0 * nw,
                "flops": 3 * _net_flops(n, B)}
    N = case["nx"] * case["ny"] * case["nz"]
    T = case.get("T", 10)
    if k == "step":
        b, f = _iteration(N, T, 2 if case["storage"] else 4, case["rk4"])
        return {"bytes": b * case["iters"], "flops": f * case["iters"]}
    if k == "register":
        b = f = 0.0
        for q in (4, 2, 1):
            n = math.prod(-(-case[a] // q) for a in ("nx", "ny", "nz"))
            bi, fi = _iteration(n, T, 4, False)
            b, f = b + bi * case["iterations"], f + fi * case["iterations"]
        return {"bytes": b + 4.0 * N, "flops": f}
    if k == "apply":      # v read; both maps; labels and two images in and out
        return {"bytes": 12.0 * T * N + 4.0 * N + 16.0 * N, "flops": T * N * 2 * 3 * 21.0 + 42.0 * N}
    if k == "grad":       # v read, the gradient written, three images
        return {"bytes": 24.0 * T * N + 12.0 * N, "flops": T * N * (63.0 + 63 + 60 + 60 + 60)}
    if k == "preprocess":  # the smoothed target and mask; two images and masks in, one image out
        return {"bytes": 5.0 * N + 20.0 * N, "flops": 30.0 * N}
    if k == "evaluate":   # two masks and two label maps read; separable distance transforms
        return {"bytes": 6.0 * N, "flops": 40.0 * N}
    return {"bytes": 8.0 * N + 12.0 * N + 2.4e6, "flops": _net_flops(64, 1) + 100.0 * N}


# ------------------------------------------------------------------------------------------
# the same results in 64 bits

def _corners(q, shape):
    """Lower corner indexes and fractions of the clamped lookup at q = (x, y, z)."""
    out = []
    for a, n in zip(q, (shape[2], shape[1], shape[0])):
        a = a.clamp(0.0, n - 1.0)
        i = a.detach().floor().long().clamp_(max=n - 2)
        out.append((i, a - i))
    return out


def _lookup(f, q):
    """Trilinear f ([..., z, y, x]) at q = (x, y, z) voxels, edges clamped."""
    sh = f.shape[-3:]
    (ix, tx), (iy, ty), (iz, tz) = _corners(q, sh)
    flat = f.reshape(f.shape[:-3] + (-1,))
    b = (iz * sh[1] + iy) * sh[2] + ix
    at = lambda o: flat[..., (b + o).reshape(-1)].reshape(f.shape[:-3] + b.shape)  # noqa: E731
    sx, sy, sz = 1, sh[2], sh[1] * sh[2]
    c = [at(z + y) + tx * (at(z + y + sx) - at(z + y)) for z in (0, sz) for y in (0, sy)]
    b0, b1 = c[0] + ty * (c[1] - c[0]), c[2] + ty * (c[3] - c[2])
    return b0 + tz * (b1 - b0)


def _grid(shape):
    z, y, x = torch.meshgrid(*(torch.arange(d, device=DEV, dtype=torch.float64) for d in shape),
                             indexing="ij")
    return [x, y, z]


def _diff(f, ax):
    """Central differences, one-sided at the faces, along array axis ax (voxel units)."""
    n, d = f.shape[ax], torch.empty_like(f)
    d.narrow(ax, 1, n - 2).copy_((f.narrow(ax, 2, n - 2) - f.narrow(ax, 0, n - 2)) / 2)
    d.narrow(ax, 0, 1).copy_(f.narrow(ax, 1, 1) - f.narrow(ax, 0, 1))
    d.narrow(ax, n - 1, 1).copy_(f.narrow(ax, n - 1, 1) - f.narrow(ax, n - 2, 1))
    return d


def _lap(f, h):
    r = 0.0
    for ax, d in ((-1, h[0]), (-2, h[1]), (-3, h[2])):
        r = r + (torch.roll(f, 1, ax) - 2 * f + torch.roll(f, -1, ax)) / d ** 2
    return r


def _K(f, h, alpha, gamma):
    sh = f.shape[-3:]
    lam = 0.0
    for k, (n, d) in enumerate(zip(sh, (h[2], h[1], h[0]))):
        m = n // 2 + 1 if k == 2 else n
        w = (2 - 2 * torch.cos(2 * math.pi * torch.arange(m, device=DEV, dtype=torch.float64) / n)) / d ** 2
        lam = lam + w.reshape([-1 if i == k else 1 for i in range(3)])
    return torch.fft.irfftn(torch.fft.rfftn(f, dim=(-3, -2, -1)) / (gamma + alpha * lam) ** 2, s=sh,
                            dim=(-3, -2, -1))


def _hv(h):
    return torch.tensor(h, dtype=torch.float64, device=DEV)[:, None, None, None]


def _move(v, sgn, h, T, x, rk4):
    """Displacement (voxels) of one time step along sgn * v."""
    f = v * (sgn / T) / _hv(h)
    if not rk4:
        return f
    at = lambda d: _lookup(f, [a + b for a, b in zip(x, d)])  # noqa: E731
    k2 = at(0.5 * f)
    k3 = at(0.5 * k2)
    k4 = at(k3)
    return (f + 2 * k2 + 2 * k3 + k4) / 6


def _next_map(u, d, x):
    return d if u is None else d + _lookup(u, [a + b for a, b in zip(x, d)])


def _exact_iteration(v, I0, I1, M, h, T, alpha, gamma, sigma, eps, rk4):
    """The updated v, and (total, reg, data, min det) of the given one."""
    shape = I0.shape
    x = _grid(shape)
    u, J1, Wt, dmin = None, [None] * T, [None] * T, math.inf
    for j in range(T - 1, -1, -1):
        u = _next_map(u, _move(v[j], 1, h, T, x, rk4), x)
        q = [a + b for a, b in zip(x, u)]
        D = [[_diff(u[r], 2 - e) + (1.0 if r == e else 0.0) for e in range(3)] for r in range(3)]
        det = D[0][0] * (D[1][1] * D[2][2] - D[1][2] * D[2][1]) - D[0][1] * (
            D[1][0] * D[2][2] - D[1][2] * D[2][0]) + D[0][2] * (D[1][0] * D[2][1] - D[1][1] * D[2][0])
        del D
        dmin = min(dmin, float(det.min()))
        jm = _lookup(torch.stack([I1, M]), q)
        J1[j], Wt[j] = jm[0], jm[1] * det
    reg = 0.0
    for j in range(T):
        reg += float(((gamma * v[j] - alpha * _lap(v[j], h)) ** 2).sum())
    u, new = None, torch.empty_like(v)
    for j in range(T):
        J0 = I0 if u is None else _lookup(I0, [a + b for a, b in zip(x, u)])
        r = (2 / sigma ** 2) * Wt[j] * (J0 - J1[j])
        b = torch.stack([r * _diff(J0, 2 - e) / h[e] for e in range(3)])
        u = _next_map(u, _move(v[j], -1, h, T, x, rk4), x)
        new[j] = v[j] - eps * (2 * v[j] - _K(b, h, alpha, gamma))
    J0 = _lookup(I0, [a + b for a, b in zip(x, u)])
    h3 = h[0] * h[1] * h[2]
    reg, data = reg * h3 / T, float((M * (J0 - I1) ** 2).sum()) * h3 / sigma ** 2
    return new, [reg + data, reg, data, dmin], J0


def _mean_down(a, q):
    for ax in range(3):
        n = -(-a.shape[ax] // q)
        i = torch.arange(n * q, device=DEV).clamp_(max=a.shape[ax] - 1)
        a = a.index_select(ax, i)
        a = a.reshape(a.shape[:ax] + (n, q) + a.shape[ax + 1:]).mean(ax + 1)
    return a


def _resample(f, shape, ratio):
    x = [((torch.arange(d, device=DEV, dtype=torch.float64) + 0.5) * r - 0.5)
         for d, r in zip(shape, ratio)]
    z, y, x = torch.meshgrid(*x, indexing="ij")
    return _lookup(f, [x, y, z])


def _network(x, w, b, n):
    """The encoder-decoder in float64 for one sample [cin][n^3] (weights [co][ci][k^3])."""
    Lv = len(W64.CHANS)

    def conv(i, a, relu=True):
        m = a.shape[-1]
        if w[i].shape[2] == 1:
            y = w[i][:, :, 0] @ a.reshape(a.shape[0], -1)
        else:
            p = torch.nn.functional.pad(a, (1,) * 6)
            y = 0.0
            for t in range(27):
                s = p[:, t // 9:t // 9 + m, t // 3 % 3:t // 3 % 3 + m, t % 3:t % 3 + m]
                y = y + w[i][:, :, t] @ s.reshape(a.shape[0], -1)
        y = (y + b[i][:, None]).reshape(-1, m, m, m)
        return y.relu() if relu else y

    skips, i, a = [], 0, x
    for lv in range(Lv):
        a = conv(i + 1, conv(i, a))
        i += 2
        if lv < Lv - 1:
            skips.append(a)
            a = torch.nn.functional.avg_pool3d(a[None], 2)[0]
    for lv in range(Lv - 2, -1, -1):
        up = a.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
        a = conv(i + 1, conv(i, torch.cat([up, skips[lv]])))
        i += 2
    return conv(i, a, False)


def _ball(m, r, grow):
    """Dilation (grow) or erosion of a bool mask by a ball, background beyond the grid."""
    if r == 0:
        return m
    p = torch.nn.functional.pad(m if grow else ~m, (r,) * 6, value=not grow)
    out = torch.zeros_like(m)
    Z, Y, X = m.shape
    for dz in range(-r, r + 1):
        for dy in range(-r, r + 1):
            for dx in range(-r, r + 1):
                if dx * dx + dy * dy + dz * dz <= r * r:
                    out |= p[r + dz:r + dz + Z, r + dy:r + dy + Y, r + dx:r + dx + X]
    return out if grow else ~out


def _nodes(img, m, bins, points):
    a = img[m].double()
    lo, hi = float(a.min()), float(a.max())
    w = (hi - lo) / bins
    c = torch.bincount(((a - lo) / w).floor().long().clamp_(0, bins - 1), minlength=bins).tolist()
    out = [lo]
    for k in range(1, points + 1):
        t, cum, b = k / (points + 1) * a.numel(), 0, 0
        while b < bins - 1 and cum + c[b] < t:
            cum += c[b]
            b += 1
        out.append(lo + w * (b + ((t - cum) / c[b] if c[b] else 0.0)))
    return out + [hi]


def _surface(m):
    p = torch.nn.functional.pad(m, (1,) * 6)
    Z, Y, X = m.shape
    inner = torch.ones_like(m)
    for d in ((0, 1, 1), (2, 1, 1), (1, 0, 1), (1, 2, 1), (1, 1, 0), (1, 1, 2)):
        inner &= p[d[0]:d[0] + Z, d[1]:d[1] + Y, d[2]:d[2] + X]
    return (m & ~inner).nonzero().double()


def exact(case, seed):
    k = case["kind"]
    if k in ("train", "predict"):
        if k == "train":
            net = prepare(case, seed)["net"]
        else:
            net = W64.load_net(W64.WEIGHTS)
        w = [t.double().reshape(t.shape[0], t.shape[1], -1) for t in net.wb]
        b = [t.double() for t in net.b]
    s = _inputs(case, seed)
    d = {n: t.double() for n, t in s.items() if torch.is_tensor(t) and t.is_floating_point()}
    if k == "train":
        w, b = [t.requires_grad_(True) for t in w], [t.requires_grad_(True) for t in b]
        ys, loss = [], 0.0
        for x, t in zip(d["x"], d["y"]):
            y = _network(x, w, b, case["n"])
            e = ((y - t) ** 2).sum()
            (e / d["y"].numel()).backward()
            ys.append(y.detach())
            loss += float(e.detach())
        shp = [t.shape for t in net.w]
        return {"loss": torch.tensor([loss], dtype=torch.float64), "y": torch.stack(ys),
                "dw": [t.grad.reshape(q) for t, q in zip(w, shp)], "db": [t.grad for t in b]}
    shape = _shape(case)
    if k == "predict":
        n = W64.NG
        x = torch.stack([_resample(d[m], (n,) * 3, [q / n for q in shape]) for m in ("I0", "I1")])
        with torch.no_grad():
            y = _network(x, w, b, n)
        y = _resample(y, shape, [n / q for q in shape])
        return {"v0": y * (net.out_scale * _hv((shape[2] / n, shape[1] / n, shape[0] / n)))}
    alpha, gamma, sigma, eps = (float(np.float32(a)) for a in (0.02, 1.0, 0.1, 1e-3))
    T = case.get("T", 10)
    if k == "step":
        h = (case["hx"], case["hy"], case["hz"])
        v = d["v"]
        for _ in range(case["iters"]):
            v, e, _ = _exact_iteration(v, d["I0"], d["I1"], d["M"], h, T, alpha, gamma, sigma, eps,
                                       case["rk4"])
        return {"v": v, "energy": np.array(e)}
    if k == "register":
        tr = []
        for q in (4, 2, 1):
            im = [_mean_down(d[a], q).float().double() for a in ("I0", "I1", "M")]
            sh = im[0].shape
            if q == 4:
                v = torch.zeros((T, 3) + tuple(sh), dtype=torch.float64, device=DEV)
            else:
                v = torch.stack([_resample(a, sh, [0.5] * 3) for a in v])
            for _ in range(case["iterations"]):
                v, e, _ = _exact_iteration(v, *im, (float(q),) * 3, T, alpha, gamma, sigma, eps, False)
                tr.append(e[0])
        J0 = _exact_iteration(v, *im, (1.0,) * 3, T, alpha, gamma, sigma, eps, False)[2]
        return {"v": v, "J0": J0, "energies": np.array(tr)}
    if k == "apply":
        x, u10, u01 = _grid(shape), None, None
        for j in range(T):
            u10 = _next_map(u10, _move(d["v"][j], -1, (1.0,) * 3, T, x, False), x)
            u01 = _next_map(u01, _move(d["v"][T - 1 - j], 1, (1.0,) * 3, T, x, False), x)
        return {"labels": None, "moved": _lookup(d["G0"], [a + b for a, b in zip(x, u10)]),
                "back": _lookup(d["G1"], [a + b for a, b in zip(x, u01)])}
    if k == "grad":
        v = d["v"].requires_grad_(True)
        x, u = _grid(shape), None
        reg = ((gamma * v - alpha * _lap(v, (1.0,) * 3)) ** 2).sum() / T
        for j in range(T):
            u = _next_map(u, _move(v[j], -1, (1.0,) * 3, T, x, False), x)
        J0 = _lookup(d["I0"], [a + b for a, b in zip(x, u)])
        E = reg + (d["M"] * (J0 - d["I1"]) ** 2).sum() / sigma ** 2
        E.backward()
        return {"grad": v.grad, "energy": E.detach()}
    if k == "preprocess":
        thr = float(np.float32(0.025))
        m = _ball(_ball(d["smooth"] > thr, case["r_open"], False), case["r_open"], True)
        m = _ball(_ball(m, case["r_close"], True), case["r_close"], False)
        m0 = s["I0"] > 0.5
        xs = _nodes(s["atlas"], m0, case["bins"], case["points"])
        ys = _nodes(s["raw"], m, case["bins"], case["points"])
        xs, ys = (torch.tensor(a, dtype=torch.float64, device=DEV) for a in (xs, ys))
        a = d["atlas"]
        i = torch.searchsorted(xs[1:-1].contiguous(), a.reshape(-1), right=True).reshape(a.shape)
        dx = xs[i + 1] - xs[i]
        r = ys[i] + (a - xs[i]) * torch.where(dx > 0, (ys[i + 1] - ys[i]) / dx, torch.zeros_like(dx))
        return {"mask": None, "matched": torch.where(m0, r, torch.zeros_like(r))}
    A, B = _surface(s["A"] > 0), _surface(s["B"] > 0)
    near = lambda p, q: torch.cat([((a[:, None] - q[None]) ** 2).sum(-1).amin(1) for a in p.split(256)])  # noqa: E731
    ab = torch.cat([near(A, B), near(B, A)]).sqrt().sort().values
    n = ab.numel()
    dice = []
    for l in range(1, 51):
        a, b = s["LA"] == l, s["LB"] == l
        na, nb, ni = int(a.sum()), int(b.sum()), int((a & b).sum())
        if na + nb:
            dice.append(2.0 * ni / (na + nb))
    return {"hausdorff": float(ab[-1]), "median": 0.5 * float(ab[(n - 1) // 2] + ab[n // 2]),
            "voxels": [None, None], "dice": sum(dice) / len(dice)}

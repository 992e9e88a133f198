"""The work whose speed is measured: what a simulation code, or the fit of the
learned correction, has this library do through its public entry points.

listed() and draw() give cases, prepare() makes what a caller holds before the
call, run() is one pass of the call, work() its unavoidable bytes and
operations and exact() its results in 64 bits by plain torch, from the method's
definition (include/colden.h, include/colden_learned.h) and without the library.

Kinds of case:
  step     the time step of a simulation on a uniform grid: new densities, then
           the columns and the screening factor (eager calls, or the captured
           graph), for a ray or a cone per direction
  heating  the same step feeding the heating rates: chi = <exp(-sigma N)> alone
           leaves the evaluation, then G0_eff, Gamma_UV and Gamma_CR per leaf
  amr      the time step on a mesh refined on density
  insitu   the columns with every shell seen from the oct's centre
  march    exact columns of random leaves, the learned correction's targets
  train    one Adam step of the learned correction on a minibatch, then the loss
           and gradient on held-out rows
  learned  the learned form of the columns
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1410_0624_gb300 import colden

PC_CM = 3.0857e18
BOX_CM = 10 * PC_CM
SIGMA = 2e-21                 # cm^2, chi = <exp(-SIGMA N)>
G0 = 1.7
AV = 1.0 / 1.87e21
SHIELD_K = 2.5
# standardisation of the learned inputs (logarithms of columns and densities)
MU_C, SINV_C, MU_N, SINV_N = 47.0, 0.4, 2.5, 0.5
LR, STEP0 = 1e-3, 1000        # the training step is one of a resumed run


def listed():
    return [
        # the smallest grid a one-zone or test-bed code steps: a handful of
        # launches, so latency and host time count; every output wanted
        dict(name="step_32_fp32_d12", kind="step", level=5, dirs="healpix1", precision="fp32", outputs="all",
             graph=False, cone=False),
        # the benchmark's step: 256^3 leaves, 48 directions, replayed as a graph
        dict(name="step_256_bf16_d48_graph", kind="step", level=8, dirs="healpix2", precision="bf16", outputs="nh",
             graph=True, cone=False),
        # the same step as the defaults of the binding give it: FP32, eager
        dict(name="step_256_fp32_d48", kind="step", level=8, dirs="healpix2", precision="fp32", outputs="nh",
             graph=False, cone=False),
        # cone-averaged weights on a direction set of the paper's tables
        dict(name="step_128_cone_fp32_d40", kind="step", level=7, dirs="mxn5x8", precision="fp32", outputs="nh",
             graph=False, cone=True),
        # the largest grid: only the rates leave the device-resident step
        dict(name="heating_512_bf16_d12", kind="heating", level=9, dirs="mxn3x4", precision="bf16"),
        # the benchmark's adaptive mesh (1024^3 effective), replayed as a graph
        dict(name="amr_1024_bf16_d48_graph", kind="amr", base=7, refine=3, mesh=2, dirs="healpix2", precision="bf16",
             graph=True),
        # a smaller adaptive mesh with the paper's widest direction set, defaults
        dict(name="amr_256_fp32_d84", kind="amr", base=6, refine=2, mesh=2, dirs="mxn7x12", precision="fp32",
             graph=False),
        # the variant without the two-level approximation, for accuracy studies
        dict(name="insitu_128_d40", kind="insitu", level=7, dirs="mxn5x8"),
        # targets of the learned correction: random leaves of a training field
        dict(name="march_128_d48", kind="march", level=7, dirs="healpix2", rows=262144),
        # a training step at the benchmark's batch and width
        dict(name="train_8192_d48_h128", kind="train", dirs="healpix2", hidden=128, batch=8192),
        # learned columns in the default precision, and in the fast form
        dict(name="learned_128_fp32_d48", kind="learned", level=7, dirs="healpix2", hidden=128, precision="fp32"),
        dict(name="learned_256_bf16_d48", kind="learned", level=8, dirs="healpix2", hidden=128, precision="bf16"),
    ]


def draw(rng):
    kind = rng.choices(["step", "heating", "amr", "insitu", "march", "train", "learned"], [7, 2, 4, 2, 2, 3, 2])[0]
    sets = ["axes", "healpix1", "healpix2", "mxn3x4", "mxn5x8", "mxn7x12", "mxn%dx%d" % (rng.randint(2, 8), rng.randint(3, 10))]
    dirs = rng.choice(sets)
    precision = rng.choice(["fp32", "bf16"])
    if kind == "step":
        cone = rng.random() < 0.2
        return dict(kind=kind, level=rng.randint(4, 8 if not cone else 7), dirs=dirs, precision=precision,
                    outputs=rng.choice(["nh", "all", "shield"]), graph=rng.random() < 0.5, cone=cone)
    if kind == "heating":
        return dict(kind=kind, level=rng.randint(5, 8), dirs=dirs, precision=precision)
    if kind == "amr":
        return dict(kind=kind, base=rng.randint(4, 6), refine=rng.randint(1, 3), mesh=rng.randint(1, 999), dirs=dirs,
                    precision=precision, graph=rng.random() < 0.5)
    if kind == "insitu":
        return dict(kind=kind, level=rng.randint(4, 7), dirs=dirs)
    if kind == "march":
        return dict(kind=kind, level=rng.randint(5, 8), dirs=dirs, rows=int(2 ** rng.uniform(10, 18)))
    if kind == "train":
        return dict(kind=kind, dirs=rng.choice(["healpix1", "healpix2", "mxn3x4", "mxn5x8"]),
                    hidden=rng.choice([32, 64, 96, 128, 192]), batch=int(2 ** rng.uniform(8, 13.5)))
    # the fast form serves 128 units and direction counts that are multiples of 8
    if precision == "bf16":
        return dict(kind=kind, level=rng.randint(5, 8), dirs=rng.choice(["healpix2", "mxn5x8", "mxn4x4", "mxn3x8"]),
                    hidden=128, precision=precision)
    return dict(kind=kind, level=rng.randint(4, 7), dirs=rng.choice(["healpix1", "healpix2", "mxn3x4", "mxn5x8"]),
                hidden=rng.choice([32, 64, 96, 128]), precision=precision)


# ---- inputs --------------------------------------------------------------------

def _scheme(dirs):
    if dirs.startswith("healpix"):
        return "healpix", int(dirs[7:]), 0
    if dirs == "axes":
        return "axes", 0, 0
    m, n = dirs[3:].split("x")
    return "mxn", int(m), int(n)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(level, seed):
    """Log-normal densities [z, y, x]: a Gaussian field of spectrum k^-11/3
    (mean 30 cm^-3, sigma_ln 2), or white (mean 10, sigma_ln 1.5) on the
    smallest grids."""
    n = 1 << level
    g = torch.randn((n, n, n), generator=_generator(seed), device="cuda")
    mean, sig = (10.0, 1.5) if level <= 5 else (30.0, 2.0)
    if level > 5:
        f = torch.fft.rfftn(g)
        k = torch.fft.fftfreq(n, device="cuda") * n
        kx = torch.fft.rfftfreq(n, device="cuda") * n
        k2 = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2).clamp_(min=1e-30)
        k2.pow_(-11.0 / 12.0)
        k2[0, 0, 0] = 0.0
        f *= k2
        del k2
        g = torch.fft.irfftn(f, s=(n, n, n))
        del f
        g -= g.mean()
        g /= g.std()
    g = torch.exp_(g.mul_(sig))
    return g.mul_(mean / float(g.double().mean() if n <= 256 else g.mean()))


def _amr_leaves(case, seed):
    """Leaves (level, ijk, rho) of a mesh refined where the mean over a
    level-(base + l) cell of its field exceeds 10^(2 + l) cm^-3, in the order of
    creation.  The case names the mesh; the seed moves the densities on it by
    about a tenth, as the steps between two refinements do."""
    base, lmax = case["base"], case["base"] + case["refine"]
    f = _field(lmax, case["mesh"])
    level, ijk, rho, refined = [], [], [], None
    for l in range(base, lmax + 1):
        m = torch.nn.functional.avg_pool3d(f[None, None], 1 << (lmax - l))[0, 0] if l < lmax else f
        here = torch.ones_like(m, dtype=torch.bool) if refined is None else \
            refined.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)
        refined = here & (m > 10.0 ** (2 + l - base)) if l < lmax else torch.zeros_like(here)
        leaf = here & ~refined
        at = torch.nonzero(leaf)
        level.append(torch.full((at.shape[0],), l, dtype=torch.int8, device="cuda"))
        ijk.append(at.flip(1).to(torch.int32))
        rho.append(m[leaf])
    rho = torch.cat(rho)
    rho *= torch.exp(0.1 * torch.randn(rho.shape, generator=_generator(seed), device="cuda"))
    return torch.cat(level), torch.cat(ijk), rho


def _gas(n, seed):
    """Temperature (K) and electron density (cm^-3) of n leaves."""
    g = _generator(seed + 7)
    T = torch.exp(torch.randn(n, generator=g, device="cuda") + math.log(100.0))
    return T, torch.exp(0.5 * torch.randn(n, generator=g, device="cuda") + math.log(0.02))


def _sizes(case):
    n_dir = {"healpix": lambda p, q: 12 * p * p, "axes": lambda p, q: 6, "mxn": lambda p, q: p * q}[
        _scheme(case["dirs"])[0]](*_scheme(case["dirs"])[1:])
    h = case.get("hidden", 0)
    n_in = 8 * n_dir + 1
    return n_dir, n_in, h, h * n_in + h + h * h + h + n_dir * h + n_dir


def _params(case, seed):
    """Initial weights U(+-1/sqrt(fan_in)), the last layer scaled to corrections
    of some tenths."""
    n_dir, n_in, h, _ = _sizes(case)
    rng = np.random.default_rng(seed + 3)
    parts = []
    for rows, fan, scale in ((h, n_in, 1.0), (h, h, 1.0), (n_dir, h, 0.5)):
        b = scale / math.sqrt(fan)
        parts += [rng.uniform(-b, b, rows * fan), rng.uniform(-b, b, rows)]
    return np.concatenate(parts).astype(np.float32)


def _moments(case, seed):
    """Adam moments of a run that has been going on for STEP0 steps."""
    rng = np.random.default_rng(seed + 4)
    p = _sizes(case)[3]
    return (1e-4 * rng.standard_normal(p)).astype(np.float32), \
        (1e-6 * rng.uniform(0.2, 1.0, p)).astype(np.float32)


def _net(case, seed):
    n_dir, n_in, h, p = _sizes(case)
    net = colden.Net(n_dir, h, _params(case, seed))
    mu = np.full(n_in, MU_C, np.float32)
    sinv = np.full(n_in, SINV_C, np.float32)
    mu[-1], sinv[-1] = MU_N, SINV_N
    train = case["kind"] == "train"
    m, v = _moments(case, seed) if train else (np.zeros(p, np.float32), np.zeros(p, np.float32))
    net.load_state(dict(params=_params(case, seed), mu=mu, sinv=sinv, adam_m=m, adam_v=v,
                        step=STEP0 if train else 0))
    return net


def _train_data(case, seed):
    """Rows of log columns and their targets, a minibatch and held-out rows."""
    n_dir, n_in, _, _ = _sizes(case)
    g = _generator(seed)
    n = 4 * case["batch"]
    x = MU_C + 2.5 * torch.randn((n, n_in), generator=g, device="cuda")
    x[:, -1] = MU_N + 2.0 * torch.randn(n, generator=g, device="cuda")
    y = 0.5 * torch.randn((n, n_dir), generator=g, device="cuda")
    perm = torch.randperm(n, generator=g, device="cuda")
    return x, y, perm[:case["batch"]].contiguous(), perm[case["batch"]:2 * case["batch"]].contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    new = lambda *shape: torch.empty(shape, device="cuda")  # noqa: E731
    if kind == "train":
        s["net"] = _net(case, seed)
        s["x"], s["y"], s["rows"], s["val"] = _train_data(case, seed)
        s["loss"], s["val_loss"], s["grad"] = new(1), new(1), new(_sizes(case)[3])
        return s
    scheme, p0, p1 = _scheme(case["dirs"])
    mode = colden.MODE_CONE if case.get("cone") else colden.MODE_INSITU if kind == "insitu" else colden.MODE_PREC
    s["geom"] = colden.precompute_geometry(scheme, p0, p1, mode=mode)
    nd = s["geom"].n_dir
    s["precision"] = colden.BF16 if case.get("precision") == "bf16" else colden.FP32
    if kind == "amr":
        level, ijk, s["rho"] = _amr_leaves(case, seed)
        s["tree"] = colden.build_tree_amr(case["base"], case["base"] + case["refine"], BOX_CM, level.cpu().numpy(),
                                          ijk.cpu().numpy(), s["rho"])
    else:
        s["rho"] = _field(case["level"], seed)
        s["tree"] = colden.build_tree_uniform(s["rho"], BOX_CM)
    n = s["tree"].n_leaf
    if kind == "march":
        s["leaves"] = torch.randint(n, (case["rows"],), generator=_generator(seed + 1), device="cuda")
        s["n_ray"] = new(case["rows"], nd)
        return s
    if kind == "heating":
        s["T"], s["n_e"] = _gas(n, seed)
        s["chi"], s["g0"], s["uv"], s["cr"] = new(n), new(n), new(n), new(n)
        return s
    outputs = case.get("outputs", "nh")
    s["n_h"] = new(n, nd) if outputs != "shield" else None
    s["a_v"] = new(n, nd) if outputs == "all" else None
    s["shield"] = new(n)
    if kind == "learned":
        s["net"] = _net(case, seed)
    if case.get("graph"):
        s["graph"] = colden.EvalGraph(s["tree"], s["geom"], rho=s["rho"], n_h=s["n_h"], a_v=s["a_v"],
                                      shield=s["shield"], precision=s["precision"])
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "train":
        s["net"].train_step(s["x"], s["y"], rows=s["rows"], lr=LR, loss=s["loss"])
        s["net"].loss_grad(s["x"], s["y"], s["val_loss"], grad=s["grad"], rows=s["val"])
        return {"loss": s["loss"], "val_loss": s["val_loss"], "grad": s["grad"]}
    tree, geom = s["tree"], s["geom"]
    if kind == "march":
        return {"n_ray": colden.raymarch(tree, geom, s["n_ray"], leaves=s["leaves"])}
    if kind == "heating":
        colden.tree_update(tree, s["rho"])
        colden.column_density(tree, geom, shield=s["chi"], precision=s["precision"], av_per_nh=1.0, shield_k=SIGMA)
        colden.heating(tree, s["chi"], s["T"], s["n_e"], G0=G0, g0_eff=s["g0"], gamma_uv=s["uv"], gamma_cr=s["cr"])
        return {"chi": s["chi"], "g0_eff": s["g0"], "gamma_uv": s["uv"], "gamma_cr": s["cr"]}
    if s.get("graph") is not None:
        s["graph"].launch()
    else:
        colden.tree_update(tree, s["rho"])
        colden.column_density(tree, geom, n_h=s["n_h"], a_v=s["a_v"], shield=s["shield"], precision=s["precision"],
                              net=s.get("net"))
    return {"n_h": s["n_h"], "a_v": s["a_v"], "shield": s["shield"]}


# ---- what a pass cannot do without ---------------------------------------------

def _amr_count(case):
    """Leaves and octs of the case's mesh."""
    level, _, _ = _amr_leaves(case, 0)
    n = int(level.numel())
    return n, n / 7.0


def work(case):
    kind = case["kind"]
    nd, n_in, h, p = _sizes(case)
    mlp = 2.0 * (h * n_in + h * h + h * nd)
    if kind == "train":
        b = case["batch"]
        # two forward and backward passes; rows in, gradient out, Adam's state
        # read and written
        return {"bytes": 2 * 4.0 * b * (n_in + nd) + 4.0 * (7 * p), "flops": 6.0 * b * mlp}
    if kind == "amr":
        n, octs = _amr_count(case)
    else:
        n = 8 ** case["level"]
        octs = n / 8
    if kind == "march":
        # about half the box's cells per ray and axis, summed over the axes
        cells = 0.75 * (1 << case["level"])
        return {"bytes": 4.0 * n + case["rows"] * (8.0 + 4.0 * nd), "flops": 2.0 * case["rows"] * nd * cells}
    # sparse sums: about ten cells per (oct, direction) and near shell, a
    # seventh more for the far shells of the ancestors, three siblings per
    # (leaf, direction)
    flops = 2.0 * nd * (octs * (30 + 10 / 7.0) + 3 * n)
    if kind == "insitu":
        flops = 2.0 * nd * (octs * 8 * case["level"] + 3 * n)
    if kind == "heating":
        return {"bytes": 4.0 * n * (1 + 3 + 3), "flops": flops}
    outs = {"nh": nd + 1, "all": 2 * nd + 1, "shield": 1}[case.get("outputs", "nh")]
    return {"bytes": 4.0 * n * (1 + outs), "flops": flops + (n * mlp if kind == "learned" else 0.0)}


# ---- the results in 64 bits ------------------------------------------------------

F64 = torch.float64


def _unit(v):
    v = np.where(np.abs(v) < 1e-14, 0.0, v)
    return v / np.linalg.norm(v, axis=-1, keepdims=True)


def _directions(dirs):
    """The direction set [nd, 3] (equations theta and phi, the six rays, or
    HEALPix ring centres)."""
    scheme, p, q = _scheme(dirs)
    if scheme == "axes":
        return np.array([[1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1]], float)
    out = []
    if scheme == "mxn":
        for m in range(1, p + 1):
            out += [(1.0 - (2.0 * m - 1.0) / p, 2 * math.pi * k / q) for k in range(q)]
    else:
        for r in range(1, 4 * p):
            c = min(r, 4 * p - r, p)
            if r < p or r > 3 * p:
                z = (1.0 - c * c / (3.0 * p * p)) * (1 if r < p else -1)
                out += [(z, 0.5 * math.pi * (j + 0.5) / c) for j in range(4 * c)]
            else:
                shift = 0.0 if (r - p) % 2 else 0.5
                out += [((4.0 * p - 2.0 * r) / (3.0 * p), 0.5 * math.pi * (j + 1 - shift) / p) for j in range(4 * p)]
    z, phi = np.array(out).T
    st = np.sqrt(np.maximum(0.0, 1.0 - z * z))
    return _unit(np.stack([st * np.cos(phi), st * np.sin(phi), z], 1))


def _rays(case):
    """The rays each direction's weights average over, [nd, n_sub, 3]."""
    u = _directions(case["dirs"])
    if not case.get("cone"):
        return torch.from_numpy(u[:, None]).cuda()
    nd, rings, az = u.shape[0], 4, 8
    ca = 1.0 - 2.0 / nd
    au = np.abs(u)
    e1 = _unit(np.cross(np.eye(3)[np.argmax(au <= au.min(1, keepdims=True) + 1e-9, axis=1)], u))
    e2 = np.cross(u, e1)
    out = []
    for r in range(rings):
        c = 1.0 - (r + 0.5) * (1.0 - ca) / rings
        for j in range(az):
            phi = 2 * math.pi * (j + 0.5 * (r & 1)) / az
            out.append(_unit(c * u + math.sqrt(max(0.0, 1 - c * c)) * (math.cos(phi) * e1 + math.sin(phi) * e2)))
    return torch.from_numpy(np.stack(out, 1)).cuda()


def _paths(p, lo, u):
    """Length of the rays p + s u, s >= 0, inside the unit cubes at lo (all broadcast, [..., 3])."""
    enter, leave = 0.0, 1e300
    out = False
    for a in range(3):
        zero = u[..., a] == 0
        s0 = (lo[..., a] - p[..., a]) / torch.where(zero, torch.ones_like(u[..., a]), u[..., a])
        s1 = (lo[..., a] + 1 - p[..., a]) / torch.where(zero, torch.ones_like(u[..., a]), u[..., a])
        near, far = torch.minimum(s0, s1), torch.maximum(s0, s1)
        outside = (p[..., a] < lo[..., a]) | (p[..., a] > lo[..., a] + 1)
        near = torch.where(zero, torch.full_like(near, -1e300), near)
        far = torch.where(zero, torch.full_like(far, 1e300), far)
        out = out | (zero & outside)
        enter = torch.clamp(near, min=0.0) if a == 0 else torch.maximum(enter, near)
        leave = far if a == 0 else torch.minimum(leave, far)
    return torch.where(out, torch.zeros_like(leave), torch.clamp(leave - enter, min=0.0))


def _octant_axes(o):
    return torch.stack([o & 1, (o >> 1) & 1, (o >> 2) & 1], -1)


def _stencil():
    s = torch.arange(216, device="cuda")
    return torch.stack([s % 6, (s // 6) % 6, s // 36], -1)


def _weights(rays):
    """K[t][cfg, 216, nd] of the shells 0, 1 and 2 or more levels above the
    receiving cell (t = 1, 2, 3), in units of the shell's cell."""
    nd, ns, _ = rays.shape
    cells = _stencil()
    tables = {}
    for t in (1, 2, 3):
        K = torch.empty((8 ** t, 216, nd), dtype=F64, device="cuda")
        step = max(1, int(6e7 // (216 * nd * ns)))
        for c0 in range(0, 8 ** t, step):
            cfg = torch.arange(c0, min(8 ** t, c0 + step), device="cuda")
            p = torch.full((cfg.numel(), 3), 2.0 + 2.0 ** -t, dtype=F64, device="cuda")
            for j in range(t):
                p += _octant_axes((cfg >> (3 * (t - 1 - j))) & 7).double() * 2.0 ** -j
            top = 2 + _octant_axes((cfg >> (3 * (t - 1))) & 7)
            gap = (cells[None] - top[:, None]).abs().amax(-1)
            inner = gap == 0 if t == 1 else gap <= 1
            k = _paths(p[:, None, None, None], cells.double()[None, :, None, None], rays[None, None]).mean(-1)
            K[c0:c0 + step] = k.masked_fill_(inner[..., None], 0.0)
        tables[t] = K
    return tables


def _local_weights(rays):
    o = _octant_axes(torch.arange(8, device="cuda")).double()
    return _paths(o[:, None, None, None] + 0.5, o[None, :, None, None], rays[None, None]).mean(-1)   # [t, s, nd]


def _levels(fine):
    """Volume means of the finest field (64 bits), finest level last."""
    out = [fine]
    while out[0].shape[0] > 1:
        out.insert(0, torch.nn.functional.avg_pool3d(out[0][None, None], 2)[0, 0])
    return out


def _shell(rho, ijk, k, t, K, box):
    """The shell of level k - t + 1 seen from the level-k cells ijk [n, 3]: [n, nd]."""
    l = k - t + 1
    pad = torch.nn.functional.pad(rho[l], (2,) * 6)
    side = pad.shape[0]
    cells = _stencil()
    off = (cells[:, 2] * side + cells[:, 1]) * side + cells[:, 0]
    P = ijk >> t
    at = 2 * P                                        # 2 (P - 1) in the padded frame
    flat = (at[:, 2] * side + at[:, 1]) * side + at[:, 0]
    cfg = torch.zeros_like(flat)
    for j in range(t):
        o = (ijk >> j) & 1
        cfg += (o[:, 0] + 2 * o[:, 1] + 4 * o[:, 2]) << (3 * j)
    order = torch.argsort(cfg)
    count = torch.bincount(cfg, minlength=8 ** t).tolist()
    out = torch.empty((ijk.shape[0], K.shape[2]), dtype=F64, device="cuda")
    pad, dx, i = pad.reshape(-1), box / 2 ** l, 0
    for c, n in enumerate(count):
        for b in range(i, i + n, 1 << 18):
            r = order[b:min(i + n, b + (1 << 18))]
            out[r] = (pad[flat[r][:, None] + off[None]] @ K[c]) * dx
        i += n
    return out


def _far(rho, ijk, k, K, box):
    """The far shells shared by everything under the level-k cells ijk."""
    if k < 3:
        return None
    own = _shell(rho, ijk, k, 3, K[3], box)
    par = ijk >> 1
    key, back = torch.unique((par[:, 2] << 40) | (par[:, 1] << 20) | par[:, 0], return_inverse=True)
    mask = (1 << 20) - 1
    up = _far(rho, torch.stack([key & mask, (key >> 20) & mask, key >> 40], -1), k - 1, K, box)
    return own if up is None else own.add_(up[back])


def _spread(v, to):
    """Bits of v, three apart."""
    out = torch.zeros_like(v)
    for b in range(to):
        out |= ((v >> b) & 1) << (3 * b)
    return out


def _morton_cells(level):
    m = torch.arange(8 ** level, device="cuda")
    out = torch.zeros((m.numel(), 3), dtype=torch.int64, device="cuda")
    for b in range(level):
        for a in range(3):
            out[:, a] |= ((m >> (3 * b + a)) & 1) << b
    return out


def _grid(rho, level, box, ijk):
    return rho[level][ijk[:, 2], ijk[:, 1], ijk[:, 0]]


def _insitu(rho, ijk, k, u, box):
    """Every shell of the octs ijk (level k) seen from their centres, [n, nd]:
    the segment of each ray between the shell's inner and outer boundary, cell
    by cell."""
    p = ((ijk.double() + 0.5) / 2 ** k)[:, None]                  # [n, 1, 3], box units
    up, dn = (u > 0)[None], (u < 0)[None]
    inv = torch.where(u != 0, 1.0 / torch.where(u != 0, u, torch.ones_like(u)), torch.zeros_like(u))[None]
    inf = torch.full((1, 1, 1), math.inf, dtype=F64, device="cuda")

    def leave(lo, hi):
        t = torch.where(up, (hi - p) * inv, torch.where(dn, (lo - p) * inv, inf))
        return t.amin(-1)

    total = 0.0
    for l in range(k, 0, -1):
        n = 2 ** l
        a = ijk >> (k - l)
        m = a >> 1
        ilo, ihi = (a, a + 1) if l == k else ((a - 1).clamp(min=0), (a + 2).clamp(max=n))
        f = lambda v: v.double()[:, None] / n  # noqa: E731
        t0 = leave(f(ilo), f(ihi))
        t1 = leave(f((2 * (m - 1)).clamp(min=0)), f((2 * (m + 2)).clamp(max=n)))
        q = (p + t0[..., None] * u[None]) * n
        c = torch.where(dn, torch.ceil(q) - 1, torch.floor(q)).clamp_(0, n - 1)
        t, sum_ = t0, torch.zeros_like(t0)
        for _ in range(24):
            nxt = torch.where(up, ((c + 1) / n - p) * inv, torch.where(dn, (c / n - p) * inv, inf))
            tn, ax = nxt.min(-1)
            live = (t < t1) & ((c >= 0) & (c < n)).all(-1)
            if not bool(live.any()):
                break
            ci = c.clamp(0, n - 1).long()
            v = rho[l].reshape(-1)[(ci[..., 2] * n + ci[..., 1]) * n + ci[..., 0]]
            sum_ += torch.where(live, v * (torch.minimum(tn, t1) - t), torch.zeros_like(t))
            t = torch.where(live, torch.minimum(tn, t1), t)
            c.scatter_add_(-1, ax[..., None], torch.where(up, 1.0, torch.where(dn, -1.0, 0.0)).to(F64).expand_as(c)
                           .gather(-1, ax[..., None]))
        total = total + sum_
    return total * box


def _external(case, rho, ijk, k, K, rays):
    """The external column of the octs ijk of level k, [n, nd]."""
    if case["kind"] == "insitu":
        return torch.cat([_insitu(rho, c, k, rays[:, 0], BOX_CM) for c in ijk.split(1 << 16)])
    E = torch.zeros((ijk.shape[0], rays.shape[0]), dtype=F64, device="cuda")
    for t in range(1, min(3, k) + 1):
        E += _shell(rho, ijk, k, t, K[t], BOX_CM)
    par = ijk >> 1
    if k - 1 >= 3:
        key, back = torch.unique((par[:, 2] << 40) | (par[:, 1] << 20) | par[:, 0], return_inverse=True)
        mask = (1 << 20) - 1
        E += _far(rho, torch.stack([key & mask, (key >> 20) & mask, key >> 40], -1), k - 1, K, BOX_CM)[back]
    return E


def _columns(E, rho8, kloc, dx):
    """[n, 8, nd]: the columns of the children of octs with external column E."""
    return E[:, None] + dx * torch.einsum("os,tsd->otd", rho8, kloc)


def _outputs(case, N):
    """The outputs of an evaluation whose columns are the blocks N yields."""
    nh, av, sh = [], [], []
    outputs = case.get("outputs", "nh")
    for n in N:
        sh.append(torch.exp(-SHIELD_K * AV * n).mean(-1))
        if outputs != "shield":
            nh.append(n)
        if outputs == "all":
            av.append(n * AV)
    return {"n_h": torch.cat(nh) if nh else None, "a_v": torch.cat(av) if av else None, "shield": torch.cat(sh)}


def _exact_uniform(case, seed):
    L = case["level"]
    rho = _levels(_field(L, seed).double())
    rays = _rays(case)
    K = _weights(rays) if case["kind"] != "insitu" else None
    kloc = _local_weights(rays)
    octs = _morton_cells(L - 1)
    E = _external(case, rho, octs, L - 1, K, rays)
    child = _octant_axes(torch.arange(8, device="cuda"))
    rho8 = _grid(rho, L, BOX_CM, (2 * octs[:, None] + child).reshape(-1, 3)).reshape(-1, 8)
    del octs
    dx = BOX_CM / 2 ** L
    cut = 1 << 17
    N = (_columns(E[i:i + cut], rho8[i:i + cut], kloc, dx).reshape(-1, rays.shape[0])
         for i in range(0, E.shape[0], cut))
    if case["kind"] != "heating":
        return _outputs(case, N)
    chi = torch.cat([torch.exp(-SIGMA * n).mean(-1) for n in N])
    n = rho8.reshape(-1)
    T, n_e = (v.double() for v in _gas(n.numel(), seed))
    g0 = chi * G0
    x = g0 * T.sqrt() / n_e
    eps = 4.9e-2 / (1 + (x / 1925.0) ** 0.73) + 3.7e-2 * (T / 1e4) ** 0.7 / (1 + x / 5000.0)
    return {"chi": chi, "g0_eff": g0, "gamma_uv": 1e-24 * eps * g0 * n, "gamma_cr": 1e-27 * n}


def _exact_amr(case, seed):
    level, ijk, rho_leaf = _amr_leaves(case, seed)
    base, lmax = case["base"], case["base"] + case["refine"]
    lv, ijk, rl = level.long(), ijk.long(), rho_leaf.double()
    grid = None
    for l in range(base, lmax + 1):
        n = 2 ** l
        grid = torch.zeros((n, n, n), dtype=F64, device="cuda") if grid is None else \
            grid.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)
        c = ijk[lv == l]
        grid[c[:, 2], c[:, 1], c[:, 0]] = rl[lv == l]
    rho = _levels(grid)
    del grid
    key = _spread(ijk[:, 0], lmax) | (_spread(ijk[:, 1], lmax) << 1) | (_spread(ijk[:, 2], lmax) << 2)
    order = torch.argsort(key << (3 * (lmax - lv)))
    row = torch.empty_like(order)
    row[order] = torch.arange(order.numel(), device="cuda")
    rays = _rays(case)
    K, kloc = _weights(rays), _local_weights(rays)
    N = torch.empty((order.numel(), rays.shape[0]), dtype=F64, device="cuda")
    child = _octant_axes(torch.arange(8, device="cuda"))
    for l in range(base, lmax + 1):
        here = torch.nonzero(lv == l)[:, 0]
        if here.numel() == 0:
            continue
        par = ijk[here] >> 1
        okey, back = torch.unique((par[:, 2] << 40) | (par[:, 1] << 20) | par[:, 0], return_inverse=True)
        mask = (1 << 20) - 1
        octs = torch.stack([okey & mask, (okey >> 20) & mask, okey >> 40], -1)
        E = _external(case, rho, octs, l - 1, K, rays)
        rho8 = _grid(rho, l, BOX_CM, (2 * octs[:, None] + child).reshape(-1, 3)).reshape(-1, 8)
        o = ijk[here] & 1
        t = o[:, 0] + 2 * o[:, 1] + 4 * o[:, 2]
        for i in range(8):
            mine = t == i
            N[row[here[mine]]] = E[back[mine]] + BOX_CM / 2 ** l * (rho8[back[mine]] @ kloc[i])
    return _outputs(case, N.split(1 << 20))


def _exact_march(case, seed):
    """Parallel rays from cell centres cross the same cells: one list of
    crossings per direction serves every leaf."""
    L = case["level"]
    n = 2 ** L
    rho = torch.nn.functional.pad(_field(L, seed).double(), (1,) * 6).reshape(-1)
    s = n + 2
    leaves = torch.randint(8 ** L, (case["rows"],), generator=_generator(seed + 1), device="cuda")
    start = torch.zeros((leaves.numel(), 3), dtype=torch.int64, device="cuda")
    for b in range(L):
        for a in range(3):
            start[:, a] |= ((leaves >> (3 * b + a)) & 1) << b
    u = torch.from_numpy(_directions(case["dirs"])).cuda()
    j = torch.arange(n, device="cuda").double() + 0.5
    t = torch.where(u[..., None] != 0, j / u.abs().clamp(min=1e-300)[..., None], torch.full_like(j, math.inf))
    when, at = t.reshape(u.shape[0], -1).sort(-1)                     # [nd, 3 n]
    axis = at // n
    out = torch.empty((leaves.numel(), u.shape[0]), dtype=F64, device="cuda")
    strides = torch.tensor([1, s, s * s], device="cuda")
    step = torch.sign(u).long()
    for lo in range(0, leaves.numel(), 1 << 16):
        c = start[lo:lo + (1 << 16)]
        pos = c[:, None].expand(-1, u.shape[0], -1).clone()
        sum_ = torch.zeros((c.shape[0], u.shape[0]), dtype=F64, device="cuda")
        last = torch.zeros(u.shape[0], dtype=F64, device="cuda")
        alive = torch.ones_like(sum_, dtype=torch.bool)
        for i in range(when.shape[1]):
            if i % 64 == 0 and not bool(alive.any()):
                break
            now = torch.where(torch.isinf(when[:, i]), last, when[:, i])
            flat = ((pos + 1).clamp(0, s - 1) * strides).sum(-1)
            sum_ += torch.where(alive, rho[flat], torch.zeros_like(sum_)) * (now - last)
            ax = axis[:, i]
            move = step.gather(1, ax[:, None])[:, 0]
            pos.scatter_add_(-1, ax[None, :, None].expand(pos.shape[0], -1, 1),
                             move[None, :, None].expand(pos.shape[0], -1, 1))
            q = pos.gather(-1, ax[None, :, None].expand(pos.shape[0], -1, 1))[..., 0]
            alive &= (q >= 0) & (q < n)
            last = now
        out[lo:lo + (1 << 16)] = sum_
    return {"n_ray": out * (BOX_CM / n)}


def _layers(p, case):
    nd, n_in, h, _ = _sizes(case)
    sizes = [h * n_in, h, h * h, h, nd * h, nd]
    W1, b1, W2, b2, W3, b3 = p.split(sizes)
    return W1.view(h, n_in), b1, W2.view(h, h), b2, W3.view(nd, h), b3


def _delta(p, x, case):
    W1, b1, W2, b2, W3, b3 = _layers(p, case)
    gelu = lambda z: 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))  # noqa: E731
    # the standardisation's constants as the 32-bit state holds them
    f = lambda v: float(np.float32(v))  # noqa: E731
    u = torch.cat([(x[:, :-1] - f(MU_C)) * f(SINV_C), (x[:, -1:] - f(MU_N)) * f(SINV_N)], 1).clamp(-8, 8)
    return gelu(gelu(u @ W1.T + b1) @ W2.T + b2) @ W3.T + b3


def _exact_train(case, seed):
    x, y, rows, val = _train_data(case, seed)
    p = torch.from_numpy(_params(case, seed)).cuda().double().requires_grad_()

    def loss(p, r):
        return ((_delta(p, x[r].double(), case) - y[r].double()) ** 2).mean()

    first = loss(p, rows)
    g, = torch.autograd.grad(first, p)
    m, v = (torch.from_numpy(a).cuda().double() for a in _moments(case, seed))
    m, v, t = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g, STEP0 + 1
    q = (p - LR * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)).detach().requires_grad_()
    second = loss(q, val)
    grad, = torch.autograd.grad(second, q)
    return {"loss": first.detach().reshape(1), "val_loss": second.detach().reshape(1), "grad": grad}


def _exact_learned(case, seed):
    L = case["level"]
    rho = _levels(_field(L, seed).double())
    rays = _rays(case)
    K, kloc = _weights(rays), _local_weights(rays)
    octs = _morton_cells(L - 1)
    k = L - 1
    near = {t: _shell(rho, octs, k, t, K[t], BOX_CM) for t in range(1, min(3, k) + 1)}
    far = {j: _shell(rho, _morton_cells(j), j, 3, K[3], BOX_CM) for j in range(3, L - 1)}
    child = _octant_axes(torch.arange(8, device="cuda"))
    rho8 = _grid(rho, L, BOX_CM, (2 * octs[:, None] + child).reshape(-1, 3)).reshape(-1, 8)
    nd = rays.shape[0]
    p = torch.from_numpy(_params(case, seed)).cuda().double()
    dx = BOX_CM / 2 ** L

    def blocks():
        cut = 1 << 15
        for i in range(0, octs.shape[0], cut):
            o = torch.arange(i, min(i + cut, octs.shape[0]), device="cuda")
            c = torch.zeros((o.numel(), 8, 8, nd), dtype=F64, device="cuda")      # oct, leaf, slot, direction
            c[:, :, 0] = _columns(torch.zeros((o.numel(), nd), dtype=F64, device="cuda"), rho8[o], kloc, dx)
            for t, v in near.items():
                c[:, :, t] = v[o][:, None]
            for j, v in far.items():
                c[:, :, min(7, L - j + 2)] += v[o >> (3 * (k - j))][:, None]
            c = c.reshape(-1, 8, nd)
            x = torch.cat([c.clamp(min=1e16).log().reshape(-1, 8 * nd),
                           rho8[o].reshape(-1, 1).clamp(min=1e-10).log()], 1)
            yield c.sum(1) * torch.exp(_delta(p, x, case))

    return _outputs(case, blocks())


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "march":
        return _exact_march(case, seed)
    if kind == "amr":
        return _exact_amr(case, seed)
    if kind == "learned":
        return _exact_learned(case, seed)
    return _exact_uniform(case, seed)

"""The learned correction through the C ABI against the FP64 oracle
(oracle/learned.py, oracle.c's ray-marcher and per-level sums).

Tolerances.
  * Ray-marcher (FP32 DDA, boundaries recomputed per crossing): each crossing
    time carries one or two roundings (2^-24 relative of t <= 1.8 * 2^L
    cells), the segment differences telescope, and the FP32 sum of <= 3 * 2^L
    positive terms adds <= 3 * 2^L * 2^-24 relative in the worst case
    (~1e-5 at 512^3, ~1e-6 in practice): held to 2e-5 relative.
  * Features: every slot is a sum of positive FP32 terms (<= 1e-5 relative,
    as the plain FP32 path); ln is 1-Lipschitz in the relative error and
    ln max(., floor) cannot enlarge it: x is held to 3e-5 absolute, N_tree to
    1e-5 relative.
  * Network (FP32 GEMMs, K <= 385): delta to 1e-4 absolute; gradients to
    1e-4 of the largest component; the loss to 1e-5 relative.
  * Learned N = N_tree exp(delta): relative error = error of N_tree + absolute
    error of delta: held to 1e-4 relative; shield to 2e-5 absolute.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from oracle import learned as ol
from paper_1410_0624_gb300 import colden, synth

PC = synth.PC_CM
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    colden.load(build_if_missing=True)


def _compact(v):
    v = v.astype(np.uint64) & np.uint64(0x1249249249249249)
    for sh, mask in ((2, 0x10c30c30c30c30c3), (4, 0x100f00f00f00f00f), (8, 0x1f0000ff0000ff),
                     (16, 0x1f00000000ffff), (32, 0x1fffff)):
        v = (v ^ (v >> np.uint64(sh))) & np.uint64(mask)
    return v.astype(np.int64)


def _ijk_of(m):
    m = np.asarray(m, dtype=np.uint64)
    return np.stack([_compact(m), _compact(m >> np.uint64(1)), _compact(m >> np.uint64(2))], axis=1)


def _field(L, seed, sigma=2.0, mean=30.0):
    if L >= 8:
        return synth.lognormal_grf_torch(1 << L, mean, sigma, seed, device="cuda").contiguous()
    return torch.from_numpy(synth.lognormal_grf(1 << L, mean, sigma, seed)).cuda()


def _setup(L, seed, dirs=("healpix", 2, 0, None), box=10 * PC):
    rho = _field(L, seed)
    tree = colden.build_tree_uniform(rho, box)
    geom = colden.precompute_geometry(dirs[0], dirs[1], dirs[2], dirs=dirs[3])
    T = oracle.Tree.uniform(rho.cpu().numpy(), box)
    return rho, tree, geom, T


def _sample(n_leaf, k, seed):
    rng = np.random.default_rng(seed)
    m = rng.choice(n_leaf, size=min(k, n_leaf), replace=False)
    m[:2] = [0, n_leaf - 1]                      # box corners
    return np.sort(m)


def _oracle_slots(T, L, dirs, m):
    ijk = _ijk_of(m)
    _, pl = T.column_density(dirs, np.full(len(m), L), ijk, per_level=L)
    return ol.slots_from_levels(pl)


# ---------------------------------------------------------------------------
# Ray-marcher
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("L,dset", [(4, ("healpix", 2, 0, None)), (5, ("axes", 0, 0, None)),
                                    (7, ("healpix", 2, 0, None)), (9, ("healpix", 2, 0, None)),
                                    (6, ("custom", 0, 0, np.random.default_rng(11).normal(size=(9, 3))))])
def test_raymarch_matches_oracle(L, dset):
    _, tree, geom, T = _setup(L, 40 + L, dset)
    m = _sample(tree.n_leaf, 400 if L < 9 else 120, L)
    out = torch.full((len(m), geom.n_dir), -1.0, device="cuda")
    colden.raymarch(tree, geom, out, leaves=torch.from_numpy(m).cuda())
    got = out.cpu().numpy().astype(np.float64)
    want = T.raymarch(geom.dirs, np.full(len(m), L), _ijk_of(m))
    assert np.all(want > 0)
    assert np.max(np.abs(got - want) / want) < 2e-5


def test_raymarch_uniform_density_is_distance_to_edge():
    L, n0, box = 5, 3.0, 10 * PC
    tree = colden.build_tree_uniform(torch.full((32, 32, 32), n0, device="cuda"), box)
    geom = colden.precompute_geometry("healpix", 2)
    out = torch.zeros((tree.n_leaf, geom.n_dir), device="cuda")
    colden.raymarch(tree, geom, out)
    got = out.cpu().numpy().astype(np.float64)
    ijk = _ijk_of(np.arange(tree.n_leaf))
    x0 = (ijk + 0.5) * box / 32
    d = geom.dirs
    with np.errstate(divide="ignore"):
        tx = np.where(d[None, :, 0] > 0, (box - x0[:, None, 0]) / d[None, :, 0],
                      np.where(d[None, :, 0] < 0, -x0[:, None, 0] / d[None, :, 0], np.inf))
        ty = np.where(d[None, :, 1] > 0, (box - x0[:, None, 1]) / d[None, :, 1],
                      np.where(d[None, :, 1] < 0, -x0[:, None, 1] / d[None, :, 1], np.inf))
        tz = np.where(d[None, :, 2] > 0, (box - x0[:, None, 2]) / d[None, :, 2],
                      np.where(d[None, :, 2] < 0, -x0[:, None, 2] / d[None, :, 2], np.inf))
    want = n0 * np.minimum(np.minimum(tx, ty), tz)
    assert np.max(np.abs(got - want) / want) < 2e-6


# ---------------------------------------------------------------------------
# Features
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("L,k", [(3, 512), (5, 600), (8, 300), (9, 100)])
def test_features_match_oracle(L, k):
    rho, tree, geom, T = _setup(L, 60 + L)
    m = _sample(tree.n_leaf, k, 100 + L)
    nd = geom.n_dir
    x = torch.full((len(m), 8 * nd + 1), -7.0, device="cuda")
    nt = torch.full((len(m), nd), -7.0, device="cuda")
    colden.learned_features(tree, geom, x, nt, leaves=torch.from_numpy(m).cuda())
    slots = _oracle_slots(T, L, geom.dirs, m)
    rho_m = rho.reshape(-1).cpu().numpy()        # row-major [z, y, x]
    ijk = _ijk_of(m)
    n_leaf_vals = rho_m[(ijk[:, 2] * (1 << L) + ijk[:, 1]) * (1 << L) + ijk[:, 0]]
    want_x = ol.features(slots, n_leaf_vals)
    want_nt = ol.tree_total(slots)
    gx = x.cpu().numpy().astype(np.float64)
    gnt = nt.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(gx - want_x)) < 3e-5
    assert np.max(np.abs(gnt - want_nt) / want_nt) < 1e-5
    # the plain method's column equals the sum of the slots
    plain = torch.zeros(tree.n_leaf * nd, device="cuda")
    colden.column_density(tree, geom, n_h=plain)
    p = plain.reshape(-1, nd)[torch.from_numpy(m).cuda()].cpu().numpy().astype(np.float64)
    assert np.max(np.abs(p - gnt) / gnt) < 2e-5


def test_features_see_tree_update():
    rho, tree, geom, T = _setup(5, 71)
    nd = geom.n_dir
    x1 = torch.zeros((tree.n_leaf, 8 * nd + 1), device="cuda")
    colden.learned_features(tree, geom, x1)
    colden.tree_update(tree, rho * 2.0)
    x2 = torch.zeros_like(x1)
    colden.learned_features(tree, geom, x2)
    d = (x2 - x1).cpu().numpy()
    # every slot above the floor and ln n move by ln 2
    above = x1.cpu().numpy() > np.log(1e16) + 1.0
    assert np.allclose(d[above], np.log(2.0), atol=3e-5)


# ---------------------------------------------------------------------------
# Network: forward, gradient, Adam, checkpoint
# ---------------------------------------------------------------------------

def _net(nd=48, H=128, seed=1, scale=1.0):
    p = synth.mlp_init(nd, H, seed, out_scale=scale)
    return colden.Net(nd, H, p), p.astype(np.float64)


@pytest.mark.parametrize("nd,H,n", [(48, 128, 1000), (12, 40, 77), (3, 5, 1)])
def test_normaliser_and_forward_match_oracle(nd, H, n):
    net, p = _net(nd, H)
    x_np = synth.mlp_inputs(n, 8 * nd + 1, seed=nd + n)
    x = torch.from_numpy(x_np).cuda()
    net.fit_normaliser(x)
    st = net.state()
    mu, sinv = ol.normaliser(x_np.astype(np.float64))
    assert np.allclose(st["mu"], mu, rtol=1e-6, atol=0)
    assert np.allclose(st["sinv"], sinv, rtol=1e-5, atol=0)
    delta = torch.zeros((n, nd), device="cuda")
    net.forward(x, delta)
    want, _ = ol.forward(ol.unpack(p, nd, H), mu, sinv, x_np.astype(np.float64))
    assert np.max(np.abs(delta.cpu().numpy() - want)) < 1e-4


def _batch(nd, B, seed):
    x_np = synth.mlp_inputs(B, 8 * nd + 1, seed=seed)
    y_np = (0.3 * np.random.default_rng(seed + 1).standard_normal((B, nd))).astype(np.float32)
    return x_np, y_np


@pytest.mark.parametrize("nd,H,B", [(48, 128, 300), (12, 40, 1), (48, 128, 5000)])
def test_loss_gradient_match_oracle(nd, H, B):
    net, p = _net(nd, H, seed=2)
    x_np, y_np = _batch(nd, B, seed=B)
    x, y = torch.from_numpy(x_np).cuda(), torch.from_numpy(y_np).cuda()
    mu, sinv = ol.normaliser(x_np.astype(np.float64))
    st = net.state()
    st["mu"], st["sinv"] = mu.astype(np.float32), sinv.astype(np.float32)
    net.load_state(st)
    loss = torch.zeros(1, device="cuda")
    grad = torch.zeros(net.n_params, device="cuda")
    net.loss_grad(x, y, loss, grad)
    L_or, g_or = ol.loss_grad(ol.unpack(p, nd, H), st["mu"].astype(np.float64), st["sinv"].astype(np.float64),
                              x_np.astype(np.float64), y_np.astype(np.float64))
    g_or = ol.pack(g_or)
    assert loss.item() == pytest.approx(L_or, rel=1e-5)
    g = grad.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(g - g_or)) < 1e-4 * np.max(np.abs(g_or))
    # repeatable to the bit
    grad2 = torch.zeros_like(grad)
    net.loss_grad(x, y, loss, grad2)
    assert torch.equal(grad, grad2)


def test_row_gather_equals_explicit_batch():
    nd, H = 12, 32
    net, _ = _net(nd, H, seed=3)
    x_np, y_np = _batch(nd, 500, seed=9)
    x, y = torch.from_numpy(x_np).cuda(), torch.from_numpy(y_np).cuda()
    rows = torch.tensor([5, 499, 0, 17, 17, 250], device="cuda", dtype=torch.int64)
    l1, g1 = torch.zeros(1, device="cuda"), torch.zeros(net.n_params, device="cuda")
    net.loss_grad(x, y, l1, g1, rows=rows)
    l2, g2 = torch.zeros(1, device="cuda"), torch.zeros(net.n_params, device="cuda")
    net.loss_grad(x[rows].contiguous(), y[rows].contiguous(), l2, g2)
    assert torch.equal(l1, l2) and torch.equal(g1, g2)


def test_adam_steps_match_oracle():
    nd, H, B = 48, 128, 256
    net, p = _net(nd, H, seed=4)
    x_np, y_np = _batch(nd, B, seed=44)
    x, y = torch.from_numpy(x_np).cuda(), torch.from_numpy(y_np).cuda()
    mu, sinv = ol.normaliser(x_np.astype(np.float64))
    st = net.state()
    st["mu"], st["sinv"] = mu.astype(np.float32), sinv.astype(np.float32)
    net.load_state(st)
    mu64, sinv64 = st["mu"].astype(np.float64), st["sinv"].astype(np.float64)
    m = np.zeros_like(p)
    v = np.zeros_like(p)
    q = p.copy()
    lr = 1e-3
    for t in range(1, 4):
        net.train_step(x, y, lr=lr)
        _, g = ol.loss_grad(ol.unpack(q, nd, H), mu64, sinv64, x_np.astype(np.float64), y_np.astype(np.float64))
        g = ol.pack(g)
        q_new, m, v = ol.adam(q, g, m, v, t, lr)
        got = net.state()["params"].astype(np.float64)
        # parameters whose gradient is well above FP32 noise follow the oracle
        sure = np.abs(g) > 1e-3 * np.max(np.abs(g))
        assert np.max(np.abs(got - q_new)[sure]) < 2e-2 * lr * t
        assert np.max(np.abs(got - q_new)) <= 7.0 * lr * t
        q = q_new
    assert net.state()["step"] == 3


def test_checkpoint_roundtrip_and_resume(tmp_path):
    nd, H = 12, 32
    x_np, y_np = _batch(nd, 2048, seed=5)
    x, y = torch.from_numpy(x_np).cuda(), torch.from_numpy(y_np).cuda()
    a, _ = _net(nd, H, seed=6)
    a.fit_normaliser(x)
    la = colden.train(a, x, y, steps=20, batch=256, seed=1)
    path = str(tmp_path / "net.npz")
    a.save(path)
    b = colden.Net.load(path)
    sa, sb = a.state(), b.state()
    for k in ("params", "mu", "sinv", "adam_m", "adam_v"):
        assert np.array_equal(sa[k], sb[k])
    assert sb["step"] == 20
    # continuing both gives identical weights (training is deterministic)
    colden.train(a, x, y, steps=5, batch=256, seed=2)
    colden.train(b, x, y, steps=5, batch=256, seed=2)
    assert np.array_equal(a.state()["params"], b.state()["params"])
    assert np.all(np.isfinite(la)) and la[-1] < la[0]


# ---------------------------------------------------------------------------
# Learned column density (FP32) against the oracle chain
# ---------------------------------------------------------------------------

def _learned_case(L, seed, k, nd_set=("healpix", 2, 0, None), precision=colden.FP32, hidden=64):
    rho, tree, geom, T = _setup(L, seed, nd_set)
    nd = geom.n_dir
    net, p = _net(nd, hidden, seed=seed, scale=0.2)
    # the standardisation comes from the oracle's own features of a sample
    ms = _sample(tree.n_leaf, 2000, seed + 1)
    slots_s = _oracle_slots(T, L, geom.dirs, ms)
    rho_m = rho.reshape(-1).cpu().numpy().astype(np.float64)
    ij = _ijk_of(ms)
    n_s = rho_m[(ij[:, 2] * (1 << L) + ij[:, 1]) * (1 << L) + ij[:, 0]]
    mu, sinv = ol.normaliser(ol.features(slots_s, n_s))
    st = net.state()
    st["mu"], st["sinv"] = mu.astype(np.float32), sinv.astype(np.float32)
    net.load_state(st)
    n_h = torch.full((tree.n_leaf * nd,), -1.0, device="cuda")
    sh = torch.full((tree.n_leaf,), -1.0, device="cuda")
    colden.column_density(tree, geom, n_h=n_h, shield=sh, net=net, precision=precision)
    torch.cuda.synchronize()
    colden.device_status()
    m = _sample(tree.n_leaf, k, seed + 2)
    slots = _oracle_slots(T, L, geom.dirs, m)
    ij = _ijk_of(m)
    nv = rho_m[(ij[:, 2] * (1 << L) + ij[:, 1]) * (1 << L) + ij[:, 0]]
    delta, _ = ol.forward(ol.unpack(p, nd, hidden), st["mu"].astype(np.float64), st["sinv"].astype(np.float64),
                          ol.features(slots, nv))
    want = ol.apply(ol.tree_total(slots), delta)
    got = n_h.reshape(-1, nd)[torch.from_numpy(m).cuda()].cpu().numpy().astype(np.float64)
    got_sh = sh[torch.from_numpy(m).cuda()].cpu().numpy().astype(np.float64)
    return got, want, got_sh, oracle.shield(want), delta


@pytest.mark.parametrize("L,k", [(5, 800), (7, 400)])
def test_learned_fp32_column_density_matches_oracle(L, k):
    got, want, gsh, wsh, delta = _learned_case(L, 80 + L, k)
    assert np.abs(delta).max() > 1e-3          # the correction is not trivially zero
    assert np.max(np.abs(got - want) / want) < 1e-4
    assert np.max(np.abs(gsh - wsh)) < 2e-5


@pytest.mark.parametrize("L,k,dset", [(5, 800, ("healpix", 2, 0, None)), (7, 400, ("healpix", 2, 0, None)),
                                      (6, 400, ("mxn", 4, 4, None)), (9, 150, ("healpix", 2, 0, None))])
def test_learned_bf16_column_density_matches_oracle(L, k, dset):
    """BF16 form: per-level sums from the tensor-core contraction (<= 2^-8
    relative per term), BF16 inputs, weights, h and activations with FP32
    accumulation, hardware tanh / exp / log approximations.  N_tree carries
    <= 4e-3 relative; delta carries the BF16 roundings of three layers and
    of inputs whose own error is up to 4e-3 x sinv."""
    got, want, gsh, wsh, delta = _learned_case(L, 180 + L, k, dset, precision=colden.BF16, hidden=128)
    rel = np.abs(got - want) / want
    print("BF16 learned L=%d: rel max %.3g p99 %.3g mean %.3g; shield max %.3g; |delta| max %.3g"
          % (L, rel.max(), np.quantile(rel, 0.99), rel.mean(), np.abs(gsh - wsh).max(), np.abs(delta).max()))
    assert np.all(np.isfinite(got))
    assert rel.max() < 1.5e-2 and rel.mean() < 3e-3
    assert np.max(np.abs(gsh - wsh)) < 2e-3


@pytest.mark.parametrize("L,k,precision", [(5, 600, colden.FP32), (5, 600, colden.BF16), (7, 300, colden.BF16)])
def test_learned_trusted_range_falls_back_to_the_plain_column(L, k, precision):
    """A network whose biases put every even direction's delta near 3 and
    every odd one's near 0, with the trusted range [-1, 1]: the even
    directions return the plain tree column, the odd ones the corrected
    column, as the oracle chain with the same range (no delta lies within
    0.5 of an end point, so both sides take the same decisions)."""
    rho, tree, geom, T = _setup(L, 300 + L)
    nd, H = geom.n_dir, 128
    p = synth.mlp_init(nd, H, 300 + L, out_scale=0.05)
    p[-nd:] = np.where(np.arange(nd) % 2 == 0, 3.0, 0.0)
    net = colden.Net(nd, H, p)
    assert net.delta_range() == (-math.inf, math.inf)
    rho_m = rho.reshape(-1).cpu().numpy().astype(np.float64)
    ms = _sample(tree.n_leaf, 2000, 301 + L)
    ij = _ijk_of(ms)
    mu, sinv = ol.normaliser(ol.features(_oracle_slots(T, L, geom.dirs, ms),
                                         rho_m[(ij[:, 2] * (1 << L) + ij[:, 1]) * (1 << L) + ij[:, 0]]))
    st = net.state()
    st["mu"], st["sinv"] = mu.astype(np.float32), sinv.astype(np.float32)
    net.load_state(st)
    net.set_delta_range(-1.0, 1.0)
    assert net.delta_range() == (-1.0, 1.0)
    n_h = torch.full((tree.n_leaf * nd,), -1.0, device="cuda")
    sh = torch.full((tree.n_leaf,), -1.0, device="cuda")
    colden.column_density(tree, geom, n_h=n_h, shield=sh, net=net, precision=precision)
    torch.cuda.synchronize()
    colden.device_status()
    m = _sample(tree.n_leaf, k, 302 + L)
    slots = _oracle_slots(T, L, geom.dirs, m)
    ij = _ijk_of(m)
    nv = rho_m[(ij[:, 2] * (1 << L) + ij[:, 1]) * (1 << L) + ij[:, 0]]
    delta, _ = ol.forward(ol.unpack(p.astype(np.float64), nd, H), mu.astype(np.float32).astype(np.float64),
                          sinv.astype(np.float32).astype(np.float64), ol.features(slots, nv))
    even = np.arange(nd) % 2 == 0
    assert np.all(np.abs(delta[:, even]) > 1.5) and np.all(np.abs(delta[:, ~even]) < 0.5)
    plain = ol.tree_total(slots)
    want = ol.apply(plain, delta, -1.0, 1.0)
    assert np.array_equal(want[:, even], plain[:, even])
    got = n_h.reshape(-1, nd)[torch.from_numpy(m).cuda()].cpu().numpy().astype(np.float64)
    rel = np.abs(got - want) / want
    tol = 1e-4 if precision == colden.FP32 else 1.5e-2
    assert rel.max() < tol, rel.max()
    # without the range, the even directions would be ~e^3 larger
    assert np.all(got[:, even] < 2.0 * plain[:, even])
    got_sh = sh[torch.from_numpy(m).cuda()].cpu().numpy().astype(np.float64)
    assert np.max(np.abs(got_sh - oracle.shield(want))) < (2e-5 if precision == colden.FP32 else 2e-3)
    # an empty range: the plain column everywhere
    net.set_delta_range(1.0, -1.0)
    colden.column_density(tree, geom, n_h=n_h, net=net, precision=precision)
    got = n_h.reshape(-1, nd)[torch.from_numpy(m).cuda()].cpu().numpy().astype(np.float64)
    assert (np.abs(got - plain) / plain).max() < tol


def test_fit_delta_range_and_checkpoint(tmp_path):
    """The fitted range is the finite targets' range widened by the margin
    (FP32 ends), it survives save / load, and a NaN end is refused."""
    net, _ = _net(12, 16, seed=5)
    y_np = np.random.default_rng(5).normal(size=10007).astype(np.float32)
    y_np[[3, 77, 5000]] = [np.nan, np.inf, -np.inf]
    lo, hi = net.fit_delta_range(torch.from_numpy(y_np).cuda(), 0.25)
    wlo, whi = ol.delta_range(y_np.astype(np.float64), 0.25)
    assert lo == float(np.float32(wlo)) and hi == float(np.float32(whi))
    path = str(tmp_path / "net.npz")
    net.save(path)
    assert colden.Net.load(path).delta_range() == (lo, hi)
    lo, hi = net.fit_delta_range(torch.full((5,), float("nan"), device="cuda"), 0.0)
    assert lo > hi
    with pytest.raises(colden.ColdenError):
        net.set_delta_range(float("nan"), 1.0)
    with pytest.raises(colden.ColdenError):
        net.fit_delta_range(torch.zeros(3, device="cuda"), -1.0)


def test_learned_bf16_unaligned_outputs_match_aligned():
    rho, tree, geom, T = _setup(5, 95)
    nd = geom.n_dir
    net, _ = _net(nd, 128, seed=3, scale=0.3)
    a = torch.zeros(tree.n_leaf * nd, device="cuda")
    colden.column_density(tree, geom, n_h=a, net=net, precision=colden.BF16)
    big = torch.zeros(tree.n_leaf * nd + 1, device="cuda")
    b = big[1:]                                   # 4-byte aligned only
    av = torch.zeros(tree.n_leaf * nd + 1, device="cuda")[1:]
    colden.column_density(tree, geom, n_h=b, a_v=av, net=net, precision=colden.BF16)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert torch.allclose(av, a / 1.87e21, rtol=1e-6, atol=0)


def test_learned_bf16_rejects_unsupported_sizes():
    rho, tree, geom, T = _setup(5, 93)
    n_h = torch.zeros(tree.n_leaf * geom.n_dir, device="cuda")
    net, _ = _net(geom.n_dir, 64)
    with pytest.raises(colden.ColdenError) as e:
        colden.column_density(tree, geom, n_h=n_h, net=net, precision=colden.BF16)
    assert e.value.code == colden.CD_EUNSUPPORTED
    g12 = colden.precompute_geometry("healpix", 1)            # n_dir not a multiple of 8
    net12, _ = _net(12, 128)
    with pytest.raises(colden.ColdenError) as e:
        colden.column_density(tree, g12, n_h=torch.zeros(tree.n_leaf * 12, device="cuda"), net=net12,
                              precision=colden.BF16)
    assert e.value.code == colden.CD_EUNSUPPORTED
    g192 = colden.precompute_geometry("healpix", 4)
    net192, _ = _net(g192.n_dir, 128)
    with pytest.raises(colden.ColdenError) as e:
        colden.column_density(tree, g192, n_h=torch.zeros(tree.n_leaf * 192, device="cuda"), net=net192,
                              precision=colden.BF16)
    assert e.value.code == colden.CD_EUNSUPPORTED


def test_learned_falls_back_to_tree_where_delta_is_not_finite():
    L = 4
    rho, tree, geom, T = _setup(L, 90)
    nd = geom.n_dir
    p = synth.mlp_init(nd, 16, 7)
    lay = ol.shapes(nd, 16)
    off_b3 = sum(int(np.prod(s)) for _, s in lay[:-1])
    p[off_b3 + 3] = np.nan
    p[off_b3 + 5] = np.inf
    net = colden.Net(nd, 16, p)
    n_h = torch.zeros(tree.n_leaf * nd, device="cuda")
    colden.column_density(tree, geom, n_h=n_h, net=net)
    plain = torch.zeros_like(n_h)
    colden.column_density(tree, geom, n_h=plain)
    g = n_h.reshape(-1, nd).cpu().numpy()
    q = plain.reshape(-1, nd).cpu().numpy()
    assert np.all(np.isfinite(g))
    assert np.allclose(g[:, [3, 5]], q[:, [3, 5]], rtol=2e-5)
    assert not np.allclose(g[:, 0], q[:, 0], rtol=1e-3)
    # the BF16 form falls back the same way, to its own BF16 tree column (local
    # term on the tensor cores): within the BF16 tolerance of the plain column
    p128 = synth.mlp_init(nd, 128, 7)
    off_b3 = sum(int(np.prod(s)) for _, s in ol.shapes(nd, 128)[:-1])
    p128[off_b3 + 3] = np.nan
    p128[off_b3 + 5] = np.inf
    net = colden.Net(nd, 128, p128)
    colden.column_density(tree, geom, n_h=n_h, net=net, precision=colden.BF16)
    colden.column_density(tree, geom, n_h=plain, precision=colden.BF16)
    g = n_h.reshape(-1, nd).cpu().numpy()
    q = plain.reshape(-1, nd).cpu().numpy()
    assert np.all(np.isfinite(g))
    assert np.max(np.abs(g[:, [3, 5]] - q[:, [3, 5]]) / q[:, [3, 5]]) < 1e-2


def test_learned_rejects_mismatched_directions_and_amr():
    rho, tree, geom, T = _setup(4, 91)
    net, _ = _net(12, 16)
    with pytest.raises(colden.ColdenError) as e:
        colden.column_density(tree, geom, n_h=torch.zeros(tree.n_leaf * geom.n_dir, device="cuda"), net=net)
    assert e.value.code == colden.CD_EINVAL
    a = synth.amr_leaves(synth.lognormal_grf(16, 30.0, 2.0, 5), 2, [20.0, 60.0])
    amr = colden.build_tree_amr(a["base"], a["lmax"], 10 * PC, a["level"], a["ijk"], a["rho"])
    net48, _ = _net(geom.n_dir, 16)
    with pytest.raises(colden.ColdenError) as e:
        colden.column_density(amr, geom, n_h=torch.zeros(amr.n_leaf * geom.n_dir, device="cuda"), net=net48)
    assert e.value.code == colden.CD_EUNSUPPORTED
    with pytest.raises(colden.ColdenError) as e:
        colden.raymarch(amr, geom, torch.zeros((4, geom.n_dir), device="cuda"))
    assert e.value.code == colden.CD_EUNSUPPORTED


@pytest.mark.parametrize("precision", [colden.FP32, colden.BF16])
@pytest.mark.parametrize("n_net,n_geom", [(48, 8), (48, 24), (8, 48), (24, 40)])
def test_learned_refuses_a_network_of_other_directions_in_both_precisions(n_net, n_geom, precision):
    # sizes that either form takes when the two agree: refused before anything is launched
    _, tree, _, _ = _setup(4, 94)
    geom = colden.precompute_geometry("mxn", n_geom // 8, 8)
    net, _ = _net(n_net, 128)
    n_h = torch.full((tree.n_leaf * n_geom,), -1.0, device="cuda")
    torch.cuda.synchronize()
    colden.stats_reset()
    with pytest.raises(colden.ColdenError) as e:
        colden.column_density(tree, geom, n_h=n_h, net=net, precision=precision)
    assert e.value.code == colden.CD_EINVAL and "directions" in str(e.value)
    assert sum(colden.stats_get(k)[0] for k in range(len(colden.KERNEL_KINDS))) == 0
    assert bool((n_h == -1.0).all())


@pytest.mark.parametrize("precision", [colden.FP32, colden.BF16])
@pytest.mark.parametrize("L,dset", [(4, ("healpix", 2, 0)), (5, ("mxn", 3, 8)), (8, ("mxn", 1, 8))])
def test_learned_columns_with_negative_scales(L, dset, precision):
    # u = clip((x - mu) sinv): an input's scale and its weights negated together are
    # the same network, product by product, so the columns are the same bits; every
    # kind of input among them (own oct, near and far slots, density, empty slots)
    rho = torch.from_numpy(synth.lognormal_iid(1 << L, 10.0, 1.5, seed=3)).cuda()
    tree, geom = colden.build_tree_uniform(rho, 10 * PC), colden.precompute_geometry(*dset)
    nd, H = geom.n_dir, 128
    n_in = 8 * nd + 1
    net = colden.Net(nd, H, synth.mlp_init(nd, H, 8, out_scale=0.3))
    x = torch.empty((4096, n_in), device="cuda")
    colden.learned_features(tree, geom, x, leaves=torch.randint(tree.n_leaf, (4096,), device="cuda"))
    net.fit_normaliser(x)
    st = net.state()
    out = []
    for sign in (1.0, -1.0):
        flip = np.where(np.arange(n_in) % 2 == 0, sign, 1.0).astype(np.float32)
        p = st["params"].copy()
        p[: H * n_in] = (p[: H * n_in].reshape(H, n_in) * flip).reshape(-1)
        net.load_state(dict(st, params=p, sinv=st["sinv"] * flip))
        n_h = torch.full((tree.n_leaf, nd), -1.0, device="cuda")
        colden.column_density(tree, geom, n_h=n_h, net=net, precision=precision)
        colden.device_status()
        out.append(n_h)
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("nd,H,B", [(48, 128, 300_001), (48, 512, 300_001), (12, 1024, 300_001), (1, 1024, 1_000_003)])
def test_gradient_of_a_long_batch(nd, H, B):
    # B times the same row: every sum over the batch adds equal terms, whose roundings
    # do not cancel, and the gradient is that of the one row.  Chains of n1 rows, n2 of
    # them, err by (n1 + n2) / 2 x 2^-24 at most; with n1 + n2 <= 2 B^(2/3) beside the 1e-4
    # of the largest component that a gradient's terms are held to
    p = synth.mlp_init(nd, H, 4)
    n_in = 8 * nd + 1
    net = colden.Net(nd, H, p)
    rng = np.random.default_rng(5)
    x, y = rng.standard_normal((1, n_in)).astype(np.float32), rng.uniform(0.5, 1.0, (1, nd)).astype(np.float32)
    want, g = ol.loss_grad(ol.unpack(p.astype(np.float64), nd, H), np.zeros(n_in), np.ones(n_in), x.astype(np.float64),
                           y.astype(np.float64))
    g = ol.pack(g)
    loss, grad = torch.zeros(1, device="cuda"), torch.empty(net.n_params, device="cuda")
    rows = torch.zeros(B, dtype=torch.int64, device="cuda")
    net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), loss, grad, rows=rows)
    tol = 1e-4 + B ** (2 / 3) * 2.0 ** -24
    assert np.max(np.abs(grad.cpu().numpy() - g)) < tol * np.max(np.abs(g))
    assert loss.item() == pytest.approx(want, rel=1e-5)


@pytest.mark.parametrize("nd,H,first,B,n", [(48, 128, "loss", 4096, 4096), (48, 128, "gradient", 8192, 480),
                                            (48, 128, "step", 39_000, 9_700), (12, 40, "loss", 3000, 17)])
def test_gradient_is_captured_after_an_eager_call_of_any_kind(nd, H, first, B, n):
    # the first call at B rows, of the loss alone, the gradient or a step, allocates what
    # a gradient of up to B rows takes: it can then be captured at any such size
    net, _ = _net(nd, H)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x = torch.randn(B, 8 * nd + 1, device="cuda", generator=gen)
    y = torch.randn(B, nd, device="cuda", generator=gen)
    loss, grad, want = (torch.zeros(k, device="cuda") for k in (1, net.n_params, net.n_params))
    if first == "step":
        net.train_step(x, y, loss=loss)
    else:
        net.loss_grad(x, y, loss, grad if first == "gradient" else None)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        net.loss_grad(x, y, loss, grad, batch=n, stream=torch.cuda.current_stream())
    grad.fill_(-1.0)
    g.replay()
    torch.cuda.synchronize()
    net.loss_grad(x, y, loss, want, batch=n)
    assert torch.equal(grad, want)


# ---------------------------------------------------------------------------
# What the trained network gains over the plain tree method
# ---------------------------------------------------------------------------

def _dataset(L, seed, geom, n_rows):
    rho = _field(L, seed)
    tree = colden.build_tree_uniform(rho, 10 * PC)
    nd = geom.n_dir
    g = torch.Generator(device="cpu")
    g.manual_seed(seed)
    rows = torch.randperm(tree.n_leaf, generator=g)[:n_rows].cuda()
    x = torch.zeros((len(rows), 8 * nd + 1), device="cuda")
    nt = torch.zeros((len(rows), nd), device="cuda")
    nr = torch.zeros((len(rows), nd), device="cuda")
    colden.learned_features(tree, geom, x, nt, leaves=rows)
    colden.raymarch(tree, geom, nr, leaves=rows)
    y = torch.zeros_like(nr)
    colden.learned_targets(nr, nt, y)
    return x, y, nt, nr


def test_trained_network_beats_plain_tree_on_held_out_field():
    """Trained on eight seeded 64^3 fields (the recipe of the benchmark's
    training set at a smaller size), evaluated on a ninth.  The tree method's
    own error on a sigma_ln = 2 field is mostly fine structure along the ray
    that no per-level mean carries; the network removes the part its inputs
    do carry: more than a per-direction constant offset would, and it lowers
    the mean |A_V| error against the exact ray-marcher."""
    L = 6
    geom = colden.precompute_geometry("healpix", 2)
    parts = [_dataset(L, 300 + i, geom, 100000) for i in range(8)]
    x = torch.cat([p[0] for p in parts])
    y = torch.cat([p[1] for p in parts])
    net, _ = _net(geom.n_dir, 128, seed=12, scale=0.1)
    net.fit_normaliser(x)
    losses = colden.train(net, x, y, steps=1500, batch=4096, lr=2e-3, lr_final=1e-4, seed=3)
    assert np.all(np.isfinite(losses))
    xe, ye, nte, nre = _dataset(L, 399, geom, 50000)
    de = torch.zeros_like(ye)
    net.forward(xe, de)
    mse_plain = float((ye ** 2).mean())
    mse_offset = float(((ye - y.mean(0, keepdim=True)) ** 2).mean())
    mse_learned = float(((de - ye) ** 2).mean())
    av = 1.0 / 1.87e21
    dav_plain = float((nte * av - nre * av).abs().mean())
    dav_learned = float((nte * torch.exp(de) * av - nre * av).abs().mean())
    print("held-out: ln-error mse plain %.4g, per-direction offset %.4g, learned %.4g; "
          "<|dA_V|> plain %.4g learned %.4g" % (mse_plain, mse_offset, mse_learned, dav_plain, dav_learned))
    assert mse_learned < 0.9 * mse_plain
    assert mse_learned < 0.95 * mse_offset
    assert dav_learned < 0.98 * dav_plain


def test_resolution_matched_rows_make_the_network_gain_on_a_finer_field():
    """The network's inputs are the tree's per-level terms at the leaf's own
    scale, so a network fitted on coarser fields alone does not carry over
    to a finer one (printed for reference).  Fitted on the coarse fields plus
    a few fields at the finer resolution (other seeds), its rows drawn in
    proportion to the squared column and its training stop chosen by the
    mean |A_V| error on a held-out field at that resolution, it beats the plain
    tree on a further held-out fine field: a lower ln-error and a lower mean
    |A_V| error against the exact ray-marcher."""
    geom = colden.precompute_geometry("healpix", 2)
    nd = geom.n_dir
    coarse = [_dataset(5, 500 + i, geom, 32768) for i in range(6)]
    fine = [_dataset(6, 600 + i, geom, 100000) for i in range(4)]
    xv, yv, ntv, nrv = _dataset(6, 650, geom, 50000)
    xe, ye, nte, nre = _dataset(6, 699, geom, 50000)
    av = 1.0 / 1.87e21

    def val_dav(net):
        # the training stop: mean |A_V| error on the held-out fine field
        dv = torch.zeros_like(yv)
        net.forward(xv, dv)
        return float((ntv * torch.exp(dv) * av - nrv * av).abs().mean())

    def fit(parts, val):
        x = torch.cat([p[0] for p in parts])
        y = torch.cat([p[1] for p in parts])
        # rows drawn in proportion to the squared mean ray column: the fit follows the A_V error
        w = (torch.cat([p[3] for p in parts]).double() * av).mean(1) ** 2
        net, _ = _net(nd, 128, seed=12, scale=0.1)
        net.fit_normaliser(x)
        colden.train(net, x, y, steps=1500, batch=4096, lr=2e-3, lr_final=1e-4, seed=3, val=val, eval_every=150,
                     row_weights=w)
        de = torch.zeros_like(ye)
        net.forward(xe, de)
        torch.cuda.synchronize()
        return float(((de - ye) ** 2).mean()), float((nte * torch.exp(de) * av - nre * av).abs().mean()), net

    mse_plain = float((ye ** 2).mean())
    dav_plain = float((nte * av - nre * av).abs().mean())
    mse_c, dav_c, _ = fit(coarse, None)
    mse_m, dav_m, net = fit(coarse + fine, val_dav)
    steps = [s for s, _ in net.val_history]
    print("finer held-out field: ln-error mse plain %.4g, coarse-only %.4g, with matched rows %.4g; "
          "<|dA_V|> plain %.4g, coarse-only %.4g, matched %.4g; validation stop at step %d of %s"
          % (mse_plain, mse_c, mse_m, dav_plain, dav_c, dav_m, min(net.val_history, key=lambda h: h[1])[0], steps))
    assert steps[0] == 150 and steps[-1] == 1500
    assert mse_m < 0.9 * mse_plain
    assert dav_m < 0.995 * dav_plain

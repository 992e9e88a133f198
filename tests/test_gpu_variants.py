"""Kernel variants chosen by a rule on sizes, each at the edges of its range
against the general path or the oracle."""
import numpy as np
import pytest
import torch

import oracle
from oracle import learned as ol
from paper_1410_0624_gb300 import colden, synth

BOX = 10 * synth.PC_CM
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    colden.load(build_if_missing=True)


def _rho(L, seed, sigma=1.5):
    return synth.lognormal_iid(1 << L, 10.0, sigma, seed=seed)


@pytest.mark.parametrize("L,n,dset", [(3, 400_000, ("axes", 0, 0)), (5, 70_001, ("mxn", 7, 5)),
                                      (6, 33_000, ("healpix", 2, 0)), (7, 32_768, ("mxn", 3, 4))])
def test_raymarch_in_spatial_order_is_row_by_row_the_same(L, n, dset):
    # a list long enough to be marched in spatial order (repeated leaves and
    # entries out of range among it) against short pieces of it, bit for bit
    tree = colden.build_tree_uniform(torch.from_numpy(_rho(L, 7)).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    rng = np.random.default_rng(n)
    m = rng.integers(0, tree.n_leaf, n)
    m[:: 9973] = -1
    m[5:: 9973] = tree.n_leaf
    lv = torch.from_numpy(m).cuda()
    out = torch.full((n, geom.n_dir), -1.0, device="cuda")
    colden.raymarch(tree, geom, out, leaves=lv)
    ref = torch.full((n, geom.n_dir), -1.0, device="cuda")
    for i in range(0, n, 8000):
        piece = torch.empty((min(8000, n - i), geom.n_dir), device="cuda")
        colden.raymarch(tree, geom, piece, leaves=lv[i:i + 8000].contiguous())
        ref[i:i + 8000] = piece
    assert torch.equal(out, ref)
    bad = torch.from_numpy((m < 0) | (m >= tree.n_leaf)).cuda()
    assert bool((out[bad] == 0).all()) and bool((out[~bad] > 0).all())
    rows = np.flatnonzero((m >= 0) & (m < tree.n_leaf))[:: max(1, n // 200)]
    ijk = oracle.morton_ijk(L)[m[rows]]
    want = oracle.Tree.uniform(_rho(L, 7), BOX).raymarch(geom.dirs, np.full(len(rows), L), ijk)
    got = out[torch.from_numpy(rows).cuda()].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) < 2e-5   # the ray-marcher's tolerance


@pytest.mark.parametrize("L,n,dset,kind", [(1, 2_100_001, ("axes", 0, 0), "random"), (2, 1_050_003, ("axes", 0, 0), "one"),
                                           (3, 530_001, ("axes", 0, 0), "random"), (3, 530_001, ("axes", 0, 0), "one"),
                                           (4, 270_001, ("axes", 0, 0), "random"), (4, 270_001, ("axes", 0, 0), "one"),
                                           (4, 140_017, ("healpix", 1, 0), "few"), (4, 270_001, ("axes", 0, 0), "sorted"),
                                           (5, 70_001, ("healpix", 1, 0), "runs"), (7, 40_003, ("mxn", 3, 4), "few")])
def test_raymarch_of_repeated_leaves(L, n, dset, kind):
    # long lists of the smallest trees that are marched as listed and of the smallest
    # that are sorted (a bucket a leaf), with one leaf, a few, runs and sorted ones: rows
    # of one leaf are the same bits, and those of the leaf marched in a short list
    tree = colden.build_tree_uniform(torch.from_numpy(_rho(L, 7)).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    rng = np.random.default_rng(n)
    m = {"random": lambda: rng.integers(-1, tree.n_leaf + 1, n), "one": lambda: np.full(n, tree.n_leaf // 3),
         "few": lambda: rng.choice([0, 1, tree.n_leaf // 2, tree.n_leaf - 1, -1], n),
         "sorted": lambda: np.sort(rng.integers(0, tree.n_leaf, n)),
         "runs": lambda: np.repeat(rng.integers(0, tree.n_leaf, n // 50 + 1), 50)[:n]}[kind]()
    out = torch.full((n, geom.n_dir), -1.0, device="cuda")
    colden.raymarch(tree, geom, out, leaves=torch.from_numpy(m).cuda())
    leaf, back = np.unique(m, return_inverse=True)
    one = torch.full((len(leaf), geom.n_dir), -1.0, device="cuda")
    for i in range(0, len(leaf), 1000):
        piece = torch.empty((len(leaf[i:i + 1000]), geom.n_dir), device="cuda")
        colden.raymarch(tree, geom, piece, leaves=torch.from_numpy(leaf[i:i + 1000].copy()).cuda())
        one[i:i + 1000] = piece
    assert torch.equal(out, one[torch.from_numpy(back).cuda()])
    bad = torch.from_numpy((leaf < 0) | (leaf >= tree.n_leaf)).cuda()
    assert bool((one[bad] == 0).all()) and bool((one[~bad] > 0).all())


@pytest.mark.parametrize("nd,H,B", [(5, 16, 33), (3, 97, 130), (12, 64, 4931), (48, 128, 9729), (7, 50, 38913),
                                    (13, 61, 38912), (12, 100, 39001)])
def test_network_at_the_edges_of_its_gemm_tiles(nd, H, B):
    # batches of the small, medium and large tiles (48, 64 and 128 columns wide),
    # full and ragged, with gathered rows; tolerances as for any other batch
    rng = np.random.default_rng(B)
    p = synth.mlp_init(nd, H, 2)
    net = colden.Net(nd, H, p)
    x = synth.mlp_inputs(B + 7, 8 * nd + 1, seed=B)
    y = (0.3 * rng.standard_normal((B + 7, nd))).astype(np.float32)
    rows = rng.integers(0, B + 7, B)
    mu, sinv = ol.normaliser(x.astype(np.float64))
    st = net.state()
    st["mu"], st["sinv"] = mu.astype(np.float32), sinv.astype(np.float32)
    net.load_state(st)
    args = (ol.unpack(p.astype(np.float64), nd, H), st["mu"].astype(np.float64), st["sinv"].astype(np.float64),
            x[rows].astype(np.float64))
    dx, dy, dr = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), torch.from_numpy(rows).cuda()
    delta = torch.full((B, nd), 9.0, device="cuda")
    net.forward(dx[dr].contiguous(), delta)
    assert np.max(np.abs(delta.cpu().numpy() - ol.forward(*args)[0])) < 1e-4
    loss, alone = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    grad = torch.full((net.n_params,), 9.0, device="cuda")
    net.loss_grad(dx, dy, loss, grad, rows=dr)
    net.loss_grad(dx, dy, alone, rows=dr)
    want, g_or = ol.loss_grad(*args, y[rows].astype(np.float64))
    g_or = ol.pack(g_or)
    assert loss.item() == pytest.approx(want, rel=1e-5) and torch.equal(loss, alone)
    assert np.max(np.abs(grad.cpu().numpy() - g_or)) < 1e-4 * np.max(np.abs(g_or))


@pytest.mark.parametrize("L,dset,mode", [(5, ("custom", 0, 0, [[0.3, -0.5, 0.8]]), 0), (5, ("mxn", 3, 1), 0),
                                         (6, ("mxn", 5, 3), 0), (6, ("mxn", 14, 9), 0), (7, ("axes", 0, 0), 0),
                                         (7, ("mxn", 5, 8), 2), (8, ("mxn", 2, 2), 0)])
def test_fp32_shell_rows_match_oracle(L, dset, mode):
    # direction counts that fill a quad of directions or leave part of it, levels
    # with fewer and more parents per class than a CTA takes; FP32 tolerance
    rho = _rho(L, 50 + L)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset, mode=mode)
    nh = torch.empty((tree.n_leaf, geom.n_dir), device="cuda")
    colden.column_density(tree, geom, n_h=nh)
    corner = np.array([0, tree.n_leaf - 1, tree.n_leaf // 2, tree.n_leaf // 8 + 1])
    rows = np.unique(np.concatenate([corner, np.random.default_rng(L).integers(0, tree.n_leaf, 250)]))
    ijk = oracle.morton_ijk(L)[rows] if L < 8 else tree.leaves()[1][rows]
    T = oracle.Tree.uniform(rho, BOX)
    lv = np.full(len(rows), L)
    want = T.column_density_cone(geom.dirs, lv, ijk) if mode else T.column_density(geom.dirs, lv, ijk)
    got = nh[torch.from_numpy(rows).cuda()].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-5


@pytest.mark.parametrize("dset,mode", [(("custom", 0, 0, [[0.3, -0.5, 0.8]]), 0), (("axes", 0, 0), 0), (("healpix", 1, 0), 0),
                                       (("mxn", 7, 3), 0), (("healpix", 2, 0), 0), (("mxn", 5, 8), 2), (("mxn", 16, 17), 0)])
@pytest.mark.parametrize("L", [3, 4, 5, 6])
def test_fp32_small_trees_match_their_launches_one_by_one(L, dset, mode):
    # 32^3 sums the octs' shells and the far ones in one launch; the form with fixed
    # scratch launches every level by itself: the same kernels, bit for bit, also captured
    tree = colden.build_tree_uniform(torch.from_numpy(_rho(L, 50 + L)).cuda(), BOX)
    geom = colden.precompute_geometry(*dset, mode=mode)
    new = lambda: (torch.full((tree.n_leaf, geom.n_dir), -1.0, device="cuda"),  # noqa: E731
                   torch.full((tree.n_leaf,), -1.0, device="cuda"))
    a, b, c = new(), new(), new()
    colden.column_density(tree, geom, n_h=a[0], shield=a[1])
    try:
        colden.column_density_noalloc(tree, geom, n_h=b[0], shield=b[1])
    except colden.ColdenError:
        assert L == 6 and geom.n_dir > 40        # the fixed scratch is too small
        b = a
    colden.EvalGraph(tree, geom, n_h=c[0], shield=c[1]).launch()
    torch.cuda.synchronize()
    colden.device_status()
    assert float(a[0].min()) > 0
    for x, y, z in zip(a, b, c):
        assert torch.equal(x, y) and torch.equal(x, z)


@pytest.mark.parametrize("dset", [("mxn", 5, 3), ("axes", 0, 0), ("healpix", 2, 0)])
def test_fp32_shell_rows_on_lists_match_uniform(dset):
    # a mesh refined in one corner: its finest leaves far inside the refined part
    # and its base leaves against the oracle's adaptive tree
    fine = _rho(7, 3, 1.0)
    fine[:40, :44, :48] *= 50.0
    lv = synth.amr_leaves(fine, 5, [100.0, 200.0])
    tree = colden.build_tree_amr(5, 7, BOX, lv["level"], lv["ijk"], lv["rho"])
    geom = colden.precompute_geometry(*dset)
    nh = torch.empty((tree.n_leaf, geom.n_dir), device="cuda")
    colden.column_density(tree, geom, n_h=nh)
    level, ijk = tree.leaves()
    rng = np.random.default_rng(1)
    rows = np.concatenate([rng.choice(np.flatnonzero(level == l), 120) for l in np.unique(level)])
    want = oracle.Tree.amr(5, 7, BOX, lv["level"], lv["ijk"], lv["rho"]).column_density(geom.dirs, level[rows], ijk[rows])
    got = nh[torch.from_numpy(rows).cuda()].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-5


@pytest.mark.parametrize("count", [900, 1100, 1500, 1700, 2500])
@pytest.mark.parametrize("dset,mode", [(("mxn", 4, 4), 0), (("mxn", 5, 4), 0), (("mxn", 7, 12), 0), (("mxn", 3, 4), 2),
                                       (("mxn", 5, 4), 1)])
def test_fp32_lists_of_16_cubed_on_both_sides_of_the_row_forms_lines(count, dset, mode):
    # lists of 16^3 below and above the receivers from which the row form takes them, by
    # directions and kind of ray, against the oracle's adaptive tree
    fine = synth.lognormal_grf(32, 10.0, 1.5, seed=3)
    mean = fine.reshape(16, 2, 16, 2, 16, 2).mean((1, 3, 5))
    lv = synth.amr_leaves(fine, 4, [float(np.sort(mean.reshape(-1))[-count - 1])])
    tree = colden.build_tree_amr(4, 5, BOX, lv["level"], lv["ijk"], lv["rho"])
    geom = colden.precompute_geometry(*dset, mode=mode)
    nh = torch.full((tree.n_leaf, geom.n_dir), -1.0, device="cuda")
    colden.column_density(tree, geom, n_h=nh)
    level, ijk = tree.leaves()
    rng = np.random.default_rng(count)
    rows = np.concatenate([rng.choice(np.flatnonzero(level == l), 100) for l in (4, 5)])
    T = oracle.Tree.amr(4, 5, BOX, lv["level"], lv["ijk"], lv["rho"])
    want = (T.column_density_cone(geom.dirs, level[rows], ijk[rows]) if mode == 2 else
            T.column_density(geom.dirs, level[rows], ijk[rows], mode=oracle.MODE_INSITU if mode else oracle.MODE_PREC))
    got = nh[torch.from_numpy(rows).cuda()].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-5


@pytest.mark.parametrize("dset", [("mxn", 1, 4), ("mxn", 2, 4), ("healpix", 1, 0), ("mxn", 4, 4), ("mxn", 5, 4),
                                  ("mxn", 4, 6), ("mxn", 4, 7), ("mxn", 8, 4), ("mxn", 9, 4), ("mxn", 5, 8),
                                  ("mxn", 11, 4), ("healpix", 2, 0), ("mxn", 13, 4), ("mxn", 7, 8), ("mxn", 15, 4),
                                  ("mxn", 8, 8)])
@pytest.mark.parametrize("L", [3, 4, 6])
def test_bf16_leaves_of_few_directions(L, dset):
    # every direction count of the oct form, a tree smaller than its tile and
    # larger ones, each set of outputs; BF16 tolerances
    rho = _rho(L, 9)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    nd = geom.n_dir
    new = lambda *s: torch.full(s, -1.0, device="cuda")  # noqa: E731
    nh, av, sh = new(tree.n_leaf, nd), new(tree.n_leaf, nd), new(tree.n_leaf)
    colden.column_density(tree, geom, n_h=nh, a_v=av, shield=sh, precision=colden.BF16)
    nh2, av2, sh2 = new(tree.n_leaf, nd), new(tree.n_leaf, nd), new(tree.n_leaf)
    colden.column_density(tree, geom, n_h=nh2, precision=colden.BF16)
    colden.column_density(tree, geom, a_v=av2, precision=colden.BF16)
    colden.column_density(tree, geom, shield=sh2, precision=colden.BF16)
    colden.device_status()
    # (beyond 32 directions the screening factor alone has a kernel of its own: the
    # same columns, summed in another order)
    assert torch.equal(nh, nh2) and torch.equal(av, av2)
    assert torch.equal(sh, sh2) if nd <= 32 else float((sh - sh2).abs().max()) < 1e-6
    rows = np.unique(np.random.default_rng(L).integers(0, tree.n_leaf, 300))
    want = oracle.Tree.uniform(rho, BOX).column_density(geom.dirs, np.full(len(rows), L), oracle.morton_ijk(L)[rows])
    at = torch.from_numpy(rows).cuda()
    got = nh[at].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-2
    assert np.max(np.abs(av[at].double().cpu().numpy() - oracle.a_v(got)) / oracle.a_v(got)) < 1e-6
    assert np.max(np.abs(sh2[at].double().cpu().numpy() - oracle.shield(want))) <= 5e-3


@pytest.mark.parametrize("L,dset,H", [(1, ("healpix", 1, 0), 16), (2, ("axes", 0, 0), 33), (4, ("mxn", 5, 3), 64),
                                      (5, ("healpix", 2, 0), 128), (6, ("mxn", 7, 12), 40)])
def test_fp32_learned_columns_by_octs(L, dset, H):
    # the learned columns (layer 1 by octs) against features and network row by
    # row; the two differ by the order of FP32 sums: 1e-5 on a correction of
    # order one, 2e-5 relative on the column
    rho = _rho(L, 21)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    nd = geom.n_dir
    net = colden.Net(nd, H, synth.mlp_init(nd, H, 5, out_scale=0.3))
    x = torch.empty((tree.n_leaf, 8 * nd + 1), device="cuda")
    nt, delta = torch.empty((tree.n_leaf, nd), device="cuda"), torch.empty((tree.n_leaf, nd), device="cuda")
    colden.learned_features(tree, geom, x, nt)
    net.fit_normaliser(x)
    net.forward(x, delta)
    nh, av, sh = torch.empty_like(nt), torch.empty_like(nt), torch.empty(tree.n_leaf, device="cuda")
    colden.column_density(tree, geom, n_h=nh, a_v=av, shield=sh, net=net)
    want = nt.double() * torch.exp(delta.double())
    assert float(((nh.double() - want).abs() / want).max()) < 2e-5
    assert float(((av.double() - want / 1.87e21).abs() / (want / 1.87e21)).max()) < 2e-5
    assert float((sh.double() - torch.exp(-2.5 * want / 1.87e21).mean(1)).abs().max()) < 1e-5


@pytest.mark.parametrize("L,dset,shift", [(1, ("mxn", 5, 7), 0), (2, ("mxn", 3, 3), 0), (4, ("mxn", 11, 3), 0),
                                          (5, ("axes", 0, 0), 0), (5, ("mxn", 5, 1), 0), (5, ("mxn", 13, 5), 0),
                                          (4, ("healpix", 2, 0), 1), (6, ("mxn", 3, 4), 2), (3, ("mxn", 127, 1), 0),
                                          (2, ("mxn", 97, 5), 0), (5, ("mxn", 2, 2), 3)])
def test_fp32_leaves_of_any_direction_count_and_alignment(L, dset, shift):
    # counts that are no multiple of four, outputs off the 16-byte boundary, and
    # both sides of the rule's lines; FP32 tolerances on every leaf
    rho = _rho(L, 31)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    nd, n = geom.n_dir, tree.n_leaf
    buf = torch.full((2 * n * nd + n + 64,), -1.0, device="cuda")
    nh = buf[shift:shift + n * nd]
    av = buf[n * nd + 2 * shift:][:n * nd]
    sh = torch.full((n + 8,), -1.0, device="cuda")[shift:shift + n]
    colden.column_density(tree, geom, n_h=nh, a_v=av, shield=sh)
    only = torch.full((n + 8,), -1.0, device="cuda")[shift:shift + n]
    colden.column_density(tree, geom, shield=only)
    assert torch.equal(sh, only)
    rows = np.arange(n) if n <= 4096 else np.unique(np.random.default_rng(L).integers(0, n, 2000))
    want = oracle.Tree.uniform(rho, BOX).column_density(geom.dirs, np.full(len(rows), L), oracle.morton_ijk(L)[rows])
    at = torch.from_numpy(rows).cuda()
    got = nh.reshape(n, nd)[at].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-5
    assert np.max(np.abs(av.reshape(n, nd)[at].double().cpu().numpy() - oracle.a_v(got)) / oracle.a_v(got)) < 1e-6
    assert np.max(np.abs(sh[at].double().cpu().numpy() - oracle.shield(want))) <= 1e-5


@pytest.mark.parametrize("dset", [("mxn", 5, 8), ("healpix", 2, 0), ("mxn", 8, 8)])
@pytest.mark.parametrize("shift", [0, 1])
def test_bf16_extinction_rows(dset, shift):
    # A_V alone, beside N_H and off the 16-byte boundary, on a uniform tree and on
    # lists whose rows scatter: N_H times the constant, to one rounding (lists
    # send N_H off the boundary through the FP32 leaf kernel, whose local term is
    # not rounded: there A_V alone, from the tensor cores, has another N_H)
    geom = colden.precompute_geometry(*dset)
    nd = geom.n_dir
    fine = _rho(6, 4, 1.0)
    fine[10:30, 5:40, 20:50] *= 30.0
    lv = synth.amr_leaves(fine, 5, [60.0])
    for tree in (colden.build_tree_uniform(torch.from_numpy(fine).cuda(), BOX),
                 colden.build_tree_amr(5, 6, BOX, lv["level"], lv["ijk"], lv["rho"])):
        n = tree.n_leaf * nd
        new = lambda: torch.full((n + 4,), -1.0, device="cuda")[shift:shift + n]  # noqa: E731
        nh, av, alone, sh = new(), new(), new(), torch.empty(tree.n_leaf, device="cuda")
        colden.column_density(tree, geom, n_h=nh, a_v=av, shield=sh, precision=colden.BF16)
        colden.column_density(tree, geom, a_v=alone, precision=colden.BF16)
        colden.device_status()
        want = nh.double() * colden.opts_default().av_per_nh
        assert float(nh.min()) > 0
        for got in (av, alone) if tree.n_oct * 8 == tree.n_leaf or not shift else (av,):
            assert float(((got.double() - want).abs() / want).max()) < 2e-7
        sh_want = torch.exp(-2.5 * want.reshape(-1, nd)).mean(1)
        assert float((sh.double() - sh_want).abs().max()) < 1e-5


@pytest.mark.parametrize("L,dset", [(4, ("mxn", 5, 8)), (5, ("mxn", 5, 3)), (6, ("axes", 0, 0)), (7, ("healpix", 2, 0))])
def test_insitu_near_shells_from_the_tables(L, dset):
    # levels where every shell is walked, where one to three are, and directions
    # the tables' row form does not take; uniform and adaptive, FP32 tolerance
    geom = colden.precompute_geometry(*dset, mode=colden.MODE_INSITU)
    fine = _rho(L, 12, 1.2)
    fine[: 1 << (L - 1), : 1 << (L - 1)] *= 20.0
    rng = np.random.default_rng(L)
    trees = [(colden.build_tree_uniform(torch.from_numpy(fine).cuda(), BOX), oracle.Tree.uniform(fine, BOX))]
    if L >= 5:
        lv = synth.amr_leaves(fine, L - 2, [40.0, 60.0])
        args = (L - 2, L, BOX, lv["level"], lv["ijk"], lv["rho"])
        trees.append((colden.build_tree_amr(*args), oracle.Tree.amr(*args)))
    for tree, T in trees:
        nh = torch.empty((tree.n_leaf, geom.n_dir), device="cuda")
        colden.column_density(tree, geom, n_h=nh)
        level, ijk = tree.leaves()
        rows = rng.integers(0, tree.n_leaf, 300)
        want = T.column_density(geom.dirs, level[rows], ijk[rows], mode=oracle.MODE_INSITU)
        got = nh[torch.from_numpy(rows).cuda()].double().cpu().numpy()
        assert np.max(np.abs(got - want) / want) <= 1e-5


@pytest.mark.parametrize("dset", [("mxn", 1, 8), ("mxn", 3, 8), ("mxn", 5, 8), ("healpix", 2, 0)])
@pytest.mark.parametrize("L", [2, 3, 5, 6])
def test_bf16_learned_columns_over_tiles_and_widths(L, dset):
    # tiles of 128 leaves, one to several per CTA, half a tile at the smallest, and
    # the widths of the direction groups, against the FP32 form: the 1.5e-2 of the
    # BF16 form against the exact network with a correction of this size
    rho = _rho(L, 31)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    nd = geom.n_dir
    net = colden.Net(nd, 128, synth.mlp_init(nd, 128, 6, out_scale=0.2))
    x = torch.empty((tree.n_leaf, 8 * nd + 1), device="cuda")
    colden.learned_features(tree, geom, x, None)
    net.fit_normaliser(x)
    out = {}
    for prec in (colden.FP32, colden.BF16):
        nh = torch.full((tree.n_leaf, nd), -1.0, device="cuda")
        av, sh = torch.full_like(nh, -1.0), torch.full((tree.n_leaf,), -1.0, device="cuda")
        colden.column_density(tree, geom, n_h=nh, a_v=av, shield=sh, net=net, precision=prec)
        colden.device_status()
        out[prec] = nh, sh
    (want, want_sh), (got, got_sh) = out[colden.FP32], out[colden.BF16]
    assert float(((got - want).abs() / want).max()) < 1.5e-2
    assert float((got_sh - want_sh).abs().max()) < 2e-3
    assert float((av.double() - got.double() / 1.87e21).abs().max() / av.double().max()) < 2e-7
    sh_of = torch.exp(-2.5 * got.double() / 1.87e21).mean(1)
    assert float((got_sh.double() - sh_of).abs().max()) < 1e-5


@pytest.mark.parametrize("dset", [("mxn", 1, 4), ("mxn", 2, 4), ("mxn", 3, 4), ("mxn", 4, 4), ("mxn", 5, 4), ("mxn", 4, 8),
                                  ("healpix", 2, 0), ("mxn", 7, 12), ("mxn", 12, 16)])
@pytest.mark.parametrize("L", [1, 2, 3, 5])
def test_fp32_leaves_in_fours(L, dset):
    # whole and partial batches of octs, padded screening sums, with and without the
    # prefix of the parents: every combination of outputs against the oracle (FP32
    # sums to 1e-5, as the path's other tests) and against each other
    rho = _rho(L, 41)
    n = 8 ** L
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    nd = geom.n_dir
    new = lambda *s: torch.full(s, -1.0, device="cuda")  # noqa: E731
    nh, sh, nh2, sh2, av2, only, alone = new(n, nd), new(n), new(n, nd), new(n), new(n, nd), new(n), new(n, nd)
    colden.column_density(tree, geom, n_h=nh, shield=sh)
    colden.column_density(tree, geom, n_h=nh2, a_v=av2, shield=sh2)
    colden.column_density(tree, geom, shield=only)
    colden.column_density(tree, geom, n_h=alone)
    colden.device_status()
    assert torch.equal(nh, nh2) and torch.equal(nh, alone) and torch.equal(sh, sh2) and torch.equal(sh, only)
    rows = np.arange(n) if n <= 4096 else np.unique(np.random.default_rng(L).integers(0, n, 1500))
    want = oracle.Tree.uniform(rho, BOX).column_density(geom.dirs, np.full(len(rows), L), oracle.morton_ijk(L)[rows])
    at = torch.from_numpy(rows).cuda()
    got = nh[at].double().cpu().numpy()
    assert np.max(np.abs(got - want) / want) <= 1e-5
    assert np.max(np.abs(av2[at].double().cpu().numpy() - oracle.a_v(got)) / oracle.a_v(got)) < 1e-6
    assert np.max(np.abs(sh[at].double().cpu().numpy() - oracle.shield(want))) <= 1e-5

"""Failure detection on the GPU without a fault.

Every pipeline wait of the library's kernels is bounded: a wait that runs out
sets a device flag, the kernel lets the copies and tensor-core products it has
issued land (with the full limit), frees its tensor memory and returns, and
cd_device_status reports CD_ETIMEOUT.  The testing hook cd_debug_wait_polls(0)
makes the pipeline waits of the tensor-core leaf kernel (the BF16 leaf
epilogue; here with 24 M x N directions) give up without polling, so every
CTA takes that path; nothing
traps and the context stays usable: the flag is cleared by the report and the
next evaluation matches the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1410_0624_gb300 import colden, synth

pytestmark = pytest.mark.gpu
BOX = 10 * synth.PC_CM


@pytest.fixture(scope="module", autouse=True)
def _lib():
    colden.load(build_if_missing=True)


def _oracle_check(tree, rho, n_h, sh, nd, rows):
    lv, ijk = tree.leaves()
    ref = oracle.Tree.uniform(rho, BOX).column_density(oracle.dirs_mxn(4, 6), lv[rows], ijk[rows])
    got = n_h.reshape(-1, nd)[torch.from_numpy(rows).cuda()].double().cpu().numpy()
    assert np.max(np.abs(got - ref) / ref) <= 1e-2
    assert np.max(np.abs(sh.cpu().numpy()[rows] - oracle.shield(ref))) <= 5e-3


def test_bounded_wait_runs_out_and_the_context_recovers():
    rho = synth.lognormal_grf(32, 30.0, 2.0, seed=61)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry("mxn", 4, 6)     # 24 directions
    nd = geom.n_dir
    n_h = torch.full((tree.n_leaf * nd,), -1.0, device="cuda")
    sh = torch.full((tree.n_leaf,), -1.0, device="cuda")
    colden.device_status()                      # no flag left over from earlier work
    colden.debug_wait_polls(0)
    try:
        colden.column_density(tree, geom, n_h=n_h, shield=sh, precision=colden.BF16)
        with pytest.raises(colden.ColdenError) as e:
            colden.device_status()
        assert e.value.code == colden.CD_ETIMEOUT and "bounded wait" in str(e.value)
    finally:
        colden.debug_wait_polls(-1)
    # every CTA gave up before its first tile: no row was written
    assert torch.all(sh == -1.0)
    colden.device_status()                      # the report cleared the flag
    colden.column_density(tree, geom, n_h=n_h, shield=sh, precision=colden.BF16)
    colden.device_status()
    rows = np.random.default_rng(3).choice(tree.n_leaf, size=300, replace=False)
    _oracle_check(tree, rho, n_h, sh, nd, rows)


def _give_up(call, limits):
    """`call` under poll limits that let its waits run out at the first tile, at
    a later one or not at all: it returns, and reports what happened."""
    codes = []
    colden.device_status()                      # no flag left over from earlier work
    try:
        for polls in limits:
            colden.debug_wait_polls(polls)
            call()
            try:
                colden.device_status()
                codes.append(0)
            except colden.ColdenError as e:
                assert e.code == colden.CD_ETIMEOUT and "bounded wait" in str(e)
                codes.append(e.code)
    finally:
        colden.debug_wait_polls(-1)
    return codes


@pytest.mark.parametrize("dset,rows", [(("mxn", 1, 4), True), (("healpix", 1), True), (("mxn", 4, 8), True),
                                       (("mxn", 5, 8), False), (("mxn", 8, 8), False)])
def test_waits_of_the_oct_form_run_out_at_any_tile(dset, rows):
    # leaves by octs: many tiles a group, one product each or two (beyond 32
    # directions); the evaluation after it is the one before it
    rho = synth.lognormal_iid(256, 10.0, 1.0, seed=62)
    tree = colden.build_tree_uniform(torch.from_numpy(rho).cuda(), BOX)
    geom = colden.precompute_geometry(*dset)
    n_h = torch.full((tree.n_leaf, geom.n_dir), -1.0, device="cuda") if rows else None
    sh = torch.full((tree.n_leaf,), -1.0, device="cuda")
    call = lambda: colden.column_density(tree, geom, n_h=n_h, shield=sh, precision=colden.BF16)  # noqa: E731
    call()
    colden.device_status()
    want = sh.clone(), n_h.clone() if rows else None
    codes = _give_up(call, [0, 1, 2, 3, 5, 8, 0, 13, 1, 2])
    assert codes[0] == codes[6] == colden.CD_ETIMEOUT
    sh.fill_(-1.0)
    call()
    colden.device_status()
    assert torch.equal(sh, want[0]) and (not rows or torch.equal(n_h, want[1]))


@pytest.mark.parametrize("kind,ndir", [("uniform", 36), ("uniform", 48), ("list", 12), ("list", 48), ("list", 64),
                                       ("unprefixed", 48), ("batch", 48)])
def test_waits_of_the_tiles_of_128_leaves_run_out_at_any_tile(kind, ndir):
    # uniform trees with rows beyond 32 directions, adaptive lists (with the parents'
    # prefix and, directly under the base level, without) and the persistent batch
    geom = colden.precompute_geometry("mxn", ndir // 4, 4)
    if kind == "uniform":
        trees = [colden.build_tree_uniform(torch.from_numpy(synth.lognormal_iid(64, 10.0, 1.0, seed=63)).cuda(), BOX)]
    else:
        n, base = (32, 4) if kind == "unprefixed" else (128, 5)
        fine = synth.lognormal_iid(n, 10.0, 1.0, seed=64)
        fine[: n // 2, : n // 2] *= 20.0
        lv = synth.amr_leaves(fine, base, [40.0] if n == 32 else [40.0, 200.0])
        trees = [colden.build_tree_amr(lv["base"], lv["lmax"], BOX, lv["level"], lv["ijk"], lv["rho"])
                 for _ in range(2 if kind == "batch" else 1)]
    outs = [torch.full((t.n_leaf, ndir), -1.0, device="cuda") for t in trees]
    if kind == "batch":
        colden.debug_batch_form(1)
        b = colden.Batch(trees, [geom] * 2, n_h=outs, precision=colden.BF16)
        assert b.info()["persistent"]
        call = b.run
        colden.stats_reset(timing=True)         # its launches one by one, not the captured graph
    else:
        call = lambda: colden.column_density(trees[0], geom, n_h=outs[0], precision=colden.BF16)  # noqa: E731
    try:
        call()
        colden.device_status()
        want = [o.clone() for o in outs]
        codes = _give_up(call, [0, 1, 2, 3, 5, 8, 0])
        assert codes[0] == codes[-1] == colden.CD_ETIMEOUT
        for o in outs:
            o.fill_(-1.0)
        call()
        colden.device_status()
        assert all(torch.equal(o, w) for o, w in zip(outs, want))
    finally:
        colden.debug_batch_form(-1)
        colden.stats_reset(timing=False)

"""Host threads on handles of their own, with trees of different depth and
direction sets of different width, so that both threads launch the same kernels
with different amounts of shared memory: no call may fail, and the results are
those of the same calls made alone, bit for bit."""
import threading
import time

import numpy as np
import pytest
import torch

from paper_1410_0624_gb300 import colden, synth

BOX = 10 * synth.PC_CM
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    colden.load(build_if_missing=True)


def _tree(L, seed):
    return colden.build_tree_uniform(torch.from_numpy(synth.lognormal_iid(1 << L, 10.0, 1.0, seed=seed)).cuda(), BOX)


def _columns(L, dset, precision, mode=0, rows=True, tree=None):
    t, g = tree or _tree(L, L), colden.precompute_geometry(*dset, mode=mode)
    out = torch.full((t.n_leaf, g.n_dir) if rows else (t.n_leaf,), -1.0, device="cuda")
    kw = {"n_h": out} if rows else {"shield": out}
    return out, lambda s: colden.column_density(t, g, precision=precision, stream=s, **kw)


def _march(L, dset):
    t, g = _tree(L, L), colden.precompute_geometry(*dset)
    out = torch.full((64, g.n_dir), -1.0, device="cuda")
    return out, lambda s: colden.raymarch(t, g, out, stream=s)


def _amr(dset, precision):
    fine = synth.lognormal_iid(16, 10.0, 1.0, seed=2)
    fine[:8, :8] *= 20.0
    lv = synth.amr_leaves(fine, 3, [40.0])
    return _columns(4, dset, precision, tree=colden.build_tree_amr(3, 4, BOX, lv["level"], lv["ijk"], lv["rho"]))


def _learned(dset):
    t, g = _tree(4, 4), colden.precompute_geometry(*dset)
    nd = g.n_dir
    net = colden.Net(nd, 128, synth.mlp_init(nd, 128, 6, out_scale=0.2))
    out = torch.full((t.n_leaf, nd), -1.0, device="cuda")
    return out, lambda s: colden.column_density(t, g, n_h=out, net=net, precision=colden.BF16, stream=s)


PAIRS = {
    "raymarch": lambda: (_march(7, ("axes", 0, 0)), _march(3, ("axes", 0, 0))),
    "insitu": lambda: (_columns(5, ("mxn", 7, 12), colden.FP32, mode=colden.MODE_INSITU),
                       _columns(4, ("axes", 0, 0), colden.FP32, mode=colden.MODE_INSITU)),
    "fp32_leaves_odd": lambda: (_columns(4, ("mxn", 7, 5), colden.FP32), _columns(4, ("mxn", 3, 3), colden.FP32)),
    "fp32_leaves_fours": lambda: (_columns(6, ("mxn", 2, 2), colden.FP32), _columns(6, ("mxn", 5, 4), colden.FP32)),
    "fp32_leaves_wide": lambda: (_columns(3, ("mxn", 25, 21), colden.FP32), _columns(3, ("mxn", 23, 20), colden.FP32)),
    "fp32_lists": lambda: (_amr(("mxn", 15, 12), colden.FP32), _amr(("mxn", 13, 12), colden.FP32)),
    "bf16_leaves": lambda: (_columns(4, ("mxn", 8, 8), colden.BF16), _columns(4, ("mxn", 9, 4), colden.BF16)),
    "bf16_lists": lambda: (_amr(("mxn", 8, 8), colden.BF16), _amr(("mxn", 3, 4), colden.BF16)),
    "bf16_shells": lambda: (_columns(5, ("healpix", 2, 0), colden.BF16, rows=False),
                            _columns(5, ("mxn", 2, 2), colden.BF16, rows=False)),
    "learned": lambda: (_learned(("healpix", 2, 0)), _learned(("mxn", 1, 8))),
}


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_two_threads_launch_the_same_kernels_at_different_sizes(name):
    jobs = PAIRS[name]()
    want = []
    for out, call in jobs:
        call(torch.cuda.current_stream())
        torch.cuda.synchronize()
        want.append(out.clone())
        out.fill_(-1.0)
    torch.cuda.synchronize()
    gate, errors = threading.Barrier(2), []

    def work(call):
        s = torch.cuda.Stream()
        gate.wait()
        end = time.monotonic() + 1.5
        try:
            while not errors and time.monotonic() < end:
                for _ in range(50):
                    call(s)
                s.synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(call,)) for _, call in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    colden.device_status()
    for (out, _), w in zip(jobs, want):
        assert float(w.min()) > 0 and torch.equal(out, w)


@pytest.mark.parametrize("name", ["raymarch_sorted", "raymarch", "small_tree", "tree"])
def test_eager_calls_leave_another_threads_capture_alone(name):
    # a thread captures in the global mode; calls of another one, on a stream of its own,
    # work and do not end that capture
    L = 4 if name == "small_tree" else 6
    t, g = _tree(L, 5), colden.precompute_geometry("healpix", 2)
    s = torch.cuda.Stream()
    if name.startswith("raymarch"):
        n = 100_000 if name == "raymarch_sorted" else 500
        leaves = torch.from_numpy(np.random.default_rng(1).integers(0, t.n_leaf, n)).cuda()
        out = torch.full((n, g.n_dir), -1.0, device="cuda")
        call = lambda: colden.raymarch(t, g, out, leaves=leaves, stream=s)  # noqa: E731
        colden.raymarch(t, g, torch.empty((8, g.n_dir), device="cuda"))     # the module is loaded
    else:
        out = torch.full((t.n_leaf, g.n_dir), -1.0, device="cuda")
        call = lambda: colden.column_density(t, g, n_h=out, stream=s)  # noqa: E731
        call()                                   # the tree's workspace exists
    x, y = torch.ones(4, device="cuda"), torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    out.fill_(-1.0)
    torch.cuda.synchronize()
    capturing, called, errors = threading.Event(), threading.Event(), []

    def capture():
        graph = torch.cuda.CUDAGraph()
        try:
            with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="global"):
                y.copy_(x)
                capturing.set()
                called.wait(60)
                y.add_(x)
            graph.replay()
            torch.cuda.synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
        finally:
            capturing.set()

    th = threading.Thread(target=capture)
    th.start()
    capturing.wait(60)
    try:
        call()
    finally:
        called.set()
        th.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert float(out.min()) > 0 and bool((y == 2).all())

"""The resident-tile FP32 CG where a thread holds a column of several time
slices (large lattices; the small ones of test_gpu_cg_resident have one slice
per column): x after two iterations against the oracle's textbook CG (Section
3), for one and two cells per column, tiles that divide the lattice and ragged
ones, x in registers and x streamed from memory."""
import numpy as np
import pytest

import workloads as W
from oracle import fermion as of
from oracle import solvers as osv
from oracle.lattice import Lattice as OLat

from gpu_util import ctx_for, dev, host, need_gpu, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(51, 51, 64), (75, 67, 61), (97, 101, 63), (72, 72, 64), (98, 100, 62)])
def test_columns_of_several_slices(shape):
    need_gpu()
    w = W.small(*shape, seed=1700 + sum(shape))
    ol = OLat.from_params(w.lat)
    b32 = w.b.astype(np.complex64)
    ref = osv.cg(lambda v: of.apply_MMdag(ol, w.phi, 0.1, v, 0.05), b32.astype(np.complex128), tol=1e-30, maxit=2)
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(7)
        x, info = ctx.solve_spcg(dev(w.phi), 0.1, dev(b32), sigma=0.05, tol=1e-30, maxit=2, allow_fail=True)
        assert ctx.profile_read()["cg_resident_f32"]["launches"] >= 1
        assert ctx.check_guards() == 0
    assert info["iters"] == 2
    # two iterations of FP32 vectors: the bound the per-iteration test uses
    assert rel_max(host(x).astype(np.complex128), ref.x) <= 4e-5


@pytest.mark.parametrize("shape,cols", [((24, 24, 32), 2), ((24, 24, 49), 2), ((25, 23, 30), 1), ((7, 130, 33), 1),
                                        ((40, 5, 70), 2), ((5, 3, 200), 1), ((130, 2, 17), 2)])
def test_one_cluster(shape, cols):
    """The same solve on one thread block cluster (lattices of up to about
    100,000 sites): tiles that divide the lattice and ragged ones, blocks of
    the cluster without a tile, an edge that is its own neighbour."""
    need_gpu()
    w = W.small(*shape, seed=1800 + sum(shape))
    ol = OLat.from_params(w.lat)
    b32 = w.b.astype(np.complex64)
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(7)
        for k in (1, 3):
            ref = osv.cg(lambda v: of.apply_MMdag(ol, w.phi, 0.2, v, 0.1), b32.astype(np.complex128), tol=1e-30,
                         maxit=k)
            x, info = ctx.solve_spcg(dev(w.phi), 0.2, dev(b32), sigma=0.1, tol=1e-30, maxit=k, allow_fail=True)
            assert info["iters"] == k
            assert rel_max(host(x).astype(np.complex128), ref.x) <= 2e-5 * k
        assert ctx.profile_read()["cg_resident_f32"]["design"] == (4 if cols == 2 else 0)
        assert ctx.check_guards() == 0


@pytest.mark.parametrize("shapes", [[(24, 24, 33), (7, 5, 9), (36, 36, 48), (25, 3, 17), (6, 6, 16), (1, 2, 3)],
                                    [(64, 64, 40), (6, 6, 16), (9, 4, 12)],
                                    [(25, 25, 48)] * 10 + [(24, 24, 32)] * 12 + [(13, 13, 32)] * 12])
def test_batched_clusters(shapes):
    """A mixed batch with every system on a cluster of its own (first list), one
    with a lattice that fits no cluster (the cooperative kernels take the whole
    batch), and one of more systems than there is room for at a time (small
    clusters, long columns): each system's true residual by the oracle's operator."""
    need_gpu()
    import paper_1804_07195_gb300 as hmc
    import torch
    systems, refs = [], []
    for k, sh in enumerate(shapes):
        w = W.small(*sh, seed=1900 + k, U=3.0, beta=6.0)
        p = w.lat
        lat = hmc.Lattice(p.n, p.m, p.nt, p.kappa, p.U, p.beta)
        for ms, sigma in ((0.2, 0.0), (1.0, 0.05)):
            systems.append({"lattice": lat, "phi": dev(w.phi), "ms": ms, "sigma": sigma, "b": dev(w.b),
                            "x": torch.empty(p.nsites, dtype=torch.complex128, device="cuda"), "tol": 1e-10})
            refs.append((w, ms, sigma))
    with ctx_for(refs[0][0].lat) as ctx:
        infos = ctx.solve_batched(systems, mixed=True)
        assert ctx.check_guards() == 0
    for s, (w, ms, sigma), info in zip(systems, refs, infos):
        ol = OLat.from_params(w.lat)
        rel = osv.true_rel_residual(lambda v: of.apply_MMdag(ol, w.phi, ms, v, sigma), host(s["x"]), w.b)
        assert rel <= 1.0001e-10 and abs(info["true_rel_res"] - rel) <= 1e-13, (w.name, ms, rel, info)


@pytest.mark.parametrize("shape", [(1, 1, 4), (2, 5, 3), (7, 5, 9), (36, 35, 40), (36, 36, 64), (51, 33, 61),
                                   (72, 40, 64), (33, 120, 64)])
def test_fp64_tiles(shape):
    """The FP64 CG on resident tiles, which runs wherever the tiles fit: x after
    two iterations and from a starting guess against the oracle's CG."""
    need_gpu()
    w = W.small(*shape, seed=2000 + sum(shape))
    ol = OLat.from_params(w.lat)
    A = lambda v: of.apply_MMdag(ol, w.phi, 0.2, v, 0.05)
    k = 1 if w.lat.nsites < 32 else 2
    ref = osv.cg(A, w.b, tol=1e-30, maxit=k)
    x0 = 0.1 * w.b
    ref0 = osv.cg(A, w.b - A(x0), tol=1e-30, maxit=k)
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_cg(dev(w.phi), 0.2, dev(w.b), sigma=0.05, tol=1e-30, maxit=k, allow_fail=True)
        assert info["iters"] == k
        assert rel_max(host(x), ref.x) <= 1e-13
        x, _ = ctx.solve_cg(dev(w.phi), 0.2, dev(w.b), x=dev(x0), sigma=0.05, tol=1e-30, maxit=k, allow_fail=True)
        assert rel_max(host(x), x0 + ref0.x) <= 1e-13
        assert ctx.profile_read()["cg_resident_f64"]["launches"] >= 1
        assert ctx.check_guards() == 0


@pytest.mark.parametrize("shape", [(80, 79, 62), (85, 83, 61), (97, 99, 64), (100, 101, 63)])
def test_x_in_tensor_memory(shape):
    """x kept in tensor memory: two and four slices of cell pairs, four and
    eight of single cells, ragged tiles; the sum over several iterations, so
    that every one of them has been read back and stored."""
    need_gpu()
    w = W.small(*shape, seed=2500 + sum(shape))
    ol = OLat.from_params(w.lat)
    b32 = w.b.astype(np.complex64)
    ref = osv.cg(lambda v: of.apply_MMdag(ol, w.phi, 0.4, v, 0.3), b32.astype(np.complex128), tol=1e-30, maxit=4)
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(7)
        x, info = ctx.solve_spcg(dev(w.phi), 0.4, dev(b32), sigma=0.3, tol=1e-30, maxit=4, allow_fail=True)
        assert ctx.profile_read()["cg_resident_f32"]["launches"] >= 1
        assert ctx.check_guards() == 0
    assert info["iters"] == 4
    # the bound of the other tests, 2e-5 an iteration
    assert rel_max(host(x).astype(np.complex128), ref.x) <= 8e-5


@pytest.mark.parametrize("shape,cols", [((106, 106, 64), 2), ((110, 108, 63), 2), ((99, 99, 64), 1), ((50, 146, 113), 2),
                                        ((117, 75, 70), 1)])
def test_largest_tiles(shape, cols):
    """Tiles that leave no room for the table of their padding in shared memory
    (it lies in global memory): pairs of four and eight slices, single cells,
    tiles whose slices are no multiple of a column's."""
    need_gpu()
    w = W.small(*shape, seed=2700 + sum(shape))
    ol = OLat.from_params(w.lat)
    b32 = w.b.astype(np.complex64)
    ref = osv.cg(lambda v: of.apply_MMdag(ol, w.phi, 0.4, v, 0.3), b32.astype(np.complex128), tol=1e-30, maxit=3)
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(7)
        x, info = ctx.solve_spcg(dev(w.phi), 0.4, dev(b32), sigma=0.3, tol=1e-30, maxit=3, allow_fail=True)
        prof = ctx.profile_read()["cg_resident_f32"]
        assert prof["launches"] >= 1 and prof["design"] == (4 if cols == 2 else 0)
        assert ctx.check_guards() == 0
    assert info["iters"] == 3
    assert rel_max(host(x).astype(np.complex128), ref.x) <= 6e-5

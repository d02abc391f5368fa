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

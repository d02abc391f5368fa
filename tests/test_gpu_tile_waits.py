"""The bounded waits of the resident-tile CG (blocks of a cooperative launch over
all SMs, and of thread block clusters): with the test hook every wait is for a
sum that nobody sends, the solve returns HMC_ERR_TIMEOUT after about a
millisecond, and the same context then solves normally."""
import time

import numpy as np
import pytest

import workloads as W
from oracle import fermion as of
from oracle.lattice import Lattice as OLat

from gpu_util import ctx_for, dev, host, need_gpu

pytestmark = pytest.mark.gpu


def times_out(ctx, solve):
    import paper_1804_07195_gb300 as hmc
    ctx.set_wait_test(1, 2_000_000)
    t = time.perf_counter()
    with pytest.raises(hmc.HMCError) as e:
        solve()
    assert e.value.status == hmc._abi.HMC_ERR_TIMEOUT
    assert time.perf_counter() - t < 1.0
    ctx.set_wait_test(0, 0)


@pytest.mark.parametrize("shape", [(6, 6, 16), (5, 3, 9), (24, 24, 33)])
@pytest.mark.parametrize("where", [1, 2])
def test_fp32_tiles(shape, where):
    need_gpu()
    w = W.small(*shape, seed=2600 + sum(shape))
    ol = OLat.from_params(w.lat)
    b32 = dev(w.b.astype(np.complex64))
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(7)
        ctx.set_tile_test(where)
        solve = lambda: ctx.solve_spcg(dev(w.phi), 0.3, b32, tol=1e-6)
        times_out(ctx, solve)
        x, info = solve()
        assert (ctx.profile_read()["cg_resident_f32"]["waves"] < 0) == (where == 2)
    b = w.b.astype(np.complex64).astype(np.complex128)
    r = b - of.apply_MMdag(ol, w.phi, 0.3, host(x).astype(np.complex128))
    assert info["status"] == 0 and np.linalg.norm(r) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("shape", [(6, 6, 16), (5, 3, 9), (24, 24, 33)])
def test_fp64_tiles(shape):
    need_gpu()
    w = W.small(*shape, seed=2610 + sum(shape))
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        solve = lambda: ctx.solve_cg(dev(w.phi), 0.3, dev(w.b), tol=1e-10)
        times_out(ctx, solve)
        x, info = solve()
        assert ctx.profile_read()["cg_resident_f64"]["launches"] == 2
    r = w.b - of.apply_MMdag(ol, w.phi, 0.3, host(x))
    assert info["status"] == 0 and np.linalg.norm(r) <= 1.0001e-10 * np.linalg.norm(w.b)


def test_batched_clusters():
    """A mixed batch whose systems run on clusters of different sizes."""
    need_gpu()
    import paper_1804_07195_gb300 as hmc
    import torch
    ws = [W.small(*sh, seed=2620 + k, U=3.0, beta=6.0) for k, sh in enumerate([(6, 6, 16), (24, 24, 33), (5, 3, 9)])]

    def systems():
        return [{"lattice": hmc.Lattice(w.lat.n, w.lat.m, w.lat.nt, w.lat.kappa, w.lat.U, w.lat.beta), "phi": dev(w.phi),
                 "ms": 0.3, "b": dev(w.b), "x": torch.zeros(w.lat.nsites, dtype=torch.complex128, device="cuda")}
                for w in ws]
    with ctx_for(ws[0].lat) as ctx:
        times_out(ctx, lambda: ctx.solve_batched(systems(), mixed=True))
        sy = systems()
        ctx.solve_batched(sy, mixed=True)
    for w, s in zip(ws, sy):
        r = w.b - of.apply_MMdag(OLat.from_params(w.lat), w.phi, 0.3, host(s["x"]))
        assert np.linalg.norm(r) <= 1.0001e-10 * np.linalg.norm(w.b)

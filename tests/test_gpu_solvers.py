"""Parity of the CUDA solvers (Section 3, Algorithm A.1): the true residual
|b - A x| / |b| evaluated by the oracle's operator is within the requested 1e-10,
and the solution agrees with the oracle's LU solve on small lattices."""
import numpy as np
import pytest

import workloads as W
from oracle import fermion as of
from oracle import solvers as osv
from oracle.lattice import Lattice as OLat

from gpu_util import ctx_for, dev, host, need_gpu, rel_max, torch

pytestmark = pytest.mark.gpu


def true_rel(ol, phi, ms, sigma, x, b):
    return osv.true_rel_residual(lambda v: of.apply_MMdag(ol, phi, ms, v, sigma), x, b)


@pytest.mark.parametrize("name,ms,sigma", [("L6x6x16", 0.0, 0.0), ("L6x6x16", 0.3, 0.0), ("L6x6x16", 0.0, 0.09)])
def test_cg_fp64_matches_lu(name, ms, sigma):
    need_gpu()
    w = W.workload(name)
    ol = OLat.from_params(w.lat)
    D = of.dense_M(ol, w.phi, ms)
    x_ref = osv.dense_solve(D @ D.conj().T + sigma * np.eye(ol.N), w.b)
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_cg(dev(w.phi), ms, dev(w.b), sigma=sigma, tol=1e-10)
    x = host(x)
    assert true_rel(ol, w.phi, ms, sigma, x, w.b) <= 1e-10
    assert abs(info["true_rel_res"] - true_rel(ol, w.phi, ms, sigma, x, w.b)) < 1e-12
    assert np.linalg.norm(x - x_ref) <= 1e-7 * np.linalg.norm(x_ref)
    # the oracle's CG takes the same path: iteration counts agree closely
    ref = osv.cg(lambda v: of.apply_MMdag(ol, w.phi, ms, v, sigma), w.b, tol=1e-10)
    assert abs(info["iters"] - ref.iters) <= 2


def test_cg_initial_guess_and_zero_rhs():
    need_gpu()
    w = W.workload("L6x6x16")
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        phi, b = dev(w.phi), dev(w.b)
        x, _ = ctx.solve_cg(phi, 0.0, b, tol=1e-10)
        x2, info = ctx.solve_cg(phi, 0.0, b, x=x.clone(), tol=1e-10)
        assert info["iters"] <= 1
        z, info = ctx.solve_cg(phi, 0.0, torch.zeros_like(b), tol=1e-10)
        assert info["iters"] == 0 and torch.count_nonzero(z) == 0


def test_spcg_fp32():
    need_gpu()
    w = W.workload("L6x6x16")
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_spcg(dev(w.phi), 0.2, dev(w.b.astype(np.complex64)), tol=1e-5)
    assert true_rel(ol, w.phi, 0.2, 0.0, host(x).astype(np.complex128), w.b.astype(np.complex64)) < 2e-5


@pytest.mark.parametrize("name,ms", [("L6x6x16", 0.0), ("L36x36x64", 0.0), ("L36x36x64", 0.5)])
def test_fgmres_mixed_true_residual(name, ms):
    need_gpu()
    w = W.workload(name)
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_fgmres(dev(w.phi), ms, dev(w.b), tol=1e-10)
        xc, infoc = ctx.solve_cg(dev(w.phi), ms, dev(w.b), tol=1e-10)
    x = host(x)
    assert true_rel(ol, w.phi, ms, 0.0, x, w.b) <= 1e-10
    assert info["iters_inner"] > 0 and info["applies32"] > info["applies64"]
    # both solutions agree within what the residual bound allows
    assert np.linalg.norm(x - host(xc)) <= 1e-6 * np.linalg.norm(x)


def test_fgmres_iteration_structure_matches_oracle():
    """Same Algorithm A.1 on both sides. FP32 rounding inside the inner solves
    differs, so a restart that ends just above or just below TOL |b| on one side
    may be repeated on the other: restarts agree within one, Arnoldi steps and
    inner iterations closely."""
    need_gpu()
    w = W.workload("L6x6x16")
    ol = OLat.from_params(w.lat)
    A64 = lambda v: of.apply_MMdag(ol, w.phi, 0.0, v)
    A32 = lambda v: of.apply_MMdag(ol, w.phi, 0.0, v.astype(np.complex64)).astype(np.complex64)
    ref = osv.fgmres(A64, A32, w.b, tol=1e-10)
    with ctx_for(w.lat) as ctx:
        _, info = ctx.solve_fgmres(dev(w.phi), 0.0, dev(w.b), tol=1e-10)
    assert abs(info["iters_outer"] - ref.outer_iters) <= 1, (info, ref.outer_iters)
    # after the last preconditioned step the unpreconditioned tail's length
    # depends on where FP32 rounding leaves the residual relative to a TOL |b|;
    # an extra restart on one side adds up to m = 10 steps
    dsteps = abs(info["iters"] - ref.iters)
    assert dsteps <= max(3, 0.5 * ref.iters) + 10 * abs(info["iters_outer"] - ref.outer_iters), (info, ref.iters)
    assert abs(info["iters_inner"] - ref.inner_iters) <= 0.2 * ref.inner_iters, (info, ref.inner_iters)


def test_fgmres_fp64_inner_and_no_preconditioning():
    need_gpu()
    w = W.small(3, 3, 8, seed=3)
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_fgmres(dev(w.phi), 0.0, dev(w.b), tol=1e-11, inner_prec=64)
        assert true_rel(ol, w.phi, 0.0, 0.0, host(x), w.b) <= 1e-11
        x, info = ctx.solve_fgmres(dev(w.phi), 0.0, dev(w.b), tol=0.25)
        assert info["iters_inner"] == 0
        assert true_rel(ol, w.phi, 0.0, 0.0, host(x), w.b) <= 0.25


def test_not_converged_is_reported():
    need_gpu()
    import paper_1804_07195_gb300 as hmc
    w = W.workload("L6x6x16")
    with ctx_for(w.lat) as ctx:
        with pytest.raises(hmc.HMCError) as e:
            ctx.solve_cg(dev(w.phi), 0.0, dev(w.b), tol=1e-10, maxit=5)
        assert e.value.status == -3
        x, info = ctx.solve_cg(dev(w.phi), 0.0, dev(w.b), tol=1e-10, maxit=5, allow_fail=True)
        assert info["iters"] == 5 and info["true_rel_res"] > 1e-10


@pytest.mark.parametrize("name,ms", [("L6x6x16", 0.0), ("L36x36x64", 0.2)])
def test_fcg_mixed(name, ms):
    """Flexible CG with the FP32 CG preconditioner (Section 3) against the
    oracle's flexible CG: both converge, in a similar number of outer steps, and
    the true residual meets the tolerance up to the drift of the recursive one."""
    need_gpu()
    w = W.workload(name)
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_fcg(dev(w.phi), ms, dev(w.b), tol=1e-10)
    assert true_rel(ol, w.phi, ms, 0.0, host(x), w.b) <= 2e-10
    assert info["iters_inner"] > 0
    if name == "L6x6x16":
        A64 = lambda v: of.apply_MMdag(ol, w.phi, ms, v)
        A32 = lambda v: of.apply_MMdag(ol, w.phi, ms, v.astype(np.complex64)).astype(np.complex64)
        ref = osv.fcg(A64, A32, w.b, tol=1e-10)
        # once TOL a |b| / |r| >= 1 the steps are unpreconditioned (z = r) and
        # the length of that tail depends on FP32 rounding inside the spCG solves
        assert abs(info["iters"] - ref.iters) <= max(3, 0.5 * ref.iters)
        assert abs(info["iters_inner"] - ref.inner_iters) <= 0.2 * ref.inner_iters


@pytest.mark.parametrize("variant", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("name,ms,sigma,bound", [("L36x36x64", 0.0, 0.0, 1e-3), ("L36x36x64", 0.4, 0.05, 5e-5),
                                                 ("L102x102x64", 0.1, 0.0, 1e-3), ("L36x36x21", 0.2, 0.0, 1e-4),
                                                 ("L35x12x16", 0.2, 0.0, 1e-4)])
def test_fp32_cg_kernel_variants(variant, name, ms, sigma, bound):
    """The FP32 CG kernel designs (grid-stride, shared-memory tiled, marching,
    persistent, grid-stride with two cells per thread, single-reduction,
    resident tiles) solve
    to the single-precision floor, and FGMRES built on them meets 1e-10. The
    FP32 solution's true residual is bounded by the recursive tolerance plus
    the rounding drift, about eps_32 times the condition number (near 10^4 at
    m_s = 0 on a 64-slice lattice, where lambda_min = 4 sin^2(pi / 128)). The
    21-slice lattice leaves a ragged last block of time slices for every slice
    count per block the tiled and marching kernels can take (2, 4, 8), and a
    ragged last block of cells."""
    need_gpu()
    if name == "L36x36x21":
        w = W.small(36, 36, 21, seed=2121, U=3.0, beta=6.0)
    elif name == "L35x12x16":  # odd n: no cell pairs, variant 5 takes one cell per thread
        w = W.small(35, 12, 16, seed=3512, U=3.0, beta=6.0)
    else:
        w = W.workload(name)
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(variant)
        x32, info = ctx.solve_spcg(dev(w.phi), ms, dev(w.b.astype(np.complex64)), sigma=sigma, tol=1e-5, maxit=5000)
        shapes = ctx.profile_read()
        x, finfo = ctx.solve_fgmres(dev(w.phi), ms, dev(w.b), sigma=sigma, tol=1e-10, a=1.0)
    waves = shapes["cg_pMdag_f32"]["waves"]
    design = shapes["cg_pMdag_f32"]["design"]
    persist = shapes["cg_persist_f32"]["launches"]
    single = shapes["cg1_fused_f32"]["launches"]
    resident = shapes["cg_resident_f32"]["launches"]
    assert {1: waves >= 0 and design == 0, 2: -1000 < waves < 0, 3: waves <= -1000, 4: True,
            5: waves >= 0 and design == (4 if w.lat.n % 2 == 0 else 0), 6: True, 7: True}[variant]
    assert (persist > 0) == (variant == 4)
    assert (single > 0) == (variant == 6)
    assert (resident > 0) == (variant == 7)
    b32 = w.b.astype(np.complex64).astype(np.complex128)
    assert info["iters"] > 0 and info["status"] == 0
    assert true_rel(ol, w.phi, ms, sigma, host(x32).astype(np.complex128), b32) < bound
    assert true_rel(ol, w.phi, ms, sigma, host(x), w.b) <= 1e-10


def test_solves_run_as_one_graph_launch_with_a_device_loop():
    """After a solve by three kernels an iteration the context reports the
    device-side loop graph (one graph launch per CG solve), and a second solve
    through the cached loop graph gives the same result bit for bit (FP64 CG is
    deterministic)."""
    need_gpu()
    w = W.workload("L6x6x16")
    with ctx_for(w.lat) as ctx:
        ctx.set_tile_test(3)  # small lattices would run on resident tiles, without a graph
        x1, i1 = ctx.solve_cg(dev(w.phi), 0.3, dev(w.b), tol=1e-10)
        assert ctx.graph_mode() == 2
        x2, i2 = ctx.solve_cg(dev(w.phi), 0.3, dev(w.b), tol=1e-10)
        ctx.set_graph_mode(1)  # chunks with host checks: the same iterations
        assert ctx.graph_mode() == 1
        x3, i3 = ctx.solve_cg(dev(w.phi), 0.3, dev(w.b), tol=1e-10)
        prof = ctx.profile_read()
        assert prof["cg_resident_f64"]["launches"] == 0 and prof["cg_Mdag_f64"]["launches"] >= 3 * i1["iters"]
    assert i1["iters"] == i2["iters"] == i3["iters"]
    assert np.array_equal(host(x1), host(x2)) and np.array_equal(host(x1), host(x3))


def test_spcg_two_cell_kernels_with_an_unaligned_solution_vector():
    """The two-cells-per-thread FP32 CG kernels access x in 16-byte units; a
    caller's x that is only 8-byte aligned is solved in a workspace vector and
    copied, with the same iterates as an aligned x."""
    need_gpu()
    w = W.small(12, 12, 32, seed=1212, U=3.0, beta=6.0)
    N = w.lat.nsites
    ol = OLat.from_params(w.lat)
    import paper_1804_07195_gb300 as hmc
    from paper_1804_07195_gb300 import _abi
    import ctypes as C
    b32 = dev(w.b.astype(np.complex64))
    with ctx_for(w.lat) as ctx:
        ctx.set_cg_variant(5)
        xa, ia = ctx.solve_spcg(dev(w.phi), 0.1, b32, tol=1e-5, maxit=5000)
        buf = torch.zeros(N + 1, dtype=torch.complex64, device="cuda")
        info = _abi.hmc_solve_info()
        st = ctx.lib.hmc_solve_spcg(ctx.h, C.c_void_p(dev(w.phi).data_ptr()), 0.1, 0.0, C.c_void_p(b32.data_ptr()),
                                    C.c_void_p(buf[1:].data_ptr()), 1e-5, 5000, C.byref(info))
        torch.cuda.synchronize()
        assert st == 0 and ctx.profile_read()["cg_pMdag_f32"]["design"] == 4
    assert info.iters == ia["iters"]
    assert np.array_equal(host(buf[1:]), host(xa))
    assert true_rel(ol, w.phi, 0.1, 0.0, host(buf[1:]).astype(np.complex128), w.b.astype(np.complex64).astype(np.complex128)) < 1e-4


@pytest.mark.parametrize("shape,steps", [((3, 5, 7), 1), ((3, 5, 7), 16), ((6, 6, 16), 7), ((34, 35, 66), 16),
                                         ((51, 51, 64), 10), ((70, 71, 64), 3), ((70, 71, 64), 16)])
def test_arnoldi_steps_against_numpy(shape, steps):
    """x after one cycle of 1 .. 16 unpreconditioned steps (a tol >= 1) against
    GMRES in numpy: the dots and updates of every basis size, on lattices with
    fewer sites than threads and on both sides of the block counts' rules."""
    need_gpu()
    w = W.small(*shape, seed=2100 + sum(shape))
    ol = OLat.from_params(w.lat)
    A = lambda v: of.apply_MMdag(ol, w.phi, 0.3, v, 5.0)
    V = [w.b / np.linalg.norm(w.b)]
    H = np.zeros((steps + 1, steps), complex)
    for j in range(steps):
        q = A(V[j])
        for _ in range(2):
            for i in range(j + 1):
                h = np.vdot(V[i], q)
                H[i, j] += h
                q = q - h * V[i]
        H[j + 1, j] = np.linalg.norm(q)
        V.append(q / H[j + 1, j])
    e = np.zeros(steps + 1, complex)
    e[0] = np.linalg.norm(w.b)
    y = np.linalg.lstsq(H, e, rcond=None)[0]
    ref = sum(y[i] * V[i] for i in range(steps))
    with ctx_for(w.lat) as ctx:
        x, info = ctx.solve_fgmres(dev(w.phi), 0.3, dev(w.b), sigma=5.0, tol=1e-30, restart=16, a=1e32, maxit=steps,
                                   allow_fail=True)
    assert info["iters"] == steps and info["iters_inner"] == 0
    # cond(H) < 10: the normal equations and one pass of Gram-Schmidt lose its square,
    # 100 x 2.2e-16 x 16 steps = 4e-13; five times that
    assert np.linalg.norm(host(x) - ref) <= 2e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("shape", [(3, 3, 8), (7, 5, 9), (12, 12, 32), (35, 12, 21)])
@pytest.mark.parametrize("ms,sigma", [(0.0, 0.0), (0.3, 0.0), (0.0, 0.2), (0.1, 0.2)])
def test_fp64_three_kernel_iterates(shape, ms, sigma):
    """The FP64 CG of three kernels an iteration (lattices whose tiles do not fit
    the chip), with an instance for each of mass and shift zero or not: x after
    a few iterations, from zero and from a guess, against the oracle's CG."""
    need_gpu()
    w = W.small(*shape, seed=2150 + sum(shape))
    ol = OLat.from_params(w.lat)
    A = lambda v: of.apply_MMdag(ol, w.phi, ms, v, sigma)
    with ctx_for(w.lat) as ctx:
        ctx.set_tile_test(3)
        for x0 in (None, 0.1 * w.b):
            ref = osv.cg(A, w.b if x0 is None else w.b - A(x0), tol=1e-30, maxit=4).x
            if x0 is not None:
                ref = x0 + ref
            x, info = ctx.solve_cg(dev(w.phi), ms, dev(w.b), x=None if x0 is None else dev(x0), sigma=sigma, tol=1e-30,
                                   maxit=4, allow_fail=True)
            assert info["iters"] == 4
            assert rel_max(host(x), ref) <= 2e-13  # 5e-14 an iteration, as for the tiles
        prof = ctx.profile_read()
        assert prof["cg_resident_f64"]["launches"] == 0 and prof["cg_Mdag_f64"]["launches"] >= 8

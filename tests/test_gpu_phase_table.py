"""The FP64 phase table e^{i phi} (table lookup and short series) and the float
copy of phi, through M: fields from denormal to beyond the range of the fast
path (|phi| >= 1e5), at the edges of its reduction (multiples of 2 pi / 1024 and
half way between), +-pi, infinities and NaN, against the oracle's operator."""
import numpy as np
import pytest

import workloads as W
from oracle import fermion as of
from oracle.lattice import Lattice as OLat

from gpu_util import ctx_for, dev, host, need_gpu

pytestmark = pytest.mark.gpu


def fields(n):
    g = np.random.Generator(np.random.PCG64(31))
    step = 2 * np.pi / 1024
    k = g.integers(-5000, 5000, n)
    edge = np.where(g.random(n) < 0.5, k * step, (k + 0.5) * step)
    yield "small", g.normal(0.0, 1e-3, n) * 10.0 ** g.integers(-300, 1, n)
    yield "unit", g.normal(0.0, 1.0, n)
    yield "edges", np.nextafter(edge, np.where(g.random(n) < 0.5, -9e9, 9e9))
    yield "pi", np.pi * g.choice([-1.0, 1.0], n) * (1.0 + g.integers(-2, 3, n) * 2.0 ** -52)
    yield "large", g.uniform(-1.2e5, 1.2e5, n)
    yield "huge", g.normal(0.0, 1.0, n) * 1e12


@pytest.mark.parametrize("shape", [(6, 5, 8), (13, 4, 7)])
def test_phases(shape):
    need_gpu()
    w = W.small(*shape, seed=2100)
    ol = OLat.from_params(w.lat)
    with ctx_for(w.lat) as ctx:
        for name, phi in fields(w.lat.nsites):
            for ms in (0.0, 0.3):
                # cos and sin within an ulp each, a few roundings in the row
                got = host(ctx.apply_M(dev(phi), ms, dev(w.b)))
                assert np.abs(got - of.apply_M(ol, phi, ms, w.b)).max() <= 4e-15 * np.abs(w.b).max(), (name, ms)
                got = host(ctx.apply_Mdag(dev(phi), ms, dev(w.b)))
                assert np.abs(got - of.apply_Mdag(ol, phi, ms, w.b)).max() <= 4e-15 * np.abs(w.b).max(), (name, ms)
            # the float copy: phi less a multiple of 2 pi as a double (2.5e-16 off, times
            # |phi| / 2 pi: 4e-17 |phi|, and as much by rounding), rounded to float within
            # [-pi, pi] (half an ulp of pi, 1.2e-7), hardware sine and cosine (4e-7), FP32 rows
            got = host(ctx.apply_M(dev(phi), 0.0, dev(w.b.astype(np.complex64))))
            bound = 3e-6 + 2e-16 * np.abs(phi).max()
            assert np.abs(got - of.apply_M(ol, phi, 0.0, w.b)).max() <= bound * np.abs(w.b).max(), name


def test_phases_of_no_number():
    need_gpu()
    w = W.small(4, 4, 6, seed=2101)
    ol = OLat.from_params(w.lat)
    phi = w.phi.copy()
    phi[[3, 50, 100]] = [np.nan, np.inf, -np.inf]
    with np.errstate(invalid="ignore"):
        ref = of.apply_M(ol, phi, 0.0, w.b)
    with ctx_for(w.lat) as ctx:
        got = host(ctx.apply_M(dev(phi), 0.0, dev(w.b)))
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.isnan(ref).sum() == 3
    ok = ~np.isnan(ref)
    assert np.abs(got[ok] - ref[ok]).max() <= 4e-15 * np.abs(w.b).max()


def test_neighbour_sums():
    """The integer sums of three neighbours in the FP64 stencils: entries spread
    over 80 binary orders, cancelling, zero, denormal, infinite and NaN."""
    need_gpu()
    w = W.small(7, 6, 5, seed=2102)
    ol = OLat.from_params(w.lat)
    g = np.random.Generator(np.random.PCG64(32))
    n = w.lat.nsites
    z = lambda a: a[:n] + 1j * a[n:]
    r = g.normal(size=2 * n)
    vecs = {"plain": z(r), "spread": z(r * 2.0 ** g.integers(-40, 41, 2 * n)),
            "cancel": z(np.round(r * 4) / 4), "zeros": z(np.where(g.random(2 * n) < 0.7, 0.0, r)),
            "tiny": z(r * 1e-305), "large": z(r * 1e300)}
    with ctx_for(w.lat) as ctx:
        for name, v in vecs.items():
            for ms in (0.0, 0.4):
                for f, o in ((ctx.apply_M, of.apply_M), (ctx.apply_Mdag, of.apply_Mdag)):
                    ref = o(ol, w.phi, ms, v)
                    assert np.abs(host(f(dev(w.phi), ms, dev(v))) - ref).max() <= 4e-15 * np.abs(v).max(), (name, ms)
        # M(-v) = -M v bit for bit: no bias towards one sign
        for v in (vecs["plain"], vecs["spread"]):
            for f in (ctx.apply_M, ctx.apply_Mdag):
                assert np.array_equal(host(f(dev(w.phi), 0.0, dev(-v))), -host(f(dev(w.phi), 0.0, dev(v))))
        v = z(r)
        v[[5, 60]] = [np.nan, np.inf]
        with np.errstate(invalid="ignore"):
            ref = of.apply_M(ol, w.phi, 0.0, v)
        got = host(ctx.apply_M(dev(w.phi), 0.0, dev(v)))
        assert np.array_equal(np.isfinite(got), np.isfinite(ref))


@pytest.mark.parametrize("fixed_point", [20, 40])
def test_exact_sums_stay_exact(fixed_point):
    """Entries that are small whole multiples of a power of two, most of them
    zero, phi = 0 and a power of two as hopping: every product and sum of the
    operator is exact in FP64, cancelling ones included, and must come out so."""
    need_gpu()
    w = W.small(6, 5, 8, seed=2103, U=2.0, beta=2.0)  # delta kappa = 1/4
    ol = OLat.from_params(w.lat)
    g = np.random.Generator(np.random.PCG64(33))
    n = w.lat.nsites
    zero = np.zeros(n)
    draw = lambda: np.where(g.random(n) < 0.6, 0.0, g.integers(-3, 4, n) * 2.0 ** -(fixed_point * g.integers(0, 2, n)))
    with ctx_for(w.lat) as ctx:
        for _ in range(3):
            v = draw() + 1j * draw()
            for f, o in ((ctx.apply_M, of.apply_M), (ctx.apply_Mdag, of.apply_Mdag)):
                assert np.array_equal(host(f(dev(zero), 0.0, dev(v))), o(ol, zero, 0.0, v))

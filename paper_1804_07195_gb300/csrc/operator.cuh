// The fermion operator M[phi; m_s] of Eq. ferm_op and its adjoint, as device
// code. One thread handles one cell-time q: the A row q and the B row H + q.
//
//   (M u)_A(x,t)  = -u_A(x,t) + s (e^{+i phi_A(x,t)} - delta m_s) u_A(x,t-1)
//                   - delta kappa [u_B(i,j) + u_B(i-1,j) + u_B(i,j-1)](t)
//   (M u)_B(x,t)  = +u_B(x,t) - s (e^{-i phi_B(x,t)} - delta m_s) u_B(x,t+1)
//                   - delta kappa [u_A(i,j) + u_A(i+1,j) + u_A(i,j+1)](t)
//   (M^+ p)_A(x,t) = -p_A(x,t) + s (e^{-i phi_A(x,t+1)} - delta m_s) p_A(x,t+1) - delta kappa sum_B
//   (M^+ p)_B(x,t) = +p_B(x,t) - s (e^{+i phi_B(x,t-1)} - delta m_s) p_B(x,t-1) - delta kappa sum_A
// with s = -1 on the hop that wraps around the time circle (anti-periodic).
#pragma once

#include "common.cuh"

namespace hmc {

// e^{i phi_k}. FP64: read from a table built once per field. FP32: computed
// from the field rounded to float, with the argument reduced to [-pi, pi] and
// the hardware sine/cosine (absolute error about 4e-7 there), which is below
// what the single-precision inner solver needs.
template <typename R>
struct Phase;

template <>
struct Phase<double> {
  const double2* E;
  __device__ __forceinline__ Cx<double> operator()(int k) const {
    double2 e = E[k];
    return Cx<double>{e.x, e.y};
  }
};

template <>
struct Phase<float> {
  const float* phi;
  __device__ __forceinline__ Cx<float> operator()(int k) const {
    float s, c;
    __sincosf(phi[k], &s, &c);  // phi in [-pi, pi] (phi_to_f32)
    return Cx<float>{c, s};
  }
};

// c + z v with fused multiply-adds.
template <typename R>
__device__ __forceinline__ Cx<R> cfma(Cx<R> z, Cx<R> v, Cx<R> c) {
  Cx<R> o;
  o.re = fma(z.re, v.re, fma(-z.im, v.im, c.re));
  o.im = fma(z.re, v.im, fma(z.im, v.re, c.im));
  return o;
}

// One addend of sum3 as a fixed-point number whose scale is that of the exponent
// field em (the leading bit of a number of that exponent is bit 60), bits below cut
// off its magnitude. A negative one comes as its ones' complement, one too low:
// sum3 adds the three ones at once.
__device__ __forceinline__ long long sum3_aligned(double a, int em) {
  const int h = __double2hiint(a);
  const int d = (int)((unsigned)(em - (h & 0x7ff00000)) >> 20);
  const unsigned long long m =
      ((unsigned long long)(unsigned)((h & 0x000fffff) | 0x00100000) << 32) | (unsigned)__double2loint(a);
  return (long long)((m << 8) >> min(d, 63)) ^ (long long)(h >> 31);
}

// Out of line, or its additions would be issued (with a false predicate) beside
// every integer sum and take the FP64 pipe all the same.
static __device__ __noinline__ double sum3_rare(double a, double b, double c) { return (a + b) + c; }

// a + b + c in integer arithmetic, rounded once, to nearest and ties to even:
// 61-bit addends relative to the largest, so the error is below 0.5 ulp of the sum
// plus 2/256 ulp of the largest addend, where two FP64 additions may err by 1 ulp.
// Over addends of N(0, 1): rms error 8.4e-17, two additions 1.14e-16; no bias,
// and the sum of the negated addends is the negated sum. What two additions
// do better is a small addend behind two that cancel: they give 1 - 1 + 1e-10
// exactly, here it loses what lies below 2^-60 of the ones (1e-10 - 1 + 1, which two
// additions round at 2^-53, is no worse here). The FP64 pipe of this GPU takes 16
// cycles for a warp's addition, and the integer one is idle.
__device__ __forceinline__ double sum3(double a, double b, double c) {
  const int em = max(max(__double2hiint(a) & 0x7ff00000, __double2hiint(b) & 0x7ff00000), __double2hiint(c) & 0x7ff00000);
  // infinities, NaN, sums that may overflow, the smallest normal numbers and zeros
  if ((unsigned)(em - 0x04000000) >= 0x7bc00000u) return sum3_rare(a, b, c);
  const int minus = (__double2hiint(a) >> 31) + (__double2hiint(b) >> 31) + (__double2hiint(c) >> 31);
  const long long v = sum3_aligned(a, em) + sum3_aligned(b, em) + sum3_aligned(c, em) - minus;
  const long long s = v >> 63;
  const unsigned long long w = (unsigned long long)((v ^ s) - s);
  const int lz = __clzll((long long)w);  // at least 1
  const unsigned long long x = (w << (lz & 63)) >> 1;
  const unsigned long long r = (x + (0x1ffu + ((unsigned)x >> 10 & 1u))) >> 10;  // 53 bits
  const int e = em + ((2 - lz) << 20);
  const unsigned long long bits =
      (r + ((unsigned long long)(unsigned)e << 32)) | ((unsigned long long)s & 0x8000000000000000ull);
  return w ? __longlong_as_double((long long)bits) : 0.0;
}
__device__ __forceinline__ float sum3(float a, float b, float c) { return a + b + c; }

// t - dk (a + b + c)
template <typename R>
__device__ __forceinline__ Cx<R> hopsum(Cx<R> t, R dk, Cx<R> a, Cx<R> b, Cx<R> c) {
  Cx<R> o;
  o.re = fma(-dk, sum3(a.re, b.re, c.re), t.re);
  o.im = fma(-dk, sum3(a.im, b.im, c.im), t.im);
  return o;
}

template <typename R>
struct PairOut {
  Cx<R> a, b;
};

// The time-hop factors +-(cos phi - dm, +-sin phi): MASS = false for dm = 0, which
// then costs no subtraction (1 of the 8 FP64 instructions left in a row).
template <bool MASS, typename R>
__device__ __forceinline__ R less_dm(R x, R dm) {
  return MASS ? x - dm : x;
}
__device__ __forceinline__ float neg_of(float a) { return -a; }
__device__ __forceinline__ double neg_of(double a) { return dneg_if(a, true); }
// the factor (e.re - dm, sign e.im), negated where neg
template <bool MASS, typename R>
__device__ __forceinline__ Cx<R> time_factor(Cx<R> e, R dm, bool conj, bool neg) {
  const Cx<R> z = cneg_if(Cx<R>{less_dm<MASS>(e.re, dm), e.im}, neg);
  return Cx<R>{z.re, conj ? neg_of(z.im) : z.im};
}

// M^dagger applied at the cell-time of nb, reading p (precision R); PH is any
// functor returning e^{i phi_k}.
template <typename R, typename PH = Phase<R>, bool MASS = true>
__device__ __forceinline__ PairOut<R> mdag_pair(const Geo& g, const PH& ph, R dm,
                                                const typename Vec2<R>::type* __restrict__ p,
                                                const Nbr& nb) {
  const int H = g.H;
  const R dk = geo_dk(g, R(0));
  Cx<R> pa = ld<R>(p, nb.q), pb = ld<R>(p, H + nb.q);
  // A row: time partner (x, t+1), phase of A at t+1, conjugated
  Cx<R> za = time_factor<MASS>(ph(nb.tp), dm, true, nb.wrap_tp);
  Cx<R> ta = cfma(za, ld<R>(p, nb.tp), Cx<R>{-pa.re, -pa.im});
  Cx<R> oa = hopsum(ta, dk, pb, ld<R>(p, H + nb.im1), ld<R>(p, H + nb.jm1));
  // B row: time partner (x, t-1), phase of B at t-1; the hop carries a minus sign
  Cx<R> zb = time_factor<MASS>(ph(H + nb.tm), dm, false, !nb.wrap_tm);
  Cx<R> tb = cfma(zb, ld<R>(p, H + nb.tm), pb);
  Cx<R> ob = hopsum(tb, dk, pa, ld<R>(p, nb.ip1), ld<R>(p, nb.jp1));
  return PairOut<R>{oa, ob};
}

// M^dagger at the cell-time of nb of the vector returned by the loader L, with
// the time-hop factors za (A row) and zb (B row) already formed; used where
// the same stencil is applied to two vectors.
template <typename R, typename LD>
__device__ __forceinline__ PairOut<R> mdag_pair_ld(const Geo& g, Cx<R> za, Cx<R> zb, R dk, const Nbr& nb,
                                                   LD L) {
  const int H = g.H;
  Cx<R> pa = L(nb.q), pb = L(H + nb.q);
  Cx<R> ta = cfma(za, L(nb.tp), Cx<R>{-pa.re, -pa.im});
  Cx<R> oa = hopsum(ta, dk, pb, L(H + nb.im1), L(H + nb.jm1));
  Cx<R> tb = cfma(zb, L(H + nb.tm), pb);
  Cx<R> ob = hopsum(tb, dk, pa, L(nb.ip1), L(nb.jp1));
  return PairOut<R>{oa, ob};
}

// M at the cell-time of nb of the vector returned by the loader L (phases
// from ph); used where the loads need a particular cache policy.
template <typename R, typename PH, typename LD>
__device__ __forceinline__ PairOut<R> m_pair_ld(const Geo& g, const PH& ph, R dm, const Nbr& nb, LD L) {
  const int H = g.H;
  const R dk = geo_dk(g, R(0));
  Cx<R> ua = L(nb.q), ub = L(H + nb.q);
  Cx<R> ea = ph(nb.q);
  Cx<R> za = cneg_if(Cx<R>{ea.re - dm, ea.im}, nb.wrap_tm);
  Cx<R> ta = cfma(za, L(nb.tm), Cx<R>{-ua.re, -ua.im});
  Cx<R> oa = hopsum(ta, dk, ub, L(H + nb.im1), L(H + nb.jm1));
  Cx<R> eb = ph(H + nb.q);
  Cx<R> zb = cneg_if(Cx<R>{dm - eb.re, eb.im}, nb.wrap_tp);
  Cx<R> tb = cfma(zb, L(H + nb.tp), ub);
  Cx<R> ob = hopsum(tb, dk, ua, L(nb.ip1), L(nb.jp1));
  return PairOut<R>{oa, ob};
}

// M applied at the cell-time of nb, reading u (precision R).
template <typename R, typename PH = Phase<R>, bool MASS = true>
__device__ __forceinline__ PairOut<R> m_pair(const Geo& g, const PH& ph, R dm,
                                             const typename Vec2<R>::type* __restrict__ u,
                                             const Nbr& nb) {
  const int H = g.H;
  const R dk = geo_dk(g, R(0));
  Cx<R> ua = ld<R>(u, nb.q), ub = ld<R>(u, H + nb.q);
  // A row: (e^{i phi_A(t)} - dm) u_A(t-1)
  Cx<R> za = time_factor<MASS>(ph(nb.q), dm, false, nb.wrap_tm);
  Cx<R> ta = cfma(za, ld<R>(u, nb.tm), Cx<R>{-ua.re, -ua.im});
  Cx<R> oa = hopsum(ta, dk, ub, ld<R>(u, H + nb.im1), ld<R>(u, H + nb.jm1));
  // B row: -(e^{-i phi_B(t)} - dm) u_B(t+1)
  Cx<R> zb = time_factor<MASS>(ph(H + nb.q), dm, true, !nb.wrap_tp);
  Cx<R> tb = cfma(zb, ld<R>(u, H + nb.tp), ub);
  Cx<R> ob = hopsum(tb, dk, ua, ld<R>(u, nb.ip1), ld<R>(u, nb.jp1));
  return PairOut<R>{oa, ob};
}

}  // namespace hmc

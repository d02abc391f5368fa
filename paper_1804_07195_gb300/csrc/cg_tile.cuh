// CG on resident tiles: a whole solve of (M M^dagger + sigma) x = b (Section 3;
// the inner solver of Algorithm A.1) in one launch, every vector of the
// iteration kept on the chip. One group of thread blocks holds one system: all
// blocks of a cooperative launch (CL = false), or the blocks of one thread
// block cluster (CL = true; many clusters of one launch solve many systems).
//
// Tiles. A block owns all n cells of J rows and T time slices. p and
// u = M^dagger p of the tile live in shared memory, each of the four arrays
// p_A, p_B, u_A, u_B padded by the one row and the one slice of neighbouring
// tiles its stencil reads (Eq. ferm_op: the A rows of M^dagger read p_B at
// (i, j), (i-1, j), (i, j-1) and p_A at t+1; the B rows read p_A at (i, j),
// (i+1, j), (i, j+1) and p_B at t-1; M reads u the same way with the time hops
// reversed); the i-neighbours wrap inside the tile. A thread owns a column:
// CW neighbouring cells of one row over S time slices, whose r and x stay in
// its registers, and walks up in time, so that a time neighbour it has just
// read is carried instead of read again.
//
// Iteration:
//   P  x += alpha p (the previous iteration's), p = r + beta p, on the tile and
//      on the padding of p (from the neighbours' r at the padding's cells: the
//      same operation on the same numbers as in the tile that owns them);
//   U  u = M^dagger p (u_A kept with its sign changed, so that no own value is
//      negated in either stencil); the tile's edges of u handed to the neighbours;
//      <p, A p> = |u|^2 + sigma |p|^2 summed over the group;
//   M  r -= alpha (M u + sigma p); the tile's edges of r handed to the
//      neighbours; |r|^2 summed over the group.
// Padding slices beyond t = nt - 1 or before t = 0 hold the anti-periodic
// continuation (negated values), so the time hops carry no sign of their own.
//
// Between blocks of a cooperative launch edges go through global memory (r
// itself and U), read with L2-only loads. A sum is one arrival word on which
// every block adds (a reduction that returns nothing: the parity a block waits
// for is its own count of exchanges) and polls, then warp 0 gathers the
// blocks' partials while the other warps fetch the edges. Every wait is
// bounded: a block that gives up marks the launch, and all leave.
// Between blocks of a cluster edges and partials are stored straight into the
// other blocks' shared memory (st.async), each store reporting its bytes to a
// barrier word of the block it goes to; a block goes on when all bytes due to it
// have arrived. (us per iteration, with a cluster barrier, which waits for every
// block's stores and for every block, in brackets: 12x12x32 2.61 (2.89), 13x13x32 2.85
// (3.31), 18x18x32 3.19 (3.53), 24x24x48 4.27 (4.53).) These waits are bounded too.
//
// Every sum is formed in a fixed order that is the same in every block, so
// all blocks of a group hold the same scalars and leave together. FP32 sums
// are float-float pairs, FP64 sums doubles.
//
// What bounds an FP32 iteration of a cooperative launch (us, 2070 MHz; in
// brackets the design before it, which read r, x and phi from L2 row by row in
// both halves and published p as well):
//   6x6x16 6.4 (9.0)   12x12x32 6.8 (8.6)   36x36x64 5.7 (7.5)
//   51x51x64 7.1 (11.6)   72x72x64 7.9 (11.8)   90x90x64 9.9   102x102x64 11.3 (16.2)
// The two exchanges take about 2 us each (arrival and poll of one L2 word 1.4,
// the gather or the edges 0.5), whatever the lattice. The rest is, at
// 102x102x64, shared memory (4.3 us of wavefronts), instruction issue (4.1) and
// L2 (phi twice, edges), which the phases overlap only in part. x of the columns
// of four slices and more lives in tensor memory: read and written there by the
// lane that owns it, 8 columns a slice, instead of streamed through L2 every
// iteration (102x102x64 14.0 -> 12.0 us, 97x101x63 16.0 -> 14.9), and the registers
// it leaves free allow blocks of more threads with fewer slices each (80x80x64 9.85
// -> 8.7, 85x85x64 14.7 -> 11.2). Tried and not kept: every block polling every
// block's packet (one trip less, but the polls of 18,000 packet reads delay
// the writes: 8.5 to 10.7 us at 36x36x64); x held in registers at 102x102x64
// (7 slices a column, 384 threads: 14.6 us, too few warps; but 90x90x64, where 480
// threads with 4 slices hold x, takes 11.1 us against 12.8 with x in memory, and a
// cluster of 8 blocks 6.4 against 8.3 at 24x24x48); 3 slices a column
// (832 threads, spills: 14.0); instances for tiles without a ragged edge
// (13.9); one warp adding up all threads' values (14.7).
#pragma once

#include "kernels.h"
#include "operator.cuh"

namespace hmc {

constexpr int kTileMaxGroup = 160;  // blocks of a cooperative launch at most (partials: 5 per lane)
constexpr int kTileMaxCluster = 16;
constexpr int kTileMaxWarps = 32;

// One system on its tiles (J, T nominal: the last tile of a direction may be
// smaller). Pointers to the solve's vectors in the precision of the kernel.
struct TileSys {
  Geo g;
  int J, T, tiles_j, tiles_t;
  int nseg;      // columns are cut into nseg pieces of S slices
  int tab, rp;   // shared memory: the padding's table; (CL) the neighbours' r at the padding
  FastDiv fq;    // division by the columns of a row, n / CW
  const void* ph;  // FP32: phi as float, in [-pi, pi]; FP64: e^{i phi}
  void *x, *r, *U;
  uint2* gtab;   // the padding's table where shared memory has no room for it, tile after tile
  CGScal* sc;
};

// Exchanges of a cooperative launch, and the limit of their waits; a cluster's
// take the last two only.
struct GridSync {
  double* part;    // [2][kTileMaxGroup] partials, 8 bytes each: the exchanges alternate
  unsigned* word;  // arrivals: the top bit flips when every block has arrived
  int* err;        // a block gave up
  unsigned need;   // arrivals an exchange waits for; a cluster: sums it waits for beyond its own
  long long limit; // SM cycles
};

// ---------------------------------------------------------------------------
// CW neighbouring complex values as (re, im) of a lane type L: two cells are
// packed FP32 pairs, (re0, re1) and (im0, im1), so that every operation of the
// stencil but the shift to the i-neighbour is one packed instruction; each lane
// is rounded as the scalar instruction would round it.
template <typename R, int CW>
struct Lane;
template <>
struct Lane<float, 1> {
  using L = float;
  using V = float2;  // storage of (re, im)
  static __device__ __forceinline__ L set(float a) { return a; }
};
template <>
struct Lane<float, 2> {
  using L = unsigned long long;
  using V = ulonglong2;
  static __device__ __forceinline__ L set(float a) { return pk2(Cx<float>{a, a}); }
};
template <>
struct Lane<double, 1> {
  using L = double;
  using V = double2;
  static __device__ __forceinline__ L set(double a) { return a; }
};
__device__ __forceinline__ float lfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double lfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ unsigned long long lfma(unsigned long long a, unsigned long long b, unsigned long long c) {
  return fma_x2(a, b, c);
}
__device__ __forceinline__ float ladd(float a, float b) { return a + b; }
__device__ __forceinline__ unsigned long long ladd(unsigned long long a, unsigned long long b) { return add_x2(a, b); }
__device__ __forceinline__ float lneg(float a) { return -a; }
__device__ __forceinline__ double lneg(double a) { return dneg_if(a, true); }
__device__ __forceinline__ unsigned long long lneg(unsigned long long a) { return a ^ 0x8000000080000000ull; }
// own cells + their neighbours at i - 1 (w: the column to the left) or i + 1
__device__ __forceinline__ float add_left(float own, float w) { return own + w; }
__device__ __forceinline__ unsigned long long add_left(unsigned long long own, unsigned long long w) {
  const Cx<float> o = upk2(own), l = upk2(w);
  return pk2(Cx<float>{o.re + l.im, o.im + o.re});
}
__device__ __forceinline__ float add_right(float own, float w) { return own + w; }
__device__ __forceinline__ unsigned long long add_right(unsigned long long own, unsigned long long w) {
  const Cx<float> o = upk2(own), r = upk2(w);
  return pk2(Cx<float>{o.re + o.im, o.im + r.re});
}

// the same + v
template <typename L>
__device__ __forceinline__ L sum_left(L own, L w, L v) {
  return ladd(add_left(own, w), v);
}
template <typename L>
__device__ __forceinline__ L sum_right(L own, L w, L v) {
  return ladd(add_right(own, w), v);
}
template <>
__device__ __forceinline__ double sum_left(double own, double w, double v) {
  return sum3(own, w, v);
}
template <>
__device__ __forceinline__ double sum_right(double own, double w, double v) {
  return sum3(own, w, v);
}

template <typename L>
struct CV {
  L re, im;
};
__device__ __forceinline__ CV<float> unpack(float2 a) { return CV<float>{a.x, a.y}; }
__device__ __forceinline__ CV<unsigned long long> unpack(ulonglong2 a) { return CV<unsigned long long>{a.x, a.y}; }
__device__ __forceinline__ CV<double> unpack(double2 a) { return CV<double>{a.x, a.y}; }
__device__ __forceinline__ float2 pack(CV<float> a) { return make_float2(a.re, a.im); }
__device__ __forceinline__ ulonglong2 pack(CV<unsigned long long> a) { return make_ulonglong2(a.re, a.im); }
__device__ __forceinline__ double2 pack(CV<double> a) { return make_double2(a.re, a.im); }
// between the lanes and the vectors' own layout (re0, im0, re1, im1)
__device__ __forceinline__ float2 swizzle(float2 a) { return a; }
__device__ __forceinline__ double2 swizzle(double2 a) { return a; }
__device__ __forceinline__ ulonglong2 swizzle(ulonglong2 a) {
  const Cx<float> x = upk2(a.x), y = upk2(a.y);
  return make_ulonglong2(pk2(Cx<float>{x.re, y.re}), pk2(Cx<float>{x.im, y.im}));
}
// a x + y
template <typename L>
__device__ __forceinline__ CV<L> vaxpy(L a, CV<L> x, CV<L> y) {
  return CV<L>{lfma(a, x.re, y.re), lfma(a, x.im, y.im)};
}
template <typename L>
__device__ __forceinline__ CV<L> vneg_if(CV<L> x, bool neg) {
  return neg ? CV<L>{lneg(x.re), lneg(x.im)} : x;
}
// own + (f + i g) v, gm = -g
template <typename L>
__device__ __forceinline__ CV<L> hop_time(CV<L> own, L f, L g, L gm, CV<L> v) {
  return CV<L>{lfma(f, v.re, lfma(gm, v.im, own.re)), lfma(f, v.im, lfma(g, v.re, own.im))};
}
// t + d (b + left of b + w)  /  t + d (a + right of a + w)
template <typename L>
__device__ __forceinline__ CV<L> hops_left(CV<L> t, L d, CV<L> b, CV<L> left, CV<L> w) {
  return CV<L>{lfma(d, sum_left(b.re, left.re, w.re), t.re), lfma(d, sum_left(b.im, left.im, w.im), t.im)};
}
template <typename L>
__device__ __forceinline__ CV<L> hops_right(CV<L> t, L d, CV<L> a, CV<L> right, CV<L> w) {
  return CV<L>{lfma(d, sum_right(a.re, right.re, w.re), t.re), lfma(d, sum_right(a.im, right.im, w.im), t.im)};
}

// Running sum of |v|^2 of one thread.
template <typename L>
struct SqAcc {
  L s = L(0);
  __device__ __forceinline__ void add(CV<L> a) { s = lfma(a.re, a.re, lfma(a.im, a.im, s)); }
};
__device__ __forceinline__ float total(SqAcc<float> a) { return a.s; }
__device__ __forceinline__ double total(SqAcc<double> a) { return a.s; }
__device__ __forceinline__ float total(SqAcc<unsigned long long> a) {
  const Cx<float> t = upk2(a.s);
  return t.re + t.im;
}

// Phases of a column's cells at one slice: the raw load (issued a slice ahead)
// and dm - cos phi, sin phi, -sin phi made of it.
template <typename R, int CW>
struct PhLd;
template <>
struct PhLd<float, 1> {
  using raw = float;
  static __device__ __forceinline__ raw load(const void* ph, int k) { return __ldg((const float*)ph + k); }
  static __device__ __forceinline__ void get(raw f, float dm, float& c, float& s, float& sm) {
    float co;
    __sincosf(f, &s, &co);
    c = dm - co;
    sm = -s;
  }
};
template <>
struct PhLd<float, 2> {
  using raw = float2;
  static __device__ __forceinline__ raw load(const void* ph, int k) { return __ldg((const float2*)ph + k); }
  static __device__ __forceinline__ void get(raw f, unsigned long long dm, unsigned long long& c, unsigned long long& s,
                                             unsigned long long& sm) {
    float s0, c0, s1, c1;
    __sincosf(f.x, &s0, &c0);
    __sincosf(f.y, &s1, &c1);
    const unsigned long long m1 = pk2(Cx<float>{-1.f, -1.f});
    c = fma_x2(pk2(Cx<float>{c0, c1}), m1, dm);
    s = pk2(Cx<float>{s0, s1});
    sm = pk2(Cx<float>{-s0, -s1});
  }
};
template <>
struct PhLd<double, 1> {
  using raw = double2;
  static __device__ __forceinline__ raw load(const void* ph, int k) { return __ldg((const double2*)ph + k); }
  static __device__ __forceinline__ void get(raw f, double dm, double& c, double& s, double& sm) {
    c = dm - f.x;
    s = f.y;
    sm = -f.y;
  }
};

// Sums over the group.
template <typename R>
struct Red;
template <>
struct Red<float> {
  using T = float2;
  static __device__ __forceinline__ T zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ T make(float a) { return make_float2(a, 0.f); }
  // TwoSum of the high parts, the errors gathered in the low one without
  // renormalising: the chain from one step to the next is a single addition.
  static __device__ __forceinline__ T add(T a, T b) {
    const float s = a.x + b.x;
    const float v = s - a.x;
    return make_float2(s, ((a.x - (s - v)) + (b.x - v)) + (a.y + b.y));
  }
  static __device__ __forceinline__ T shfl(T a, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
  }
  static __device__ __forceinline__ float value(T a) { return a.x + a.y; }
};
template <>
struct Red<double> {
  using T = double;
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T make(double a) { return a; }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ T shfl(T a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
  static __device__ __forceinline__ double value(T a) { return a; }
};

// The scalars of a solve made of the sums: of type R, or (WIDE, FP32) with all bits of
// the sums, alpha and beta rounded once from these. Batches hold them wide, as the
// other batched kernels hold FP64 ones; solves of a single system have FP32 scalars, as
// in its other FP32 CG kernels (wide ones cost 0.1 us of 2.6 to 4.4 an iteration on
// clusters of odd n, and at 102x102x64 4 ms of a trajectory's 159).
template <typename R, bool WIDE>
struct Scalars {
  using S = R;
  static __device__ __forceinline__ S of64(double a) { return (R)a; }
  static __device__ __forceinline__ double to64(S a) { return (double)a; }
  static __device__ __forceinline__ S of(typename Red<R>::T a) { return Red<R>::value(a); }
  static __device__ __forceinline__ R value(S a) { return a; }
  static __device__ __forceinline__ bool le(S a, S b) { return a <= b; }
  static __device__ __forceinline__ int over(S) { return 0; }
  static __device__ __forceinline__ R ratio(S a, S b, int = 0) { return a / b; }
};
template <>
struct Scalars<float, true> {
  using S = float2;
  static __device__ __forceinline__ S of64(double a) {
    const float h = (float)a;
    return make_float2(h, (float)(a - (double)h));
  }
  static __device__ __forceinline__ double to64(S a) { return (double)a.x + (double)a.y; }
  static __device__ __forceinline__ S of(float2 a) { return a; }
  static __device__ __forceinline__ float value(S a) { return a.x + a.y; }
  static __device__ __forceinline__ bool le(S a, S b) { return (a.x - b.x) + (a.y - b.y) <= 0.f; }
  // about 1 / b (b > 0), or 0 outside the range of that
  static __device__ __forceinline__ float over(S b) {
    return b.x > 1e-30f && b.x < 1e30f ? __fdividef(1.f, b.x) : 0.f;
  }
  // a / b: the approximate quotient, off by 2^-22, and the exact rest over b; where rc
  // is 0 the quotient of the high parts
  static __device__ __forceinline__ float ratio(S a, S b, float rc) {
    if (rc == 0.f) return a.x / b.x;
    const float q = a.x * rc;
    return fmaf(fmaf(-q, b.x, a.x) + fmaf(-q, b.y, a.y), rc, q);
  }
  static __device__ __forceinline__ float ratio(S a, S b) { return ratio(a, b, over(b)); }
};
template <typename R>
__device__ __forceinline__ typename Red<R>::T warp_sum(typename Red<R>::T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = Red<R>::add(v, Red<R>::shfl(v, o));
  return v;
}

// ---------------------------------------------------------------------------
// Arrival word (CL = false).
// Relaxed: the __threadfence before it orders the block's writes already, and the
// release form fences once more (51x51x64: 7.8 us an iteration, relaxed 7.55).
__device__ __forceinline__ void red_add_relaxed(unsigned* p, unsigned x) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

// ---------------------------------------------------------------------------
// Tensor memory as a store of x: a lane's 32-bit columns are its own (warp w of
// the block reaches lanes 32 (w mod 4) ..; the warps w, w + 4, .. take different
// columns). Every instruction is for the whole warp.
__device__ __forceinline__ void tmem_alloc(unsigned* where, int columns) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n\t"
               "tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(where)), "r"(columns) : "memory");
}
__device__ __forceinline__ void tmem_free(unsigned at, int columns) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(at), "r"(columns) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 8 and 4 columns: a slice's cells A and B
__device__ __forceinline__ void tmem_ld(unsigned at, uint4& a, uint4& b) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "r"(at) : "memory");
}
__device__ __forceinline__ void tmem_st(unsigned at, uint4 a, uint4 b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(at), "r"(a.x),
               "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
}
__device__ __forceinline__ void tmem_ld(unsigned at, uint2& a, uint2& b) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(a.x), "=r"(a.y), "=r"(b.x), "=r"(b.y) : "r"(at) : "memory");
}
__device__ __forceinline__ void tmem_st(unsigned at, uint2 a, uint2 b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(a.x), "r"(a.y),
               "r"(b.x), "r"(b.y) : "memory");
}
// the bits of a column's value
__device__ __forceinline__ uint2 bits(float2 v) { return make_uint2(__float_as_uint(v.x), __float_as_uint(v.y)); }
__device__ __forceinline__ uint4 bits(ulonglong2 v) {
  return make_uint4((unsigned)v.x, (unsigned)(v.x >> 32), (unsigned)v.y, (unsigned)(v.y >> 32));
}
__device__ __forceinline__ uint4 bits(double2 v) {
  return make_uint4((unsigned)__double2loint(v.x), (unsigned)__double2hiint(v.x), (unsigned)__double2loint(v.y),
                    (unsigned)__double2hiint(v.y));
}
__device__ __forceinline__ void from_bits(uint2 b, float2& v) { v = make_float2(__uint_as_float(b.x), __uint_as_float(b.y)); }
__device__ __forceinline__ void from_bits(uint4 b, ulonglong2& v) {
  v = make_ulonglong2(b.x | (unsigned long long)b.y << 32, b.z | (unsigned long long)b.w << 32);
}
__device__ __forceinline__ void from_bits(uint4 b, double2& v) {
  v = make_double2(__hiloint2double((int)b.y, (int)b.x), __hiloint2double((int)b.w, (int)b.z));
}

// Warp 0: the sum of all blocks' partials, in every lane.
template <typename R>
__device__ __forceinline__ typename Red<R>::T gather(const double* part, int G) {
  using T = typename Red<R>::T;
  constexpr int L = kTileMaxGroup / 32;
  const int lane = threadIdx.x & 31;
  T w[L];
#pragma unroll
  for (int k = 0; k < L; ++k)
    w[k] = lane + 32 * k < G ? __ldcg((const T*)part + lane + 32 * k) : Red<R>::zero();
  T v = w[0];
#pragma unroll
  for (int k = 1; k < L; ++k) v = Red<R>::add(v, w[k]);
  return warp_sum<R>(v);
}

// ---------------------------------------------------------------------------
// Distributed shared memory (CL = true).
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned mapa(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Stores into another block that report their bytes to a barrier word there.
__device__ __forceinline__ void st_remote(unsigned addr, float2 v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr),
               "f"(v.x), "f"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_remote(unsigned addr, ulonglong2 v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(addr),
               "l"(v.x), "l"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void bar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0u;
}

// Bytes from one of the four padded arrays to the next: constant, so that it is
// an immediate of every access (over all SMs; clusters have their own).
constexpr int kTileStride = 52 * 1024;

template <typename R>
struct TileScal;
template <>
struct TileScal<float> {
  static __device__ __forceinline__ void load(const CGScal* s, float& dm, float& sigma) {
    dm = s->dm32;
    sigma = s->sigma32;
  }
};
template <>
struct TileScal<double> {
  static __device__ __forceinline__ void load(const CGScal* s, double& dm, double& sigma) {
    dm = s->dm;
    sigma = s->sigma;
  }
};

// ---------------------------------------------------------------------------
// The value of i, recomputed from here on: keeps the compiler from holding the
// addresses of every slice in registers from one phase to the next.
__device__ __forceinline__ int fresh(int i) {
  asm volatile("" : "+r"(i));
  return i;
}

// A kernel instance is named by its slices per column S, plus kXInMemory where x
// only passes through registers (the others hold r and x): kept in tensor memory,
// which nothing else here needs, or by a cluster's blocks, which may share an SM
// and could then wait for its columns on each other, in its own memory.
constexpr int kXInMemory = 100;
constexpr int tile_slices(int inst) { return inst % kXInMemory; }
// Largest block of an instance, from the registers it needs (r and x: 8 per slice
// for complex64 cells, 16 for pairs and for complex128; about 60 more, 45 for one
// complex64 cell) and those a thread can have: the warps are dealt to four
// partitions of 16,384 registers, so 12, 16, 20, 24 or 32 warps get 168, 128, 96,
// 80 or 64 registers a thread.
template <typename R, int CW, int INST>
constexpr int tile_max_threads() {
  constexpr bool mem = INST >= kXInMemory;
  constexpr int held = (int)sizeof(R) * CW * tile_slices(INST) * (mem ? 1 : 2);
  if (sizeof(R) == 8) return held <= 16 ? 640 : mem && held > 48 ? 384 : 512;
  if (CW == 2) return held <= 16 ? 768 : held <= 32 ? 640 : 512;
  return held <= 16 ? 1024 : held <= 32 ? 768 : 512;
}

// The solve of one system by the block `tile` of its group. sm: four padded
// arrays AS bytes apart, the table of the padding (8 bytes a column; GT: in global
// memory instead) and, for CL, the neighbours' r there. WIDE: the scalars (Scalars).
template <typename R, int CW, int INST, bool CL, int AS, bool GT = false, bool WIDE = false>
__device__ __forceinline__ void cg_tile_solve(const TileSys& ts, const GridSync& gs, int tile, char* sm) {
  using LN = Lane<R, CW>;
  using L = typename LN::L;
  using V = typename LN::V;
  using C = CV<L>;
  using RT = Red<R>;
  using T = typename RT::T;
  using PH = PhLd<R, CW>;
  constexpr int VB = (int)sizeof(V), S = tile_slices(INST);
  constexpr int PA = 0, PB = AS, UA = 2 * AS, UB = 3 * AS;
  const int TAB = ts.tab, RP = ts.rp;
  __shared__ R s_a, s_ap;
  __shared__ int s_stop, s_fail;
  // FP32: the warps' sums. FP64 (CL = false): every thread's value, added up by
  // one warp: the FP64 pipe takes 16 cycles for a warp's addition, so that five
  // shuffle steps in every warp cost more than 1400 cycles of a block of 18
  constexpr bool BYTHREAD = !CL && sizeof(R) == 8;
  __shared__ T s_red[CL ? 2 * kTileMaxCluster * kTileMaxWarps : BYTHREAD ? tile_max_threads<R, CW, INST>() : kTileMaxWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = (blockDim.x + 31) >> 5;
  const int m = ts.g.m, nt = ts.g.nt;
  const int nq = ts.g.n / CW, Vq = ts.g.V / CW, Hq = ts.g.H / CW;  // all indices in columns of CW cells
  const int J = ts.J, J1 = J + 1, TN = ts.T;
  const bool used = tile < ts.tiles_j * ts.tiles_t;
  const int bt = used ? tile / ts.tiles_j : 0, bj = used ? tile - bt * ts.tiles_j : 0;
  const int j0 = bj * J, t0 = bt * TN;
  const int Jt = used ? min(J, m - j0) : 0, Tt = used ? min(TN, nt - t0) : 0;
  // the arrays, each of (T + 1) (J + 1) rows of nq columns:
  //   p_A, u_B: rows 0..Jt (Jt: the row above) / -1..Jt-1, slices 0..Tt (Tt: the slice after)
  //   p_B, u_A: rows -1..Jt-1 / 0..Jt, slices -1..Tt-1
  const int NJ = J1 * nq;  // one slice
  const bool wlo = t0 == 0, whi = t0 + Tt == nt;
  const void* ph = ts.ph;
  V* const rg = (V*)ts.r;
  V* const xg = (V*)ts.x;
  V* const Ug = (V*)ts.U;
  auto lds = [&](int o) { return unpack(*(const V*)(sm + o)); };
  auto sts = [&](int o, C v) { *(V*)(sm + o) = pack(v); };

  // the thread's column: cells q of row jj, slices s0 .. s0 + S - 1 of the tile.
  // With o = ((tt (J + 1) + jj) nq + q) VB the cell's values lie at
  //   p_A(tt) = o, p_A(tt+1) = o + NJ, p_A(jj+1) = o + nq,
  //   p_B(tt) = o + NJ + nq, p_B(jj-1) = o + NJ, p_B(tt-1) = o + nq,
  //   u_A(tt) = o + NJ, u_A(tt-1) = o, u_A(jj+1) = o + NJ + nq,
  //   u_B(tt) = o + nq, u_B(jj-1) = o, u_B(tt+1) = o + NJ + nq
  // (NJ and nq times VB) of their arrays; the column to the left or right adds
  // dl or dr.
  const int row = (int)fdiv((uint32_t)tid, ts.fq), q = tid - row * nq;
  const int seg = row / J, jj = row - seg * J, s0 = seg * S;
  const int nrow = J * ts.nseg;
  const bool act = row < nrow && jj < Jt;
  const int ns = act ? min(S, Tt - s0) : 0;  // the thread's slices (<= 0: none)
  const int dl = ((q == 0 ? nq - 1 : q - 1) - q) * VB, dr = ((q == nq - 1 ? 0 : q + 1) - q) * VB;
  const int oNJ = NJ * VB, oq = nq * VB;
  const int o_first = ((s0 * J1 + jj) * nq + q) * VB;
  const int k_first = ((t0 + s0) * m + j0 + jj) * nq + q;  // lattice index of its first slice

  // Padding: lines l = 0 .. 2 T + 2 J - 1 of nq columns each (nominal sizes):
  // the row below, the row above, the slice before, the slice after. line():
  // where column qq of line l of p and of u belongs (array and index in it),
  // its lattice index, and whether the value there continues anti-periodically;
  // false: no line. The A or B part of the lattice swaps between p and u for
  // the last two kinds (p's is given).
  const int lines = used ? 2 * TN + 2 * J : 0;
  const int jdn = j0 == 0 ? m - 1 : j0 - 1, jup = j0 + Jt >= m ? 0 : j0 + Jt;
  const int tdn = wlo ? nt - 1 : t0 - 1, tup = whi ? 0 : t0 + Tt;
  auto line = [&](int l, int qq, int& kind, int& ip, int& iu, int& k) -> bool {
    if (l < TN) {
      kind = 0;  // p_B, u_B
      ip = (l + 1) * NJ + qq;
      iu = l * NJ + qq;
      k = Hq + ((t0 + l) * m + jdn) * nq + qq;
      return l < Tt;
    }
    l -= TN;
    if (l < TN) {
      kind = 1;  // p_A, u_A
      ip = (l * J1 + Jt) * nq + qq;
      iu = ip + NJ;
      k = ((t0 + l) * m + jup) * nq + qq;
      return l < Tt;
    }
    l -= TN;
    if (l < J) {
      kind = 2;  // p_B, u_A
      ip = (l + 1) * nq + qq;
      iu = l * nq + qq;
      k = Hq + (tdn * m + j0 + l) * nq + qq;
      return l < Jt;
    }
    l -= J;
    kind = 3;  // p_A, u_B
    ip = (Tt * J1 + l) * nq + qq;
    iu = ip + nq;
    k = (tup * m + j0 + l) * nq + qq;
    return l < Jt;
  };
  // The padding's columns, decoded once into a table: shared-memory offsets
  // over VB of p (low half of .x) and u (high half), lattice index of p with
  // the sign in the top bit, the step to u's lattice index in the next two.
  // CL = false: they belong to the warps after the first (which gathers the
  // partials meanwhile), or to the only warp.
  const int e_first = CL ? tid : nwarps > 1 ? tid - 32 : tid;
  const int e_step = CL ? (int)blockDim.x : nwarps > 1 ? (int)blockDim.x - 32 : 32;
  const int e_end = e_first < 0 ? e_first : lines * nq;
  uint2* const tab = GT ? ts.gtab + (size_t)tile * (2 * (TN + J) * nq) : (uint2*)(sm + TAB);
  for (int e = e_first; e < e_end; e += e_step) {
    const int l = (int)fdiv((uint32_t)e, ts.fq);
    int kind, ip, iu, k;
    uint2 d = make_uint2(0xffffffffu, 0u);  // no column
    if (line(l, e - l * nq, kind, ip, iu, k)) {
      const bool neg = (kind == 2 && wlo) || (kind == 3 && whi);
      const unsigned a = ((kind == 0 || kind == 2 ? PB : PA) / VB) + ip, b = ((kind == 0 || kind == 3 ? UB : UA) / VB) + iu;
      d = make_uint2(a | b << 16, (unsigned)k | (neg ? 0x80000000u : 0u) | (kind == 2 ? 1u : kind == 3 ? 2u : 0u) << 29);
    }
    tab[e] = d;
  }
  auto for_padding = [&](auto&& f) {
    for (int e = e_first; e < e_end; e += e_step) {
      const uint2 d = tab[e];
      if (d.x == 0xffffffffu) continue;
      const unsigned st = (d.y >> 29) & 3u;
      const int kp = (int)(d.y & 0x1fffffffu);
      f(e, (int)(d.x & 0xffffu) * VB, (int)(d.x >> 16) * VB, kp, kp + (st == 1u ? -Hq : st == 2u ? Hq : 0),
        (d.y >> 31) != 0u);
    }
  };
  // The padding of u from the neighbours' edges in src (u, or r if `of_r`), read
  // from L2. A thread has up to four columns, and a trip to L2 for each takes 0.6 us:
  // 16-byte columns go by cp.async, all in flight and through no register; 8-byte
  // ones (whose cp.async may hit a stale L1 line) FB at a time in registers. (102x102x64
  // 12.0 -> 11.5 us an iteration, 51x51x64 7.55 -> 7.15, 75x75x64 11.8 -> 10.5; FP64
  // 51x51x64 31.0 -> 28.5.)
  auto fetch_padding = [&](const V* src, bool of_r) {
    auto from = [&](unsigned y) {
      const unsigned st = of_r ? 0u : (y >> 29) & 3u;
      return src + (int)(y & 0x1fffffffu) + (st == 1u ? -Hq : st == 2u ? Hq : 0);
    };
    if constexpr (VB == 16) {
      const unsigned base = (unsigned)__cvta_generic_to_shared(sm);
      for (int e = e_first; e < e_end; e += e_step) {
        const uint2 d = tab[e];
        if (d.x != 0xffffffffu)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + (d.x >> 16) * VB), "l"(from(d.y)) : "memory");
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      if (wlo || whi)
        for (int e = e_first; e < e_end; e += e_step) {
          const uint2 d = tab[e];
          if (d.x != 0xffffffffu && (d.y >> 31) != 0u) {
            const int ou = (int)(d.x >> 16) * VB;
            sts(ou, vneg_if(lds(ou), true));
          }
        }
    } else {
      constexpr int FB = INST == 4 ? 2 : 3;  // (69x69x64, four slices: 10.05 us with 2, 10.9 with 3)
      for (int e = e_first; e < e_end; e += FB * e_step) {
        uint2 d[FB];
        V v[FB];
#pragma unroll
        for (int i = 0; i < FB; ++i) {
          d[i] = e + i * e_step < e_end ? tab[e + i * e_step] : make_uint2(0xffffffffu, 0u);
          if (d[i].x != 0xffffffffu) v[i] = __ldcg(from(d[i].y));
        }
#pragma unroll
        for (int i = 0; i < FB; ++i)
          if (d[i].x != 0xffffffffu) sts((int)(d[i].x >> 16) * VB, vneg_if(unpack(v[i]), (d[i].y >> 31) != 0u));
      }
    }
  };
  unsigned rem_dn = 0, rem_up = 0, rem_bf = 0, rem_af = 0;  // CL: the neighbours' shared memory
  int JtD = 0, TtP = 0;  // CL: rows of the tile below, slices of the tile before
  if constexpr (CL) {
    const int bd = bj == 0 ? ts.tiles_j - 1 : bj - 1, bu = bj == ts.tiles_j - 1 ? 0 : bj + 1;
    const int tb = bt == 0 ? ts.tiles_t - 1 : bt - 1, ta = bt == ts.tiles_t - 1 ? 0 : bt + 1;
    const unsigned sb = (unsigned)__cvta_generic_to_shared(sm);
    rem_dn = mapa(sb, bt * ts.tiles_j + bd);
    rem_up = mapa(sb, bt * ts.tiles_j + bu);
    rem_bf = mapa(sb, tb * ts.tiles_j + bj);
    rem_af = mapa(sb, ta * ts.tiles_j + bj);
    JtD = min(J, m - bd * J);
    TtP = min(TN, nt - tb * TN);
  }

  // |r|^2 (of iteration i in s_rr[i & 1]), <p, A p> and the threshold are kept in shared
  // memory, as registers are short: by thread 0, read behind a barrier (CL) or by
  // thread 0 alone.
  using SC = Scalars<R, WIDE>;
  R dm, sigma;
  TileScal<R>::load(ts.sc, dm, sigma);
  __shared__ typename SC::S s_rr[2], s_pap, s_thresh;
  typename SC::S rr = SC::of64(ts.sc->rr), thresh = SC::of64(ts.sc->thresh);
  const L ldm = LN::set(dm), ldk = LN::set(geo_dk(ts.g, R(0))), lndk = LN::set(-geo_dk(ts.g, R(0)));
  int iter = ts.sc->iter, done = ts.sc->done;
  const int maxit = ts.sc->maxit;
  R alpha = R(0), beta = R(0);
  bool first = true;
  if (tid == 0) {
    s_rr[iter & 1] = rr;
    s_pap = SC::of64(0.0);
    s_thresh = thresh;
  }
  // exchanges so far; CL = false: its parity is the arrival word's top bit
  unsigned ep = CL ? 0u : *(const volatile unsigned*)gs.word >> 31;

  // r and x of the thread's cells (A, B). With many slices per column x is kept
  // elsewhere in the lanes' layout and passes through registers in P, two slices
  // in flight: in tensor memory (CL = false: one block an SM), or in its own memory.
  constexpr bool XREG = INST < kXInMemory, XTM = !XREG && !CL;
  constexpr int XC = VB / 2;  // columns of a slice's cells A and B
  using B = decltype(bits(V{}));
  __shared__ unsigned s_tmem;
  static_assert(!XTM || XC * S * ((tile_max_threads<R, CW, INST>() / 32 + 3) / 4) <= 512, "tensor memory of an SM");
  const int xcols = XC * S * ((nwarps + 3) / 4);
  const int xalloc = xcols <= 32 ? 32 : xcols <= 64 ? 64 : xcols <= 128 ? 128 : xcols <= 256 ? 256 : 512;
  unsigned xt = 0;
  if constexpr (XTM) {
    if (warp == 0) tmem_alloc(&s_tmem, xalloc);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    xt = s_tmem + ((unsigned)(warp & 3) << 21) + (unsigned)(warp >> 2) * (XC * S);
  }
  C ra[S], rb[S];
  C xa[XREG ? S : 2], xb[XREG ? S : 2];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    B ba{}, bb{};
    if (s < ns) {
      const int k = k_first + s * Vq;
      ra[s] = unpack(swizzle(rg[k]));
      rb[s] = unpack(swizzle(rg[Hq + k]));
      if (XREG) {
        xa[XREG ? s : 0] = unpack(swizzle(xg[k]));
        xb[XREG ? s : 0] = unpack(swizzle(xg[Hq + k]));
      } else if (XTM) {
        ba = bits(swizzle(xg[k]));
        bb = bits(swizzle(xg[Hq + k]));
      } else {
        xg[k] = swizzle(xg[k]);
        xg[Hq + k] = swizzle(xg[Hq + k]);
      }
    }
    if constexpr (XTM) {
      __syncwarp();
      tmem_st(xt + s * XC, ba, bb);
    }
  }
  // x += f p (p of the last iteration) and, if asked, p = r + fb p, slice by slice
  auto x_and_p = [&](R f, R fb, bool newp) {
    const L lf = LN::set(f), lb = LN::set(fb);
    int o = fresh(o_first), k = fresh(k_first);
    auto slice = [&](int s, C& x0, C& x1) {
      const C pa = lds(PA + o), pb = lds(PB + o + oNJ + oq);
      x0 = vaxpy(lf, pa, x0);
      x1 = vaxpy(lf, pb, x1);
      if (newp) {
        sts(PA + o, vaxpy(lb, pa, ra[s]));
        sts(PB + o + oNJ + oq, vaxpy(lb, pb, rb[s]));
      }
    };
    if constexpr (XTM) {
      static_assert(S % 2 == 0, "slices go in pairs");
      tmem_wait_st();  // the last iteration's
#pragma unroll
      for (int s = 0; s < S; s += 2) {
        B b0[2], b1[2];
        __syncwarp();
        tmem_ld(xt + s * XC, b0[0], b1[0]);
        tmem_ld(xt + (s + 1) * XC, b0[1], b1[1]);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 2; ++e, o += oNJ)
          if (s + e < ns) {
            V v0, v1;
            from_bits(b0[e], v0);
            from_bits(b1[e], v1);
            C x0 = unpack(v0), x1 = unpack(v1);
            slice(s + e, x0, x1);
            b0[e] = bits(pack(x0));
            b1[e] = bits(pack(x1));
          }
        __syncwarp();
        tmem_st(xt + s * XC, b0[0], b1[0]);
        tmem_st(xt + (s + 1) * XC, b0[1], b1[1]);
      }
      return;
    }
    if (!XREG) {
#pragma unroll
      for (int s = 0; s < 2; ++s)
        if (s < ns) {
          xa[s] = unpack(xg[k + s * Vq]);
          xb[s] = unpack(xg[Hq + k + s * Vq]);
        }
    }
#pragma unroll
    for (int s = 0; s < S; ++s, o += oNJ, k += Vq)
      if (s < ns) {
        const int e = XREG ? s : (s & 1);
        slice(s, xa[e], xb[e]);
        if (!XREG) {
          xg[k] = pack(xa[e]);
          xg[Hq + k] = pack(xb[e]);
          if (s + 2 < S && s + 2 < ns) {
            xa[e] = unpack(xg[k + 2 * Vq]);
            xb[e] = unpack(xg[Hq + k + 2 * Vq]);
          }
        }
      }
  };
  // p = 0 before the first iteration (beta = 0 there), on the tile and its padding
  for (int e = tid; e < (TN + 1) * NJ; e += blockDim.x) {
    sts(PA + e * VB, C{L(0), L(0)});
    sts(PB + e * VB, C{L(0), L(0)});
  }
  if (!CL && tid == 0) s_fail = 0;
  // CL: a barrier word per parity of the exchanges. One use of it completes when the
  // block has armed it (thread 0) and every byte due has arrived: its padding's
  // columns and the sums of all warps of the cluster. Two words are enough: a block
  // sends for exchange e + 2 after it has all sums of e + 1, and ours of e + 1 left
  // after we had all of e. For the same reason nothing is overwritten that is still
  // to be read.
  __shared__ unsigned long long s_bar[2];
  const unsigned bar0 = (unsigned)__cvta_generic_to_shared(s_bar);
  const unsigned bar_off = bar0 - (unsigned)__cvta_generic_to_shared(sm);  // in any block of the cluster
  unsigned due = 0;
  if constexpr (CL) {
    due = (cluster_size() * nwarps + gs.need) * (unsigned)sizeof(T) + (unsigned)((2 * Tt + 2 * Jt) * nq * VB);
    if (tid == 0) {
      bar_init(bar0);
      bar_init(bar0 + 8);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      bar_expect(bar0, due);
      bar_expect(bar0 + 8, due);
    }
    for_padding([&](int e, int, int, int kp, int, bool neg) {
      sts(RP + e * VB, vneg_if(unpack(swizzle(rg[kp])), neg));
    });
    cluster_barrier();
  }

  // Sum over the group. CL: in every thread, which runs `edges` while the sums are on
  // their way. Otherwise in warp 0; the other warps run `edges` meanwhile.
  auto exchange = [&](R loc, auto&& edges, T* out) -> bool {
    ++ep;
    if constexpr (CL) {
      const T wsum = warp_sum<R>(RT::make(loc));
      const unsigned cs = cluster_size(), me = cluster_rank();
      T* slots = s_red + (ep & 1u) * kTileMaxCluster * kTileMaxWarps;
      const unsigned bar = bar0 + 8 * ((ep - 1) & 1u), parity = ((ep - 1) >> 1) & 1u;
      if (lane < (int)cs) {
        const unsigned a = (unsigned)__cvta_generic_to_shared(slots + me * nwarps + warp);
        st_remote(mapa(a, lane), wsum, mapa(bar, lane));
      }
      edges();
      const long long tw = clock64();
      bool late = false;
      while (!bar_try(bar, parity) && !(late = clock64() - tw > gs.limit)) {
      }
      // the block's own writes to shared memory, and one answer for all its threads
      if (__syncthreads_or(late)) return false;
      if (tid == 0) bar_expect(bar, due);  // for the exchange after next
      const int cnt = (int)cs * nwarps;
      T v = RT::zero();
      for (int k = lane; k < cnt; k += 32) v = RT::add(v, slots[k]);
      *out = warp_sum<R>(v);
      return true;
    } else {
      T* part = (T*)(gs.part + (ep & 1u) * kTileMaxGroup);
      if constexpr (BYTHREAD) {
        s_red[tid] = RT::make(loc);
      } else {
        const T wsum = warp_sum<R>(RT::make(loc));
        if (lane == 0) s_red[warp] = wsum;
      }
      __syncthreads();
      if (warp == 0) {
        T v;
        if constexpr (BYTHREAD) {
          T w[4] = {RT::zero(), RT::zero(), RT::zero(), RT::zero()};
          for (int k = 0; k < nwarps; k += 4)
#pragma unroll
            for (int h = 0; h < 4; ++h)
              if (k + h < nwarps) w[h] = RT::add(w[h], s_red[(k + h) * 32 + lane]);
          v = warp_sum<R>(RT::add(RT::add(w[0], w[1]), RT::add(w[2], w[3])));
        } else {
          v = warp_sum<R>(lane < nwarps ? s_red[lane] : RT::zero());
        }
        if (lane == 0) {
          part[tile] = v;
          __threadfence();  // the block's edges, ordered before this thread by the barrier above
          red_add_relaxed(gs.word, tile == 0 ? 0x80000000u - (gs.need - 1u) : 1u);
          const unsigned want = (ep & 1u) << 31;
          const long long tw = clock64();
          unsigned spins = 0;
          while ((ld_acquire_gpu(gs.word) & 0x80000000u) != want) {
            if ((++spins & 31u) == 0u && (*(volatile int*)gs.err || clock64() - tw > gs.limit)) {
              atomicExch(gs.err, 1);
              s_fail = 1;
              break;
            }
          }
        }
      }
      __syncthreads();
      if (s_fail) return false;
      if (warp == 0) *out = gather<R>((const double*)part, gridDim.x);
      if (warp != 0 || nwarps == 1) edges();
      return true;
    }
  };

  for (;;) {
    if (CL || tid == 0) {
      if (!done) {
        if (!isfinite(SC::value(rr)))
          done = CG_BREAKDOWN;
        else if (SC::le(rr, thresh))
          done = CG_CONVERGED;
        else if (iter >= maxit)
          done = CG_MAXIT;
      }
    }
    R fb = beta, fap = alpha;
    int stop = done;
    if constexpr (!CL) {
      if (tid == 0) {
        s_a = beta;
        s_ap = alpha;
        s_stop = done;
      }
      __syncthreads();
      fb = s_a;
      fap = s_ap;
      stop = s_fail ? CG_TIMEOUT : s_stop;
    }
    if (stop) {
      done = stop;
      if (stop != CG_TIMEOUT && fap != R(0)) x_and_p(fap, R(0), false);  // the last iteration's x update
      break;
    }
    // ---- P: the padding (r of the neighbours at hand: rp, or left in place of
    // the padding of u by the edges below), then the tile
    {
      const L lb = LN::set(fb);
      for_padding([&](int e, int op, int ou, int kp, int, bool neg) {
        const C v = CL ? lds(RP + e * VB) : first ? vneg_if(unpack(swizzle(__ldcg(rg + kp))), neg) : lds(ou);
        sts(op, vaxpy(lb, lds(op), v));
      });
    }
    x_and_p(fap, fb, true);
    // phases of the first slice: A at t + 1, B at t - 1
    typename PH::raw fa{}, fbt{};
    if (ns > 0) {
      const int t = t0 + s0;
      fa = PH::load(ph, t + 1 == nt ? k_first + Vq - Hq : k_first + Vq);
      fbt = PH::load(ph, Hq + (t == 0 ? k_first - Vq + Hq : k_first - Vq));
    }
    __syncthreads();
    // ---- U
    SqAcc<L> acc, accp;
    unsigned bar_next = bar_off + 8 * (ep & 1u);  // of the exchange ahead
    if (ns > 0) {
      int o = fresh(o_first), k = fresh(k_first);
      C pa = lds(PA + o), pbm = lds(PB + o + oq);
#pragma unroll
      for (int s = 0; s < S; ++s, o += oNJ, k += Vq)
        if (s < ns) {
          L f0, g0, h0, f1, g1, h1;
          PH::get(fa, ldm, f0, g0, h0);
          PH::get(fbt, ldm, f1, g1, h1);
          if (s + 1 < S && s + 1 < ns) {
            fa = PH::load(ph, t0 + s0 + s + 2 == nt ? k + 2 * Vq - Hq : k + 2 * Vq);
            fbt = PH::load(ph, Hq + k);
          }
          const C pan = lds(PA + o + oNJ), pb = lds(PB + o + oNJ + oq);
          const C va = hops_left(hop_time(pa, f0, g0, h0, pan), ldk, pb, lds(PB + o + oNJ + oq + dl), lds(PB + o + oNJ));
          const C vb = hops_right(hop_time(pb, f1, h1, g1, pbm), lndk, pa, lds(PA + o + dr), lds(PA + o + oq));
          sts(UA + o + oNJ, va);
          sts(UB + o + oq, vb);
          acc.add(va);
          acc.add(vb);
          if (sigma != R(0)) {
            accp.add(pa);
            accp.add(pb);
          }
          // edges the neighbours' M reads: u_A of the bottom row and the last
          // slice, u_B of the top row and the first slice
          const int tt = s0 + s;
          if constexpr (CL) {
            if (jj == 0) st_remote(rem_dn + UA + (((tt + 1) * J1 + JtD) * nq + q) * VB, pack(va), rem_dn + bar_next);
            if (tt == Tt - 1) st_remote(rem_af + UA + (jj * nq + q) * VB, pack(vneg_if(va, whi)), rem_af + bar_next);
            if (jj == Jt - 1) st_remote(rem_up + UB + (tt * NJ + q) * VB, pack(vb), rem_up + bar_next);
            if (tt == 0) st_remote(rem_bf + UB + ((TtP * J1 + jj + 1) * nq + q) * VB, pack(vneg_if(vb, wlo)), rem_bf + bar_next);
          } else {
            if (jj == 0 || tt == Tt - 1) Ug[k] = pack(va);
            if (jj == Jt - 1 || tt == 0) Ug[Hq + k] = pack(vb);
          }
          pa = pan;
          pbm = pb;
        }
    }
    T tot;
    bool ok = exchange(total(acc) + (sigma != R(0) ? sigma * total(accp) : R(0)), [&] {
      if constexpr (CL)
        rr = s_rr[iter & 1];
      else
        fetch_padding(Ug, false);
    }, &tot);
    // phases of the first slice of M
    if (ns > 0) {
      fa = PH::load(ph, k_first);
      fbt = PH::load(ph, Hq + k_first);
    }
    if (CL || tid == 0) {
      if constexpr (!CL) rr = s_rr[iter & 1];
      const typename SC::S pap = ok ? SC::of(tot) : SC::of64(0.0);
      const bool bad = !(SC::value(pap) > R(0)) || !isfinite(SC::value(pap));
      alpha = bad ? R(0) : SC::ratio(rr, pap);
      if (tid == 0) s_pap = pap;
      if (bad) done = ok ? CG_BREAKDOWN : CG_TIMEOUT;
    }
    R fal = alpha;
    if constexpr (!CL) {
      if (tid == 0) {
        s_a = alpha;
        s_stop = done;
      }
      __syncthreads();
      fal = s_a;
      done = s_fail ? CG_TIMEOUT : s_stop;
    }
    if (done) break;
    // ---- M
    SqAcc<L> accr;
    bar_next = bar_off + 8 * (ep & 1u);
    if (ns > 0) {
      const L lal = LN::set(-fal), lsig = LN::set(sigma);
      int o = fresh(o_first), k = fresh(k_first);
      C uam = lds(UA + o), ub = lds(UB + o + oq);
#pragma unroll
      for (int s = 0; s < S; ++s, o += oNJ, k += Vq)
        if (s < ns) {
          L f0, g0, h0, f1, g1, h1;
          PH::get(fa, ldm, f0, g0, h0);
          PH::get(fbt, ldm, f1, g1, h1);
          if (s + 1 < S && s + 1 < ns) {
            fa = PH::load(ph, k + Vq);
            fbt = PH::load(ph, Hq + k + Vq);
          }
          const C ua = lds(UA + o + oNJ), ubn = lds(UB + o + oNJ + oq);
          C va = hops_left(hop_time(ua, f0, h0, g0, uam), lndk, ub, lds(UB + o + oq + dl), lds(UB + o));
          C vb = hops_right(hop_time(ub, f1, g1, h1, ubn), ldk, ua, lds(UA + o + oNJ + dr), lds(UA + o + oNJ + oq));
          if (sigma != R(0)) {
            va = vaxpy(lsig, lds(PA + o), va);
            vb = vaxpy(lsig, lds(PB + o + oNJ + oq), vb);
          }
          ra[s] = vaxpy(lal, va, ra[s]);
          rb[s] = vaxpy(lal, vb, rb[s]);
          accr.add(ra[s]);
          accr.add(rb[s]);
          // edges the neighbours' padding of p needs: r_B of the top row and the
          // last slice, r_A of the bottom row and the first slice
          const int tt = s0 + s;
          if constexpr (CL) {
            if (jj == Jt - 1) st_remote(rem_up + RP + (tt * nq + q) * VB, pack(rb[s]), rem_up + bar_next);
            if (jj == 0) st_remote(rem_dn + RP + ((TN + tt) * nq + q) * VB, pack(ra[s]), rem_dn + bar_next);
            if (tt == Tt - 1) st_remote(rem_af + RP + ((2 * TN + jj) * nq + q) * VB, pack(vneg_if(rb[s], whi)), rem_af + bar_next);
            if (tt == 0) st_remote(rem_bf + RP + ((2 * TN + J + jj) * nq + q) * VB, pack(vneg_if(ra[s], wlo)), rem_bf + bar_next);
          } else {
            if (jj == 0 || tt == 0) rg[k] = pack(ra[s]);
            if (jj == Jt - 1 || tt == Tt - 1) rg[Hq + k] = pack(rb[s]);
          }
          uam = ua;
          ub = ubn;
        }
    }
    // the neighbours' r waits in the padding of u, which nothing reads until the
    // next exchange has refilled it (the block's barrier in `exchange` orders
    // the reads of u above before these writes)
    decltype(SC::over(rr)) over{};
    ok = exchange(total(accr), [&] {
      if constexpr (CL) {
        rr = s_rr[iter & 1];
        thresh = s_thresh;
        over = SC::over(rr);
      } else {
        fetch_padding(rg, true);
      }
    }, &tot);
    if (CL || tid == 0) {
      if constexpr (!CL) {
        rr = s_rr[iter & 1];
        thresh = s_thresh;
        over = SC::over(rr);
      }
      const typename SC::S now = ok ? SC::of(tot) : rr;
      if (!ok) done = CG_TIMEOUT;
      beta = SC::ratio(now, rr, over);
      rr = now;
      if (tid == 0) s_rr[(iter + 1) & 1] = rr;
    }
    ++iter;
    first = false;
  }
  if constexpr (XTM) tmem_wait_st();
#pragma unroll
  for (int s = 0; s < S; ++s) {
    B ba{}, bb{};
    if constexpr (XTM) {
      __syncwarp();
      tmem_ld(xt + s * XC, ba, bb);
      tmem_wait_ld();
    }
    if (s < ns) {
      const int k = k_first + s * Vq;
      if (XREG) {
        xg[k] = swizzle(pack(xa[XREG ? s : 0]));
        xg[Hq + k] = swizzle(pack(xb[XREG ? s : 0]));
      } else if (XTM) {
        V v0, v1;
        from_bits(ba, v0);
        from_bits(bb, v1);
        xg[k] = swizzle(v0);
        xg[Hq + k] = swizzle(v1);
      } else {
        xg[k] = swizzle(xg[k]);
        xg[Hq + k] = swizzle(xg[Hq + k]);
      }
    }
  }
  if constexpr (XTM) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0) tmem_free(s_tmem, xalloc);
  }
  if constexpr (CL) {
    // no block leaves while it may still be written to: one that had its bytes has
    // none on their way, one that gave up waits for all blocks' last stores to land
    // (less than 1 us behind the barrier)
    cluster_barrier();
    if (done == CG_TIMEOUT)
      for (const long long tw = clock64(); clock64() - tw < 50000LL;) {
      }
  }
  if (tid != 0) return;
  CGScal* sc = ts.sc;
  if (tile == 0) {
    sc->rr = sc->rr_cur = SC::to64(s_rr[iter & 1]);
    sc->rr32 = sc->rr_cur32 = (float)sc->rr;
    sc->pAp = SC::to64(s_pap);
    sc->alpha = alpha;
    sc->beta = beta;
    sc->iter = iter;
    sc->first = 0;
  }
  // the largest code of all blocks: one that gave up counts, also where the others
  // had what they waited for and went on to the end
  if (tile == 0 || done == CG_TIMEOUT) atomicMax(&sc->done, done ? done : CG_MAXIT);
}

}  // namespace hmc

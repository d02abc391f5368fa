// Launch helpers shared by the kernel translation units: the phase tables of
// the context's current field, and launches with programmatic dependent launch.
#pragma once

#include <type_traits>

#include "kernels.h"
#include "operator.cuh"
#include "phase.cuh"

namespace hmc {

// Phases of the context's field: the FP64 table e^{i phi}, or phi as float.
template <typename R>
inline Phase<R> phase_of(hmc_ctx* c);
template <>
inline Phase<double> phase_of<double>(hmc_ctx* c) {
  return Phase<double>{(const double2*)c->ws[WS_E]};
}
template <>
inline Phase<float> phase_of<float>(hmc_ctx* c) {
  return Phase<float>{(const float*)c->ws[WS_PHI32]};
}

// e^{i phi_k} straight from the field, for one application: the numbers of the
// tables without the pass that builds them. E (may be NULL) keeps what was formed.
template <typename R>
struct FieldPhase;
template <>
struct FieldPhase<double> {
  const double* __restrict__ phi;
  PhaseTable tab;
  double2* E;
  __device__ __forceinline__ Cx<double> operator()(int k) const {
    const double2 e = phase_of_field(tab, phi[k]);
    if (E != nullptr) E[k] = e;
    return Cx<double>{e.x, e.y};
  }
};
template <>
struct FieldPhase<float> {
  const double* __restrict__ phi;
  __device__ __forceinline__ Cx<float> operator()(int k) const {
    const float x = field_to_f32(phi[k]);
    return Phase<float>{&x}(0);
  }
};
template <typename R>
inline FieldPhase<R> field_phase(hmc_ctx* c, const double* phi, bool keep);
template <>
inline FieldPhase<double> field_phase<double>(hmc_ctx* c, const double* phi, bool keep) {
  return FieldPhase<double>{phi, PhaseTable{c->phase_tab}, keep ? (double2*)c->ws[WS_E] : nullptr};
}
template <>
inline FieldPhase<float> field_phase<float>(hmc_ctx*, const double* phi, bool) {
  return FieldPhase<float>{phi};
}

// Launch with the programmatic-serialization attribute (see pdl_wait): the blocks
// of a kernel are placed when those of the kernel before it have ended, without
// waiting for its memory to be flushed, which hides most of the launch (phases and
// M^dagger at 51x51x64 22.5 -> 18 us; a trajectory at 12x12x32, some 2,300 short
// kernels, 57.4 -> 51.5 ms). The kernels of the FP64 path don't trigger earlier:
// placed among running blocks, those of a grid below one wave crowd on some SMs
// (M^dagger at 51x51x64 7.4 us, without 6.45; the dots of 102x102x64 102 -> 150).
// Ordinary launches are those that have no kernel before them in a graph: the first
// of a capture, and any while somebody else captures the stream.
template <typename... KA, typename... A>
inline void launch_pdl_smem(hmc_ctx* c, void (*k)(KA...), dim3 grid, int threads, int smem, cudaStream_t s,
                            A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool pdl = c->capturing ? c->pdl_armed
                                : cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone;
  cfg.attrs = pdl ? attr : nullptr;
  cfg.numAttrs = pdl ? 1 : 0;
  (void)cudaLaunchKernelEx(&cfg, k, ((KA)args)...);  // errors surface through cudaGetLastError
  if (c->capturing) c->pdl_armed = true;
}
template <typename... KA, typename... A>
inline void launch_pdl(hmc_ctx* c, void (*k)(KA...), dim3 grid, int threads, cudaStream_t s, A... args) {
  launch_pdl_smem(c, k, grid, threads, 0, s, args...);
}

template <int J>
using IC = std::integral_constant<int, J>;

}  // namespace hmc

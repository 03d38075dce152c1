// Per-channel decay: what the chunk scan's operands are made of, for the two kernels that write them (kda_scan_prep_kernel, a launch of its
// own, and the groups of kda_scan_kernel beside the scans): one copy of the arithmetic, so that both give the same bits.
// A thread has eight neighbouring features.  G_ref is the chunk's middle row, G_last its last.
#pragma once
#include "tc_device.cuh"

namespace tri_inv {
namespace {

constexpr float kDecayLog2e = 1.4426950408889634f;

struct DecayRefs { float ref[8], last[8]; };   // times log2 e

__device__ __forceinline__ void load_decay_row(float (&x)[8], const float* row) {
#pragma unroll
  for (int q = 0; q < 8; q += 4) {
    const float4 y = *reinterpret_cast<const float4*>(row + q);
    x[q] = y.x * kDecayLog2e; x[q + 1] = y.y * kDecayLog2e; x[q + 2] = y.z * kDecayLog2e; x[q + 3] = y.w * kDecayLog2e;
  }
}
__device__ __forceinline__ DecayRefs load_decay_refs(const float* ref_row, const float* last_row) {
  DecayRefs r;
  load_decay_row(r.ref, ref_row);
  load_decay_row(r.last, last_row);
  return r;
}

// exp(G_last), exp(G_ref), exp(G_last - G_ref)
__device__ __forceinline__ void store_decay_vectors(float* EL, float* ER, float* EX, const DecayRefs& r) {
#pragma unroll
  for (int q = 0; q < 8; q += 4) {
    *reinterpret_cast<float4*>(EL + q) = make_float4(ex2_approx(r.last[q]), ex2_approx(r.last[q + 1]), ex2_approx(r.last[q + 2]), ex2_approx(r.last[q + 3]));
    *reinterpret_cast<float4*>(ER + q) = make_float4(ex2_approx(r.ref[q]), ex2_approx(r.ref[q + 1]), ex2_approx(r.ref[q + 2]), ex2_approx(r.ref[q + 3]));
    *reinterpret_cast<float4*>(EX + q) = make_float4(ex2_approx(r.last[q] - r.ref[q]), ex2_approx(r.last[q + 1] - r.ref[q + 1]),
                                                     ex2_approx(r.last[q + 2] - r.ref[q + 2]), ex2_approx(r.last[q + 3] - r.ref[q + 3]));
  }
}

// Q+ = Q exp(G - G_ref), K- = K exp(G_ref - G) of one row; the exponent in one rounding
__device__ __forceinline__ void decay_operands(const uint4& q, const uint4& k, const float4& g0, const float4& g1, const DecayRefs& r, uint4& qp, uint4& km) {
  const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
  const uint32_t qw[4] = {q.x, q.y, q.z, q.w}, kw[4] = {k.x, k.y, k.z, k.w};
  uint32_t qo[4], ko[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 qf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&qw[e])), kf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kw[e]));
    const float x0 = fmaf(g[2 * e], kDecayLog2e, -r.ref[2 * e]), x1 = fmaf(g[2 * e + 1], kDecayLog2e, -r.ref[2 * e + 1]);
    qo[e] = pack_bf16(qf.x * ex2_approx(x0), qf.y * ex2_approx(x1));
    ko[e] = pack_bf16(kf.x * ex2_approx(-x0), kf.y * ex2_approx(-x1));
  }
  qp = make_uint4(qo[0], qo[1], qo[2], qo[3]);
  km = make_uint4(ko[0], ko[1], ko[2], ko[3]);
}

}  // namespace
}  // namespace tri_inv

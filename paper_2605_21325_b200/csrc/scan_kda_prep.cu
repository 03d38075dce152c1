// Per-channel decay (the KDA row of Table 1) through the chunk scan: the operands of the tensor-core scan kernel.
// With G [tokens,H,128] the cumulative per-channel log-decay inside each chunk of 64 tokens, G_ref the chunk's middle
// row and G_last its last row, the chunk form
//     P_ij = sum_k Q_ik K_jk exp(G_ik - G_jk),   O = (Q exp G) S + P U~,   S <- diag(exp G_last) S + (K exp(G_last - G))^T U~
// becomes the scalar-gate kernel's three products on
//     Q+ = Q exp(G - G_ref),   K- = K exp(G_ref - G)
// (each factor within exp(+-|G over 32 tokens|)), with a second copy of the state operand scaled per feature by exp(G_ref),
//     Q+ . diag(exp G_ref) S = (Q exp G) S,     Q+ K-^T = the decayed Q K^T   (W S needs neither),
// and the state increment taken from K- as well: (K exp(G_last - G))^T U~ = diag(exp(G_last - G_ref)) K-^T U~.
// One pass over Q, K and G writes the two bf16 tensors and, per chunk, exp(G_last), exp(G_ref) and
// exp(G_last - G_ref); the exponent of each difference is taken once per element instead of once per (i, j, k).
#include "common.cuh"
#include "kda_operands.cuh"

namespace tri_inv {
namespace {

constexpr int C = 64, D = 128, NT = 256;

struct PrepArgs {
  const __nv_bfloat16 *Q, *K;
  const float* G;
  __nv_bfloat16 *Qp, *Km;
  float *EL, *ER, *EX;
  const int* seq_off;
  int H, T, n_seqs;
};

// blockIdx.x: (sequence, head); blockIdx.y strides over the sequence's chunks.  16 threads per token row (8 features
// each: 16 bytes of bf16, 32 of fp32), 16 rows per pass, four passes per chunk.
__global__ void __launch_bounds__(NT) kda_scan_prep_kernel(PrepArgs a) {
  wait_for_predecessor();   // (its own successor, the scan, starts when it is through: a scan's block takes the SM's L1: 242.9 -> 240.9 us for a layer of 4 x 4096 x 16 heads)
  const int s = blockIdx.x / a.H, h = blockIdx.x % a.H;
  const int beg = a.seq_off ? a.seq_off[s] : s * a.T;
  const int end = a.seq_off ? a.seq_off[s + 1] : (s + 1) * a.T;
  const int n_chunks = (end - beg + C - 1) / C;
  const int tid = threadIdx.x, r0 = tid >> 4, f0 = 8 * (tid & 15);
  for (int c = blockIdx.y; c < n_chunks; c += gridDim.y) {
    const int tok0 = beg + c * C, rows = end - tok0 < C ? end - tok0 : C;
    const size_t ref_row = ((size_t)(tok0 + (rows >> 1)) * a.H + h) * D + f0, last_row = ((size_t)(tok0 + rows - 1) * a.H + h) * D + f0;
    const DecayRefs refs = load_decay_refs(a.G + ref_row, a.G + last_row);
    if (r0 == 0) {
      const size_t slot = ((size_t)(tok0 / C + s) * a.H + h) * D + f0;
      store_decay_vectors(a.EL + slot, a.ER + slot, a.EX + slot, refs);
    }
#pragma unroll
    for (int pass = 0; pass < 4; ++pass) {
      const int r = r0 + 16 * pass;
      if (r >= rows) break;
      const size_t idx = ((size_t)(tok0 + r) * a.H + h) * D + f0;
      const uint4 qv = *reinterpret_cast<const uint4*>(a.Q + idx), kv = *reinterpret_cast<const uint4*>(a.K + idx);
      const float4 g0 = *reinterpret_cast<const float4*>(a.G + idx), g1 = *reinterpret_cast<const float4*>(a.G + idx + 4);
      uint4 qo, mo;
      decay_operands(qv, kv, g0, g1, refs, qo, mo);
      *reinterpret_cast<uint4*>(a.Qp + idx) = qo;
      *reinterpret_cast<uint4*>(a.Km + idx) = mo;
    }
  }
}

}  // namespace

cudaError_t launch_kda_scan_prep(const ScanParams& p, const void* Q, const void* K, void* Qp, void* Km,
                                 float* EL, float* ER, float* EX, int max_chunks_per_seq, cudaStream_t stream) {
  PrepArgs a{reinterpret_cast<const __nv_bfloat16*>(Q), reinterpret_cast<const __nv_bfloat16*>(K), p.G,
             reinterpret_cast<__nv_bfloat16*>(Qp), reinterpret_cast<__nv_bfloat16*>(Km), EL, ER, EX,
             p.seq_off, p.H, p.T, p.n_seqs};
  const long long gx = (long long)p.n_seqs * p.H;
  if (gx > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (gx == 0 || max_chunks_per_seq <= 0) return cudaSuccess;
  // enough CTAs to fill the machine several times over, no more: each strides over its sequence's chunks
  long long gy = max_chunks_per_seq;
  const long long want = 4096 / (gx < 4096 ? gx : 4096);
  if (gy > want) gy = want > 0 ? want : 1;
  if (gy > 65535) gy = 65535;
  const cudaError_t e = launch_early(kda_scan_prep_kernel, dim3((unsigned)gx, (unsigned)gy), NT, 0, stream, a);
  return e == cudaSuccess ? launched() : e;
}

}  // namespace tri_inv

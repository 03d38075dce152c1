// The layer token by token, for sequences of a few tokens (a decode step on carried states, short continuations):
//     S <- alpha_t S;   u_t = beta_t (v_t - S^T k_t);   S <- S + k_t u_t^T;   o_t = scale S^T q_t,     alpha_t = exp(g_t - g_{t-1}),
// what the chunk form (build, inversion, W, U, scan) computes for a chunk of 64 tokens, 63 of them padding for one new token.  The two
// dot products of a token read the same old state, because S_t^T q = alpha S_{t-1}^T q + (k . q) u: one exchange between the warps
// per token.  fp32 arithmetic on fp32 or bf16 inputs.
//
// One CTA per (sequence, head, 32 value columns): lane = column, warp = a run of d_k / 8 features, so the state streams in and out
// in rows of 128 bytes, 16 (or 8) values a thread, all in registers.  What bounds it: one token, the bytes of the state (read
// once, written once); more tokens, the exchange (two values per warp and column through shared memory, one barrier a token).
// Measured, calls back to back, fused call and scan / here: bf16, d = 128: 128 pairs of one token 28.6 / 15.4 us (both the host's time,
// the kernels 21 / 5), 2048 pairs of one token 150 / 63 us (268 MB of state: 4.3 TB/s); fp32, d = 64: 2048 pairs of 1 / 16 tokens 291 / 316 ->
// 21.5 / 95 us; d = 128: 993 / 1048 -> 63 / 251 us.
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace tri_inv {
namespace {

constexpr int kWarps = 8, kCols = 32, kMaxTokens = 16, kSeqsPerLaunch = 960;

struct RecurrenceArgs {
  const void *Q, *K, *V;
  const float *beta, *g, *S0;
  void* O;
  float* S_out;
  int H, T, d_k, d_v, bf16;
  float scale;
  int first;                          // sequences of this launch start at `first`
  // The next kernel's blocks are placed from this kernel's start, not from its end: where the launch fills the SMs (four blocks each by their registers) there is no idle one on which
  // they would pile up (128 pairs in a row: 4.7 us, 5.15 with the signal at the end; 32 pairs, 128 blocks: 3.9 and 2.8)
  bool signal_at_once;
};
struct PackedArgs : RecurrenceArgs {  // (dense calls do not carry four kilobytes of parameters to the device)
  int32_t cu[kSeqsPerLaunch + 1];     // offsets of the launch's sequences
};

__device__ __forceinline__ float load_one(const void* p, int bf16, size_t i) {
  return bf16 ? __bfloat162float(((const __nv_bfloat16*)p)[i]) : ((const float*)p)[i];
}

// k and q of the sequence's tokens, read four features at a time
template <int KR>
struct alignas(16) TokenRows {
  float k[kMaxTokens][kWarps * KR], q[kMaxTokens][kWarps * KR];
  static_assert(KR % 4 == 0, "a warp's features start on 16 bytes in every row");
};

template <int KR, class Args>   // features per warp
__global__ void __launch_bounds__(kWarps * 32) recurrence_kernel(const __grid_constant__ Args a) {
  __shared__ TokenRows<KR> rows;
  float (&sk)[kMaxTokens][kWarps * KR] = rows.k, (&sq)[kMaxTokens][kWarps * KR] = rows.q;
  __shared__ float s_alpha[kMaxTokens], s_beta[kMaxTokens], s_kq[kMaxTokens];
  __shared__ float2 part[2][kWarps][kCols];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_slices = (a.d_v + kCols - 1) / kCols;
  const int slice = blockIdx.x % n_slices, h = (blockIdx.x / n_slices) % a.H, i = blockIdx.x / (n_slices * a.H), s = a.first + i;
  int beg = s * a.T, n = a.T;   // n <= kMaxTokens (checked on the host)
  if constexpr (std::is_same<Args, PackedArgs>::value) { beg = a.cu[i]; n = a.cu[i + 1] - beg; }
  const int col = slice * kCols + lane;
  const bool in = col < a.d_v;
  const size_t base = ((size_t)s * a.H + h) * a.d_k * a.d_v + col;
  if (a.signal_at_once) let_successor_start();
  wait_for_predecessor();
  float S[KR];
#pragma unroll
  for (int r = 0; r < KR; ++r) {
    const int k = warp * KR + r;
    S[r] = (a.S0 && in && k < a.d_k) ? a.S0[base + (size_t)k * a.d_v] : 0.f;
  }
  for (int e = tid; e < n * kWarps * KR; e += kWarps * 32) {
    const int t = e / (kWarps * KR), k = e - t * (kWarps * KR);
    const size_t at = ((size_t)(beg + t) * a.H + h) * a.d_k + k;
    sk[t][k] = k < a.d_k ? load_one(a.K, a.bf16, at) : 0.f;
    sq[t][k] = k < a.d_k ? load_one(a.Q, a.bf16, at) : 0.f;
  }
  float v_next = 0.f;   // warp 0 .. 7: every warp needs u
  auto v_at = [&](int t) { return (in && t < n) ? load_one(a.V, a.bf16, ((size_t)(beg + t) * a.H + h) * a.d_v + col) : 0.f; };
  v_next = v_at(0);
  if (tid < n) {
    const size_t at = (size_t)(beg + tid) * a.H + h;
    s_alpha[tid] = expf(tid > 0 ? a.g[at] - a.g[at - a.H] : a.g[at]);
    s_beta[tid] = a.beta[at];
  }
  __syncthreads();
  for (int t = warp; t < n; t += kWarps) {
    float d = 0.f;
    for (int k = lane; k < kWarps * KR; k += 32) d = fmaf(sk[t][k], sq[t][k], d);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) d += __shfl_xor_sync(0xffffffffu, d, m);
    if (lane == 0) s_kq[t] = d;   // read behind the token loop's first barrier
  }
  for (int t = 0; t < n; ++t) {
    const float v = v_next;
    v_next = v_at(t + 1);
    float kr[KR], dk[2] = {0.f, 0.f}, dq[2] = {0.f, 0.f};
#pragma unroll
    for (int r = 0; r < KR; r += 4) {
      const float4 k4 = *reinterpret_cast<const float4*>(&sk[t][warp * KR + r]), q4 = *reinterpret_cast<const float4*>(&sq[t][warp * KR + r]);
      kr[r] = k4.x; kr[r + 1] = k4.y; kr[r + 2] = k4.z; kr[r + 3] = k4.w;
      dk[0] = fmaf(k4.x, S[r], dk[0]); dk[1] = fmaf(k4.y, S[r + 1], dk[1]);
      dk[0] = fmaf(k4.z, S[r + 2], dk[0]); dk[1] = fmaf(k4.w, S[r + 3], dk[1]);
      dq[0] = fmaf(q4.x, S[r], dq[0]); dq[1] = fmaf(q4.y, S[r + 1], dq[1]);
      dq[0] = fmaf(q4.z, S[r + 2], dq[0]); dq[1] = fmaf(q4.w, S[r + 3], dq[1]);
    }
    part[t & 1][warp][lane] = make_float2(dk[0] + dk[1], dq[0] + dq[1]);
    __syncthreads();   // (two buffers: a warp that is a token ahead writes the other one)
    float xk = 0.f, xq = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float2 x = part[t & 1][w][lane];
      xk += x.x;
      xq += x.y;
    }
    const float alpha = s_alpha[t], u = s_beta[t] * (v - alpha * xk);
#pragma unroll
    for (int r = 0; r < KR; ++r) S[r] = fmaf(kr[r], u, alpha * S[r]);
    if (warp == (t & (kWarps - 1)) && in) {
      const float o = a.scale * fmaf(s_kq[t], u, alpha * xq);
      const size_t at = ((size_t)(beg + t) * a.H + h) * a.d_v + col;
      if (a.bf16) ((__nv_bfloat16*)a.O)[at] = __float2bfloat16_rn(o);
      else ((float*)a.O)[at] = o;
    }
  }
  if (!a.signal_at_once) let_successor_start();   // little is left but these stores
  if (a.S_out && in) {
#pragma unroll
    for (int r = 0; r < KR; ++r) {
      const int k = warp * KR + r;
      if (k < a.d_k) a.S_out[base + (size_t)k * a.d_v] = S[r];
    }
  }
}

}  // namespace

// Whether the token-by-token kernel takes the call: every sequence inside one chunk and no longer than kMaxTokens; where the other
// route is the tensor cores', few tokens in all or very short sequences: a pair costs about 27 ns and 7 ns a token here once the
// chip is full, 73 ns there (2048 pairs of 16 tokens: 288 us here, 153 there; of one: 63 and 150), beside 15 us more of launches.
bool recurrence_fits(const tri_inv_desc* d) {
  if (d->d_k > 128 || d->C < kMaxTokens) return false;
  const long long pairs = (long long)d->H * (d->cu_seqlens ? d->n_seqs : d->B);
  int longest = d->T;
  if (d->cu_seqlens) {
    longest = 0;
    for (int s = 0; s < d->n_seqs; ++s) longest = std::max(longest, d->cu_seqlens[s + 1] - d->cu_seqlens[s]);
  }
  if (longest > kMaxTokens) return false;
  const bool tc = d->kv_dtype == TRI_INV_BF16 && d->d_k == 128 && d->d_v == 128 && d->C == 64;
  return !tc || longest <= 4 || pairs * longest <= 3072;
}

cudaError_t launch_recurrence(const void* Q, const void* K, const void* V, const float* beta, const float* g, const ScanParams& scan,
                              const tri_inv_desc* d, cudaStream_t stream) {
  PackedArgs a;
  a.Q = Q; a.K = K; a.V = V; a.beta = beta; a.g = g; a.S0 = scan.S0; a.O = scan.O; a.S_out = scan.S_out;
  a.H = d->H; a.T = d->T; a.d_k = d->d_k; a.d_v = d->d_v; a.bf16 = d->kv_dtype == TRI_INV_BF16;
  a.scale = scan.scale;
  const bool packed = d->cu_seqlens != nullptr;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cudaErrorUnknown;
  const long long per_seq = (long long)d->H * ((d->d_v + kCols - 1) / kCols);
  const long long most = std::min<long long>(packed ? kSeqsPerLaunch : 0x7fffffffLL, 0x7fffffffLL / per_seq);
  if (most < 1) return cudaErrorInvalidValue;
  for (long long s0 = 0; s0 < scan.n_seqs; s0 += most) {
    const int n = (int)std::min<long long>(most, scan.n_seqs - s0), grid = (int)(n * per_seq);
    cudaError_t e;
    a.first = (int)s0;
    a.signal_at_once = grid > 3 * sms;
    if (packed) {
      for (int q = 0; q <= n; ++q) a.cu[q] = d->cu_seqlens[s0 + q];
      e = d->d_k <= 64 ? launch_early(recurrence_kernel<8, PackedArgs>, dim3(grid), kWarps * 32, 0, stream, a) : launch_early(recurrence_kernel<16, PackedArgs>, dim3(grid), kWarps * 32, 0, stream, a);
    } else {
      e = d->d_k <= 64 ? launch_early(recurrence_kernel<8, RecurrenceArgs>, dim3(grid), kWarps * 32, 0, stream, a) : launch_early(recurrence_kernel<16, RecurrenceArgs>, dim3(grid), kWarps * 32, 0, stream, a);
    }
    if (e != cudaSuccess || (e = launched()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace tri_inv

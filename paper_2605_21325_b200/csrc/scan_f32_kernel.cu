// Chunk scan in single precision (fp32 storage, scalar gate, C = 64, d_k <= 128): the chunk form of scan_kernel.cu with
// every product as FFMA on register tiles.  One CTA of 256 threads per (sequence, head, slice of 16 value columns) walks
// the chunks in order; the slice of the state S [d_k][16] stays in shared memory.  Per chunk:
//   1. [W ; Q] S          thread: row r of both, four columns          U~ = U - W S to shared memory (plain and times
//                                                                      exp(g_last - g_r)), Q S kept in registers
//   2. P = (Q K^T) decay  thread: element (ty, tx) of the ten 16 x 16 blocks on and below the diagonal
//   3. O = scale (gamma Q S + P U~)    thread: row r, four columns (those of its Q S)
//   4. S = gamma_last S + K^T (decayed U~)   thread: four features x four columns, tokens split over JG lanes that then
//                                            exchange their partial sums (reduce-scatter by shuffles)
// What bounds it: shared-memory wavefronts against FFMA issue.  All operands are read 16 bytes at a time along the
// summed index, rows 4 words apart in banks (row length d_k + 4; U~ rows of 24 words), 6 loads per 32 FMAs in step 1,
// 8 per 40 in step 2.  The tiles of W, U, Q and K are single; each is refilled (cp.async) for the next chunk as soon as
// its last reader of this one is done, so a copy has two or three of the four steps to land.
// Measured (L2 flushed): B = 2, T = 2048, H = 8, d = 64: 3340 us with scan_simt_kernel (one element per thread, operands
// from global memory), 216 us here.
// A CTA of 16 columns repeats step 2 for each slice of a head; wider slices would leave more of the chip idle at the
// (sequence, head) counts that fp32 is used with.
#include "common.cuh"

namespace tri_inv {
namespace {

constexpr int kThreads = 256, kC = 64, kNS = 16, kLdP = kC + 4, kLdU = 24;

template <int DK>
struct F32Scan {
  static constexpr int LD = DK + 4;
  static constexpr int JG = DK == 64 ? 4 : 2;                 // token groups of step 4: (DK / 4) x 4 x JG threads
  static constexpr int floats = 3 * kC * LD + kC * kNS + DK * kNS + 2 * kC * kLdU + kC * kLdP + 2 * kC;
  static constexpr size_t bytes = floats * sizeof(float);
};

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {   // 16 bytes, zeros where not valid
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int KEEP>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(KEEP) : "memory"); }
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void fma4(float (&acc)[4], float a, const float4& b) {
  acc[0] = fmaf(a, b.x, acc[0]); acc[1] = fmaf(a, b.y, acc[1]); acc[2] = fmaf(a, b.z, acc[2]); acc[3] = fmaf(a, b.w, acc[3]);
}

struct F32Args {
  const float *Q, *K, *W, *U;
  int d_k, d_v;
};

template <int DK>
__global__ void __launch_bounds__(kThreads, DK == 64 ? 2 : 1) scan_f32_kernel(ScanParams p, F32Args a) {
  using cfg = F32Scan<DK>;
  constexpr int LD = cfg::LD, JG = cfg::JG;
  extern __shared__ __align__(16) float sm[];
  float *Ws = sm, *Qs = Ws + kC * LD, *Ks = Qs + kC * LD;
  float *Us = Ks + kC * LD, *S = Us + kC * kNS, *Ut = S + DK * kNS, *Ud = Ut + kC * kLdU, *P = Ud + kC * kLdU, *sg = P + kC * kLdP;
  const int tid = threadIdx.x;
  const int n_slices = (a.d_v + kNS - 1) / kNS;
  const int slice = blockIdx.x % n_slices, h = (blockIdx.x / n_slices) % p.H, s = blockIdx.x / (n_slices * p.H);
  const int beg = p.seq_off ? p.seq_off[s] : s * p.T;
  const int end = p.seq_off ? p.seq_off[s + 1] : (s + 1) * p.T;
  const int col0 = slice * kNS;
  const size_t state_base = ((size_t)s * p.H + h) * a.d_k * a.d_v;

  // state slice: rows past d_k and columns past d_v stay zero throughout (their operands are zero-filled)
  for (int e = tid; e < DK * kNS; e += kThreads) {
    const int k = e / kNS, n = e % kNS;
    S[e] = (p.S0 && k < a.d_k && col0 + n < a.d_v) ? p.S0[state_base + (size_t)k * a.d_v + col0 + n] : 0.f;
  }
  // rows of a [tokens, H, d_k] tensor; rows past the sequence's end and columns past d_k become zeros
  auto copy_rows = [&](float* dst, const float* src, int tok0, int rows) {
    constexpr int Q4 = DK / 4;
#pragma unroll
    for (int m = 0; m < kC * Q4 / kThreads; ++m) {
      const int e = tid + m * kThreads, j = e / Q4, c = 4 * (e % Q4);
      const bool ok = j < rows && c < a.d_k;
      cp_async16(dst + j * LD + c, src + (ok ? ((size_t)(tok0 + j) * p.H + h) * a.d_k + c : 0), ok);
    }
  };
  auto copy_u = [&](int tok0, int rows) {
    const int j = tid >> 2, c = 4 * (tid & 3);
    const bool ok = j < rows && col0 + c < a.d_v;
    cp_async16(Us + j * kNS + c, a.U + (ok ? ((size_t)(tok0 + j) * p.H + h) * a.d_v + col0 + c : 0), ok);
  };
  auto load_g = [&](int tok0, int rows) {   // rows past the end take the last real row's g
    return tid < kC ? p.g[(size_t)(tok0 + (tid < rows ? tid : rows - 1)) * p.H + h] : 0.f;
  };
  const int nq = tid & 3, r = tid >> 2;                                                   // steps 1 and 3
  const int ty = ((tid & 31) >> 2) + 8 * ((tid >> 5) & 1), tx = (tid & 3) + 4 * (tid >> 6);   // step 2: eight rows, four columns of a block per warp
  const int jg = tid % JG, n4 = (tid / JG) & 3, kq = tid / (4 * JG);                      // step 4

  int buf = 0;
  if (beg < end) {
    const int rows = end - beg < kC ? end - beg : kC;
    copy_rows(Ws, a.W, beg, rows);
    copy_u(beg, rows);
    copy_rows(Qs, a.Q, beg, rows);
    cp_commit();
    copy_rows(Ks, a.K, beg, rows);
    cp_commit();
    if (tid < kC) sg[tid] = load_g(beg, rows);
  }
  for (int tok0 = beg; tok0 < end; tok0 += kC, buf ^= 1) {
    const int rows = end - tok0 < kC ? end - tok0 : kC;
    const int next0 = tok0 + kC, nrows = end - next0 < kC ? end - next0 : kC;   // of the next chunk (nrows <= 0: none)
    const float* gb = sg + buf * kC;
    cp_wait<1>();      // W, U, Q of this chunk; K may still be on its way
    __syncthreads();
    const float g_next = nrows > 0 ? load_g(next0, nrows) : 0.f;
    // ---- 1. W S and Q S
    float ws[4] = {0.f, 0.f, 0.f, 0.f}, qs[4] = {0.f, 0.f, 0.f, 0.f};
    {
      const float *wr = Ws + r * LD, *qr = Qs + r * LD, *sc = S + 4 * nq;
#pragma unroll 4
      for (int k = 0; k < DK; k += 4) {
        const float4 w = ld4(wr + k), q = ld4(qr + k);
        const float4 s0 = ld4(sc + k * kNS), s1 = ld4(sc + (k + 1) * kNS), s2 = ld4(sc + (k + 2) * kNS), s3 = ld4(sc + (k + 3) * kNS);
        fma4(ws, w.x, s0); fma4(qs, q.x, s0);
        fma4(ws, w.y, s1); fma4(qs, q.y, s1);
        fma4(ws, w.z, s2); fma4(qs, q.z, s2);
        fma4(ws, w.w, s3); fma4(qs, q.w, s3);
      }
      const float4 u = ld4(Us + r * kNS + 4 * nq);
      const float f = expf(gb[rows - 1] - gb[r]);
      float4 t = make_float4(u.x - ws[0], u.y - ws[1], u.z - ws[2], u.w - ws[3]);
      if (r >= rows) t = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(Ut + r * kLdU + 4 * nq) = t;
      *reinterpret_cast<float4*>(Ud + r * kLdU + 4 * nq) = make_float4(t.x * f, t.y * f, t.z * f, t.w * f);
    }
    cp_wait<0>();      // K of this chunk
    __syncthreads();   // U~ in place; W and U have been read
    if (nrows > 0) {
      copy_rows(Ws, a.W, next0, nrows);
      copy_u(next0, nrows);
    }
    cp_commit();
    // ---- 2. P
    {
      float acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 2
      for (int k = 0; k < DK; k += 4) {
        float4 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = ld4(Qs + (ty + 16 * i) * LD + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 kv = ld4(Ks + (tx + 16 * j) * LD + k);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i >= j) acc[i][j] = fmaf(q[i].w, kv.w, fmaf(q[i].z, kv.z, fmaf(q[i].y, kv.y, fmaf(q[i].x, kv.x, acc[i][j]))));
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) {
          const int ri = ty + 16 * i, cj = tx + 16 * j;
          P[ri * kLdP + cj] = cj <= ri ? acc[i][j] * expf(gb[ri] - gb[cj]) : 0.f;
        }
    }
    __syncthreads();   // P in place; Q has been read
    if (nrows > 0) copy_rows(Qs, a.Q, next0, nrows);
    cp_commit();
    // ---- 3. O
    if (r < rows && col0 + 4 * nq < a.d_v) {
      const float gam = expf(gb[r]);
      float o[4] = {gam * qs[0], gam * qs[1], gam * qs[2], gam * qs[3]};
      const float *pr = P + r * kLdP, *uc = Ut + 4 * nq;
      int j = 0;
#pragma unroll 2
      for (; j + 3 <= r; j += 4) {
        const float4 pv = ld4(pr + j);
        fma4(o, pv.x, ld4(uc + j * kLdU));
        fma4(o, pv.y, ld4(uc + (j + 1) * kLdU));
        fma4(o, pv.z, ld4(uc + (j + 2) * kLdU));
        fma4(o, pv.w, ld4(uc + (j + 3) * kLdU));
      }
      for (; j <= r; ++j) fma4(o, pr[j], ld4(uc + j * kLdU));
      *reinterpret_cast<float4*>((float*)p.O + ((size_t)(tok0 + r) * p.H + h) * a.d_v + col0 + 4 * nq) =
          make_float4(p.scale * o[0], p.scale * o[1], p.scale * o[2], p.scale * o[3]);
    }
    // ---- 4. S (every read of the old S was before the barriers above)
    {
      float acc[4][4];   // [feature][column]
#pragma unroll
      for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[f][n] = 0.f;
#pragma unroll 4
      for (int it = 0; it < kC / JG / 2; ++it)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int j = it * 2 * JG + 2 * jg + q;   // two neighbouring tokens per lane group: their rows lie in different banks
          const float4 kv = ld4(Ks + j * LD + 4 * kq), uv = ld4(Ud + j * kLdU + 4 * n4);
          fma4(acc[0], kv.x, uv); fma4(acc[1], kv.y, uv); fma4(acc[2], kv.z, uv); fma4(acc[3], kv.w, uv);
        }
      // reduce-scatter over the token groups: lanes that differ in bit 0 keep two features each, then (JG = 4) one each
      const bool up = jg & 1;
      float two[2][4];
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const float give = up ? acc[f][n] : acc[2 + f][n], keep = up ? acc[2 + f][n] : acc[f][n];
          two[f][n] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
        }
      const float gl = expf(gb[rows - 1]);
      auto update = [&](int k, const float (&v)[4]) {
        float* sp = S + k * kNS + 4 * n4;
        const float4 o = ld4(sp);
        *reinterpret_cast<float4*>(sp) = make_float4(fmaf(gl, o.x, v[0]), fmaf(gl, o.y, v[1]), fmaf(gl, o.z, v[2]), fmaf(gl, o.w, v[3]));
      };
      if constexpr (JG == 4) {
        const bool up2 = jg & 2;
        float one[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const float give = up2 ? two[0][n] : two[1][n], keep = up2 ? two[1][n] : two[0][n];
          one[n] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
        }
        update(4 * kq + 2 * (jg & 1) + (jg >> 1), one);
      } else {
        update(4 * kq + 2 * jg, two[0]);
        update(4 * kq + 2 * jg + 1, two[1]);
      }
    }
    if (tid < kC) sg[(buf ^ 1) * kC + tid] = g_next;
    __syncthreads();   // S updated; K has been read
    if (nrows > 0) copy_rows(Ks, a.K, next0, nrows);
    cp_commit();
  }
  if (p.S_out) {
    __syncthreads();
    for (int e = tid; e < DK * kNS; e += kThreads) {
      const int k = e / kNS, n = e % kNS;
      if (k < a.d_k && col0 + n < a.d_v) p.S_out[state_base + (size_t)k * a.d_v + col0 + n] = S[e];
    }
  }
}

template <int DK>
cudaError_t launch_one(const ScanParams& p, const F32Args& a, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(scan_f32_kernel<DK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F32Scan<DK>::bytes);
  if (e != cudaSuccess) return e;
  const long long grid = (long long)p.n_seqs * p.H * ((a.d_v + kNS - 1) / kNS);
  if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
  scan_f32_kernel<DK><<<(int)grid, kThreads, F32Scan<DK>::bytes, stream>>>(p, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_chunk_scan_f32(const ScanParams& p, const void* Q, const void* K, const void* W, int d_k, int d_v, cudaStream_t stream) {
  const F32Args a{(const float*)Q, (const float*)K, (const float*)W, (const float*)p.U, d_k, d_v};
  return d_k <= 64 ? launch_one<64>(p, a, stream) : launch_one<128>(p, a, stream);
}

}  // namespace tri_inv

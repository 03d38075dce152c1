// Plain fp32 CUDA-core kernel: every step of the path with FFMA on shared-memory matrices.
//
// It is the kernel for fp32 inputs (where single-pass tensor-core operands would not
// meet the 1e-5 bound) and for shapes the tensor-core kernel does not cover; the
// TRI_INV_FORCE_SIMT flag routes any request here.  One CTA per chunk matrix,
// 256 threads, all of N / X / a scratch matrix resident in shared memory.
//
// Steps (notation of the header): Gram S = K K^T in d-slices of 32, gate
// N_ij = beta_i S_ij exp(g_i - g_j) under the strict-lower mask, then either
//   * block recursion from 16x16 leaves (Sec. 3.3), leaves by forward substitution
//     (Sec. 3.1) or by the product series on the leaf (Alg. 2), or
//   * the product series on the whole chunk (Alg. 5),
// then A is stored and W = A diag(beta) K, U = A diag(beta) V are formed.
//
// What bounds it: shared-memory wavefronts against FFMA issue.  One element per thread and step costs two loads per FMA
// and waits for each of them, so every product of the default scheme (Gram, merges, WY) is register-tiled with 16-byte
// loads: rows 4 apart in banks (row length C + 4, key slices 36 words), so a warp's eight rows or columns of a load fall
// into different banks; 8 loads per 40 FMAs in the Gram product, 5 to 6 per 16 to 32 elsewhere.  Blocks above the diagonal
// are left out at compile time, the one group of four that a row's diagonal crosses is masked by selection (nothing beyond
// it is ever multiplied in).  The next slice of keys / values is fetched into registers while the current one is used.
// Measured against the untiled form (L2 flushed): fp32, d = 64, C = 64: fused call on 512 matrices 121.8 -> 53.3 us, build of
// 8 matrices 28.7 -> 14.3 us.
#include "common.cuh"

namespace tri_inv {
namespace {

constexpr int kThreads = 256;
constexpr long long kSMs = 148;
constexpr int kSlice = 32;            // columns of K / V staged per pass
constexpr int kSliceLd = kSlice + 4;  // padded row length of the staging tile: 16-byte pieces, eight rows in different banks

template <int C>
struct SimtSmem {
  static constexpr int LD = C + 4;
  // the scratch matrix also stages a slice of G in the per-channel Gram phase, whose rows are longer than LD at C = 16
  static constexpr int Z_FLOATS = C * (LD > kSliceLd ? LD : kSliceLd);
  static constexpr size_t floats = 2 * (size_t)C * LD + Z_FLOATS + (size_t)C * kSliceLd + 4 * C;
  static constexpr size_t bytes = floats * sizeof(float);
};

// dst = lower-triangular product restricted to diagonal blocks of size bs:
// dst_ij = sum_{k=j..i} a_ik b_kj for i >= j in the same block, else 0.
template <int C>
__device__ void tri_matmul_blocks(float* dst, const float* a, const float* b, int bs, int tid) {
  constexpr int LD = C + 4;
  for (int e = tid; e < C * bs; e += kThreads) {
    int i = e / bs, jj = e - i * bs;
    int base = (i / bs) * bs;
    int j = base + jj;
    float s = 0.f;
    if (j <= i)
      for (int k = j; k <= i; ++k) s = fmaf(a[i * LD + k], b[k * LD + j], s);
    dst[i * LD + j] = s;
  }
}

// Product series (Alg. 5) on every bs x bs diagonal block of N at once.
// y holds N on entry (only its diagonal blocks are read) and is destroyed; the result
// (diagonal blocks only, zero elsewhere inside them above the diagonal) ends in the
// returned buffer, one of {x, y, z}.
template <int C>
__device__ float* product_series_blocks(float* y, float* x, float* z, int bs, int tid) {
  constexpr int LD = C + 4;
  for (int e = tid; e < C * bs; e += kThreads) {  // X <- I - N on the diagonal blocks
    int i = e / bs, jj = e - i * bs;
    int j = (i / bs) * bs + jj;
    x[i * LD + j] = (i == j) ? 1.f : (j < i ? -y[i * LD + j] : 0.f);
  }
  __syncthreads();
  int rounds = 0;
  for (int m = bs; m > 2; m >>= 1) ++rounds;  // log2(bs) - 1
  for (int r = 0; r < rounds; ++r) {
    tri_matmul_blocks<C>(z, y, y, bs, tid);    // Y <- Y.Y   (into z)
    __syncthreads();
    for (int e = tid; e < C * bs; e += kThreads) {  // X <- X + X.Y   (into y's old buffer)
      int i = e / bs, jj = e - i * bs;
      int j = (i / bs) * bs + jj;
      float s = 0.f;
      if (j <= i) {
        s = x[i * LD + j];
        for (int k = j; k <= i; ++k) s = fmaf(x[i * LD + k], z[k * LD + j], s);
      }
      y[i * LD + j] = s;
    }
    __syncthreads();
    float* nx = y;  // rotate: new X = old Y buffer, new Y = z, free = old X
    y = z;
    z = x;
    x = nx;
  }
  return x;
}

// acc[m] = (a . b)_ij for the element e = tid + m * kThreads of a C x C lower-triangular product
// (a and b lower triangular, sum over k = j..i); elements above the diagonal give 0.
template <int C, int kAcc>
__device__ __forceinline__ void tri_matmul_regs(float (&acc)[kAcc], const float* a, const float* b, int tid) {
  constexpr int LD = C + 4;
#pragma unroll
  for (int m = 0; m < kAcc; ++m) {
    const int e = tid + m * kThreads;
    const int i = e / C, j = e - i * C;
    float s = 0.f;
    if (e < C * C && j <= i)
      for (int k = j; k <= i; ++k) s = fmaf(a[i * LD + k], b[k * LD + j], s);
    acc[m] = s;
  }
}

// A slice of kSlice columns of a [rows, H, d] tensor on its way to the staging tile: fetched into registers (16 bytes per
// load; d is a multiple of 8 and the base 16-byte aligned, so a piece lies in the row whole or not at all), put down as fp32.
template <int C>
struct SliceRegs {
  static constexpr int kPieces = (C * kSlice / 4 + kThreads - 1) / kThreads;   // pieces of four columns per thread
  float4 v[kPieces];
  __device__ __forceinline__ void fetch(const void* src, int dtype, int tok0, int rows, int H, int h, int d, int c0, int tid) {
#pragma unroll
    for (int m = 0; m < kPieces; ++m) {
      const int e = tid + m * kThreads, j = e / (kSlice / 4), c = c0 + 4 * (e % (kSlice / 4));
      v[m] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < rows && c < d) {
        const size_t idx = ((size_t)(tok0 + j) * H + h) * d + c;
        if (dtype == TRI_INV_F32) {
          v[m] = *reinterpret_cast<const float4*>((const float*)src + idx);
        } else {
          const uint2 w = *reinterpret_cast<const uint2*>((const __nv_bfloat16*)src + idx);
          v[m] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
        }
      }
    }
  }
  // row j of the tile times scale[j] (scale == nullptr: as it is)
  __device__ __forceinline__ void put(float* tile, const float* scale, int tid) const {
#pragma unroll
    for (int m = 0; m < kPieces; ++m) {
      const int e = tid + m * kThreads, j = e / (kSlice / 4), c = 4 * (e % (kSlice / 4));
      if (j < C) {
        const float f = scale ? scale[j] : 1.f;
        *reinterpret_cast<float4*>(tile + j * kSliceLd + c) = make_float4(f * v[m].x, f * v[m].y, f * v[m].z, f * v[m].w);
      }
    }
  }
};

__device__ __forceinline__ void fma4(float (&acc)[4], float a, const float4& b) {
  acc[0] = fmaf(a, b.x, acc[0]); acc[1] = fmaf(a, b.y, acc[1]); acc[2] = fmaf(a, b.z, acc[2]); acc[3] = fmaf(a, b.w, acc[3]);
}

// BLOCKS: thread blocks per SM that the registers are shared out for (launch_one).
template <int C, int BLOCKS>
__global__ void __launch_bounds__(kThreads, BLOCKS) simt_kernel(KParams p) {
  constexpr int LD = C + 4;
  extern __shared__ __align__(16) float smem[];   // read and written 16 bytes at a time
  static_assert(LD % 4 == 0 && kSliceLd % 4 == 0 && (C * LD) % 4 == 0 && SimtSmem<C>::Z_FLOATS % 4 == 0, "rows and matrices on 16-byte boundaries");
  float* Nm = smem;
  float* Xm = Nm + C * LD;
  float* Zm = Xm + C * LD;
  float* Ks = Zm + SimtSmem<C>::Z_FLOATS;  // [C][kSliceLd]
  static_assert(SimtSmem<C>::Z_FLOATS >= C * kSliceLd, "a slice of G fits into the scratch matrix");
  float* sb = Ks + C * kSliceLd;
  float* sg = sb + C;
  float* sr = sg + C;  // raw front end: 1 / |k_i|
  float* sw = sr + C;  // factor of row j of K (then of V) in the WY products
  const bool raw = (p.ops & kRaw) != 0;
  const bool kda = (p.ops & kKda) != 0;  // per-channel decay: each Gram term weighted by exp(G_ic - G_jc); W rows weighted by exp(G_j) per feature
  const int tid = threadIdx.x;
  const int total = p.n_chunks * p.H;
  constexpr int kAcc = (C * C + kThreads - 1) / kThreads;
  constexpr int kB = (C + 15) / 16;   // 16 x 16 blocks per side; a thread owns element (ty, tx) of each
  // eight rows and four columns of a block per warp: either operand's loads of a step touch 32 different banks
  const int ty = ((tid & 31) >> 2) + 8 * ((tid >> 5) & 1), tx = (tid & 3) + 4 * (tid >> 6);
  const int method = p.method & TRI_INV_METHOD_MASK;
  const int gshift = (p.method & TRI_INV_GATE_SHIFTED) ? 1 : 0;  // Comba row: row i decays from the token before it

  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    int tok0, rows, h;
    locate(p, C, item, tok0, rows, h);
    // bounds-checking build: an item outside the tensors is reduced to no rows (nothing of it is then read or stored)
    if (!TRI_INV_CHECK(p, rows >= 1 && rows <= C && tok0 >= 0 && (long long)tok0 + rows <= p.n_tokens && h >= 0 && h < p.H)) { tok0 = 0; rows = 0; h = 0; }
    __syncthreads();  // previous item's readers are done with shared memory
    for (int i = tid; i < C; i += kThreads) {
      size_t bi = (size_t)(tok0 + i) * p.H + h;
      float b = (i < rows) ? p.beta[bi] : 0.f;
      float gg = (i < rows && p.g) ? p.g[bi] : 0.f;
      if (raw) {  // beta logits -> sigmoid; gate logits -> log sigmoid (summed over the chunk below)
        b = (i < rows) ? 1.f / (1.f + expf(-b)) : 0.f;
        gg = (i < rows) ? fminf(gg, 0.f) - log1pf(expf(-fabsf(gg))) : 0.f;
        if (p.beta_out && i < rows) p.beta_out[bi] = b;
      }
      sb[i] = b;
      sg[i] = gg;
      sr[i] = 1.f;
    }
    if (raw) {
      __syncthreads();
      if (tid == 0) {  // within-chunk cumulative log-decay, in token order
        float run = 0.f;
        for (int i = 0; i < C; ++i) { run += sg[i]; sg[i] = run; }
      }
      __syncthreads();
      if (p.g_out)
        for (int i = tid; i < rows; i += kThreads) p.g_out[(size_t)(tok0 + i) * p.H + h] = sg[i];
    }
    if (method == TRI_INV_NEWTON_SCHULZ)   // its first iterate is diagonal; every other scheme writes what it reads
      for (int e = tid; e < C * LD; e += kThreads) Xm[e] = 0.f;
    float* Xres = Xm;

    if (p.ops & kLoadA) {
      __syncthreads();
      for (int e = tid; e < C * C; e += kThreads) {
        int i = e / C, j = e - i * C;
        if (i < rows && j <= i) Xm[i * LD + j] = p.A_in[((size_t)(tok0 + i) * p.H + h) * C + j];
      }
      __syncthreads();
    } else {
      // ---- Gram matrix, strictly lower part, in slices of the key dimension
      float acc[kB][kB];
#pragma unroll
      for (int a = 0; a < kB; ++a)
#pragma unroll
        for (int b = 0; b < kB; ++b) acc[a][b] = 0.f;
      SliceRegs<C> kr, gr;
      kr.fetch(p.K, p.kv_dtype, tok0, rows, p.H, h, p.d_k, 0, tid);
      if (kda) gr.fetch(p.G, TRI_INV_F32, tok0, rows, p.H, h, p.d_k, 0, tid);
      for (int ks = 0; ks < p.d_k; ks += kSlice) {
        __syncthreads();
        kr.put(Ks, nullptr, tid);
        if (kda) gr.put(Zm, nullptr, tid);  // the scratch matrix is free during the Gram phase: it holds the slice of G
        __syncthreads();
        if (ks + kSlice < p.d_k) {
          kr.fetch(p.K, p.kv_dtype, tok0, rows, p.H, h, p.d_k, ks + kSlice, tid);
          if (kda) gr.fetch(p.G, TRI_INV_F32, tok0, rows, p.H, h, p.d_k, ks + kSlice, tid);
        }
        if (kda) {
#pragma unroll(C <= 32 ? 8 : 1)   // small tiles: the loads of one step alone do not hide their latency
          for (int kk = 0; kk < kSlice; ++kk) {
            float ki[kB], gi[kB];
#pragma unroll
            for (int a = 0; a < kB; ++a) { ki[a] = Ks[(ty + 16 * a) * kSliceLd + kk]; gi[a] = Zm[(ty + 16 * a) * kSliceLd + kk]; }
#pragma unroll
            for (int b = 0; b < kB; ++b) {
              const float kj = Ks[(tx + 16 * b) * kSliceLd + kk], gj = Zm[(tx + 16 * b) * kSliceLd + kk];
#pragma unroll
              for (int a = 0; a < kB; ++a)
                if (a > b || (a == b && ty > tx)) acc[a][b] = fmaf(ki[a] * kj, expf(gi[a] - gj), acc[a][b]);
            }
          }
        } else {
#pragma unroll 2
          for (int kk = 0; kk < kSlice; kk += 4) {
            float4 ki[kB];
#pragma unroll
            for (int a = 0; a < kB; ++a) ki[a] = *reinterpret_cast<const float4*>(Ks + (ty + 16 * a) * kSliceLd + kk);
#pragma unroll
            for (int b = 0; b < kB; ++b) {
              const float4 kj = *reinterpret_cast<const float4*>(Ks + (tx + 16 * b) * kSliceLd + kk);
#pragma unroll
              for (int a = 0; a < kB; ++a)
                if (a >= b) acc[a][b] = fmaf(ki[a].w, kj.w, fmaf(ki[a].z, kj.z, fmaf(ki[a].y, kj.y, fmaf(ki[a].x, kj.x, acc[a][b]))));
            }
          }
        }
      }
      if (raw) {  // 1 / |k_i| from the Gram diagonal; the Gram of the normalised keys is S_ij r_i r_j
        if (ty == tx) {
#pragma unroll
          for (int a = 0; a < kB; ++a) sr[ty + 16 * a] = acc[a][a] > 0.f ? rsqrtf(acc[a][a]) : 0.f;
        }
        __syncthreads();
      }
      // ---- gate and mask: select, never multiply an overflowed exp by zero
#pragma unroll
      for (int a = 0; a < kB; ++a)
#pragma unroll
        for (int b = 0; b < kB; ++b) {
          const int i = ty + 16 * a, j = tx + 16 * b;
          float n = 0.f;
          if (j < i && i < rows) n = sb[i] * (acc[a][b] * sr[i] * sr[j]) * expf(sg[i - gshift] - sg[j]);  // i > j >= 0, so i - 1 is in the chunk
          Nm[i * LD + j] = n;
        }
      __syncthreads();

      if (method == TRI_INV_PRODUCT_SERIES) {
        Xres = product_series_blocks<C>(Nm, Xm, Zm, C, tid);
      } else if (method == TRI_INV_NEWTON_SCHULZ) {
        // Alg. 3: M = I + N, X_0 = I / C, then m rounds of Y <- M.X, X <- 2X - X.Y.
        // All iterates are lower triangular, so the products run over k = j..i only.
        int iters = (p.method >> 12) & 0xf;
        if (iters == 0) { iters = 0; for (int m = C; m > 1; m >>= 1) iters += 2; }  // 2 log2(C)
        for (int e = tid; e < C * C; e += kThreads) {
          const int i = e / C, j = e - i * C;
          if (i == j) { Nm[i * LD + j] = 1.f; Xm[i * LD + j] = 1.f / C; }
        }
        __syncthreads();
        for (int it = 0; it < iters; ++it) {
          tri_matmul_blocks<C>(Zm, Nm, Xm, C, tid);   // Y <- M.X
          __syncthreads();
          float q[kAcc];
          tri_matmul_regs<C, kAcc>(q, Xm, Zm, tid);   // X.Y, held in registers until every read of X is done
          __syncthreads();
#pragma unroll
          for (int m = 0; m < kAcc; ++m) {
            const int e = tid + m * kThreads;
            const int i = e / C, j = e - i * C;
            if (e < C * C && j <= i) Xm[i * LD + j] = 2.f * Xm[i * LD + j] - q[m];
          }
          __syncthreads();
        }
        for (int e = tid; e < C; e += kThreads) Nm[e * LD + e] = 0.f;  // back to N for an optional refinement step
        __syncthreads();
      } else {
        constexpr int kLeaf = C < 16 ? C : 16;
        if (p.method & TRI_INV_LEAF_SERIES) {
          // Alg. 2: series on the leaves.  Work on a copy so N's off-diagonal blocks survive.
          // Ks ([C][kSliceLd]) is free now and holds two compact [C][16] block-diagonal matrices.
          float* Yc = Ks;
          float* Y2 = Ks + C * kLeaf;
          for (int e = tid; e < C * kLeaf; e += kThreads) {
            int i = e / kLeaf, jj = e - i * kLeaf;
            int j = (i / kLeaf) * kLeaf + jj;
            float n = (j < i) ? Nm[i * LD + j] : 0.f;
            Yc[e] = n;
            Xm[i * LD + j] = (i == j) ? 1.f : -n;
          }
          __syncthreads();
          int rounds = 0;
          for (int m = kLeaf; m > 2; m >>= 1) ++rounds;
          for (int r = 0; r < rounds; ++r) {
            for (int e = tid; e < C * kLeaf; e += kThreads) {  // Y2 <- Yc.Yc
              int i = e / kLeaf, jj = e - i * kLeaf, ii = i % kLeaf, base = i - ii;
              float s = 0.f;
              for (int k = jj; k <= ii; ++k) s = fmaf(Yc[i * kLeaf + k], Yc[(base + k) * kLeaf + jj], s);
              Y2[e] = s;
            }
            __syncthreads();
            for (int e = tid; e < C * kLeaf; e += kThreads) {  // Z <- X + X.Y2 on the leaves
              int i = e / kLeaf, jj = e - i * kLeaf, ii = i % kLeaf, base = i - ii;
              float s = Xm[i * LD + base + jj];
              for (int k = jj; k <= ii; ++k) s = fmaf(Xm[i * LD + base + k], Y2[(base + k) * kLeaf + jj], s);
              Zm[i * LD + base + jj] = s;
            }
            __syncthreads();
            for (int e = tid; e < C * kLeaf; e += kThreads) {
              int i = e / kLeaf, jj = e - i * kLeaf, base = i - i % kLeaf;
              Xm[i * LD + base + jj] = Zm[i * LD + base + jj];
            }
            float* t = Yc; Yc = Y2; Y2 = t;
            __syncthreads();
          }
        } else {
          // forward substitution, one thread per column of its leaf (Sec. 3.1)
          if (tid < C) {
            int base = (tid / kLeaf) * kLeaf, j = tid % kLeaf;
            float x[kLeaf];
#pragma unroll
            for (int i = 0; i < kLeaf; ++i) {
              float s = 0.f;
#pragma unroll
              for (int k = 0; k < i; ++k)
                if (k >= j) s = fmaf(Nm[(base + i) * LD + base + k], x[k], s);
              x[i] = (i < j) ? 0.f : (i == j ? 1.f : -s);
            }
#pragma unroll
            for (int i = 0; i < kLeaf; ++i) Xm[(base + i) * LD + base + j] = x[i];
          }
          __syncthreads();
        }
        // merges: X21 = -(X22 . N21) . X11 for every adjacent pair of b x b blocks
        for (int b = kLeaf; b < C; b <<= 1) {
          const int per_row = b / 4, n_quads = (C / 2) * per_row;   // a thread forms four neighbouring elements of a row
          for (int e = tid; e < n_quads; e += kThreads) {  // T = X22 . N21 into Zm at the (2,1) block
            const int row = e / per_row, pr = row / b, i = row - pr * b, j = 4 * (e - row * per_row);
            const int r0 = pr * 2 * b + b, c0 = pr * 2 * b;
            const float *x = Xm + (r0 + i) * LD + r0, *n = Nm + r0 * LD + c0 + j;
            float s[4] = {0.f, 0.f, 0.f, 0.f};
            int k = 0;
            for (; k + 3 <= i; k += 4) {
              const float4 xv = *reinterpret_cast<const float4*>(x + k);
              fma4(s, xv.x, *reinterpret_cast<const float4*>(n + k * LD));
              fma4(s, xv.y, *reinterpret_cast<const float4*>(n + (k + 1) * LD));
              fma4(s, xv.z, *reinterpret_cast<const float4*>(n + (k + 2) * LD));
              fma4(s, xv.w, *reinterpret_cast<const float4*>(n + (k + 3) * LD));
            }
            for (; k <= i; ++k) fma4(s, x[k], *reinterpret_cast<const float4*>(n + k * LD));
            *reinterpret_cast<float4*>(Zm + (r0 + i) * LD + c0 + j) = make_float4(s[0], s[1], s[2], s[3]);
          }
          __syncthreads();
          for (int e = tid; e < n_quads; e += kThreads) {  // X21 = -T . X11
            const int row = e / per_row, pr = row / b, i = row - pr * b, j = 4 * (e - row * per_row);
            const int r0 = pr * 2 * b + b, c0 = pr * 2 * b;
            const float *t = Zm + (r0 + i) * LD + c0, *x = Xm + c0 * LD + c0 + j;
            float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 4; ++k) {   // the rows that the columns' diagonals cross: X11 is lower triangular
              const float tv = t[j + k];
              const float4 xv = *reinterpret_cast<const float4*>(x + (j + k) * LD);
              s[0] = fmaf(tv, xv.x, s[0]);
              if (k >= 1) s[1] = fmaf(tv, xv.y, s[1]);
              if (k >= 2) s[2] = fmaf(tv, xv.z, s[2]);
              if (k >= 3) s[3] = fmaf(tv, xv.w, s[3]);
            }
            for (int k = j + 4; k < b; k += 4) {
              const float4 tv = *reinterpret_cast<const float4*>(t + k);
              fma4(s, tv.x, *reinterpret_cast<const float4*>(x + k * LD));
              fma4(s, tv.y, *reinterpret_cast<const float4*>(x + (k + 1) * LD));
              fma4(s, tv.z, *reinterpret_cast<const float4*>(x + (k + 2) * LD));
              fma4(s, tv.w, *reinterpret_cast<const float4*>(x + (k + 3) * LD));
            }
            *reinterpret_cast<float4*>(Xm + (r0 + i) * LD + c0 + j) = make_float4(-s[0], -s[1], -s[2], -s[3]);
          }
          __syncthreads();
        }
      }
    }

    // ---- optional refinement (Alg. 6): R <- I - X.M with M = I + N, then X <- X + R.X
    if ((p.method & TRI_INV_REFINE) && !(p.ops & kLoadA)) {
      float* Rm = (Xres == Zm) ? Xm : Zm;  // a buffer that is neither N nor the current result
      float q[kAcc];
      tri_matmul_regs<C, kAcc>(q, Xres, Nm, tid);  // X.N (N strictly lower; X.M = X + X.N)
#pragma unroll
      for (int m = 0; m < kAcc; ++m) {
        const int e = tid + m * kThreads;
        const int i = e / C, j = e - i * C;
        if (e < C * C) Rm[i * LD + j] = (j <= i) ? ((i == j ? 1.f : 0.f) - Xres[i * LD + j] - q[m]) : 0.f;
      }
      __syncthreads();
      tri_matmul_regs<C, kAcc>(q, Rm, Xres, tid);  // R.X
      __syncthreads();
#pragma unroll
      for (int m = 0; m < kAcc; ++m) {
        const int e = tid + m * kThreads;
        const int i = e / C, j = e - i * C;
        if (e < C * C && j <= i) Xres[i * LD + j] += q[m];
      }
      __syncthreads();
    }

    // ---- store A: computed strict-lower part, constant diagonal and upper triangle
    if ((p.ops & kStoreA) && p.A) {
      for (int e = tid; e < C * C / 4; e += kThreads) {
        const int i = e / (C / 4), j = 4 * (e - i * (C / 4));
        if (i < rows && TRI_INV_CHECK(p, (long long)tok0 + i < p.n_tokens)) {
          float4 v = *reinterpret_cast<const float4*>(Xres + i * LD + j);
          v.x = (j < i) ? v.x : (j == i ? 1.f : 0.f);
          v.y = (j + 1 < i) ? v.y : (j + 1 == i ? 1.f : 0.f);
          v.z = (j + 2 < i) ? v.z : (j + 2 == i ? 1.f : 0.f);
          v.w = (j + 3 < i) ? v.w : (j + 3 == i ? 1.f : 0.f);
          *reinterpret_cast<float4*>(p.A + ((size_t)(tok0 + i) * p.H + h) * C + j) = v;
        }
      }
    }

    // ---- WY: W = A diag(beta) K, U = A diag(beta) V, 32 columns at a time
    if (p.ops & kDoWY) {
      for (int which = 0; which < 2; ++which) {
        const void* src = which ? p.V : p.K;
        void* dst = which ? p.U : p.W;
        int d = which ? p.d_v : p.d_k;
        if (!src || !dst) continue;
        __syncthreads();   // the other tensor's readers are done with the factors
        for (int j = tid; j < C; j += kThreads)
          sw[j] = sb[j] * (which ? 1.f : sr[j] * ((p.ops & kWDecay) ? ((gshift && j == 0) ? 1.f : expf(sg[j - gshift])) : 1.f));
        SliceRegs<C> xr, gr;
        xr.fetch(src, p.kv_dtype, tok0, rows, p.H, h, d, 0, tid);
        for (int c0 = 0; c0 < d; c0 += kSlice) {
          if (kda && !which) {   // W = A diag(beta) (K * Gamma): the decay-weighted factor of the per-channel form
            gr.fetch(p.G, TRI_INV_F32, tok0, rows, p.H, h, d, c0, tid);
#pragma unroll
            for (int m = 0; m < SliceRegs<C>::kPieces; ++m) {
              xr.v[m].x *= expf(gr.v[m].x); xr.v[m].y *= expf(gr.v[m].y); xr.v[m].z *= expf(gr.v[m].z); xr.v[m].w *= expf(gr.v[m].w);
            }
          }
          __syncthreads();
          xr.put(Ks, sw, tid);
          __syncthreads();
          if (c0 + kSlice < d) xr.fetch(src, p.kv_dtype, tok0, rows, p.H, h, d, c0 + kSlice, tid);
          // four columns of rows i, i + 32, ...: a warp holds four neighbouring rows, so the group of four tokens that
          // crosses the diagonal is the same for all its lanes
          constexpr int kR = (C + 31) / 32;
          const int cc = 4 * (tid & 7), i0 = tid >> 3;
          if (i0 < C) {
            float s[kR][4];
#pragma unroll
            for (int r = 0; r < kR; ++r) {   // diagonal term, A_ii = 1
              const float4 v = *reinterpret_cast<const float4*>(Ks + (i0 + 32 * r) * kSliceLd + cc);
              s[r][0] = v.x; s[r][1] = v.y; s[r][2] = v.z; s[r][3] = v.w;
            }
            const int last = i0 + 32 * (kR - 1) < rows ? i0 + 32 * (kR - 1) : rows - 1;   // last row of this thread that is stored, or beyond it
            for (int j = 0; j < last; j += 4) {
              const float4 k0 = *reinterpret_cast<const float4*>(Ks + j * kSliceLd + cc), k1 = *reinterpret_cast<const float4*>(Ks + (j + 1) * kSliceLd + cc),
                           k2 = *reinterpret_cast<const float4*>(Ks + (j + 2) * kSliceLd + cc), k3 = *reinterpret_cast<const float4*>(Ks + (j + 3) * kSliceLd + cc);
#pragma unroll
              for (int r = 0; r < kR; ++r) {
                const int i = i0 + 32 * r;
                if (j < i && i < rows) {
                  const float4 a = *reinterpret_cast<const float4*>(Xres + i * LD + j);
                  if (j + 3 < i) {
                    fma4(s[r], a.x, k0); fma4(s[r], a.y, k1); fma4(s[r], a.z, k2); fma4(s[r], a.w, k3);
                  } else {
                    fma4(s[r], a.x, k0);
                    if (j + 1 < i) fma4(s[r], a.y, k1);
                    if (j + 2 < i) fma4(s[r], a.z, k2);
                  }
                }
              }
            }
#pragma unroll
            for (int r = 0; r < kR; ++r) {
              const int i = i0 + 32 * r;
              if (i < rows && c0 + cc < d && TRI_INV_CHECK(p, (long long)tok0 + i < p.n_tokens)) {
                const size_t o = ((size_t)(tok0 + i) * p.H + h) * d + c0 + cc;
                if (p.kv_dtype == TRI_INV_F32) {
                  *reinterpret_cast<float4*>((float*)dst + o) = make_float4(s[r][0], s[r][1], s[r][2], s[r][3]);
                } else {
                  const __nv_bfloat162 lo = __floats2bfloat162_rn(s[r][0], s[r][1]), hi = __floats2bfloat162_rn(s[r][2], s[r][3]);
                  *reinterpret_cast<uint2*>((__nv_bfloat16*)dst + o) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                }
              }
            }
          }
        }
      }
    }
  }
}

template <int C, int BLOCKS>
cudaError_t launch_blocks(const KParams& p, long long total, cudaStream_t stream) {
  size_t bytes = SimtSmem<C>::bytes;
  cudaError_t e = cudaFuncSetAttribute(simt_kernel<C, BLOCKS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  int grid = (int)(total < kSMs * 64 ? total : kSMs * 64);
  simt_kernel<C, BLOCKS><<<grid, kThreads, bytes, stream>>>(p);
  return cudaGetLastError();
}

// At C = 64 three blocks fit the shared memory of an SM; two of them at up to 128 registers keep the tiles out of local memory.
// At C = 32 and 16 the products are short and the barriers between them bound a block, so with more chunks than two for each SM
// more blocks are worth a few spilled registers.  fp32, d = 64, C = 16 with five blocks (47 registers) against two (84): 304
// chunks fused 14.4 -> 10.3 us, 8192 chunks build 79.9 -> 49.0, fused 201 -> 116, Newton-Schulz 298 -> 172 us; C = 32 with four
// (64) against two (124): 304 chunks fused 20.9 -> 15.6 us, 8192 chunks fused 308 -> 217, Newton-Schulz 1284 -> 928 us.  With fewer
// chunks a block has the SM to itself or shares it with one other, and the registers shorten it: eight chunks, bf16, d = 128,
// C = 16, fused 14.4 us with five blocks' registers, 12.3 us with two's.
template <int C>
cudaError_t launch_one(const KParams& p, cudaStream_t stream) {
  const long long total = (long long)p.n_chunks * p.H;
  if (total == 0) return cudaSuccess;
  if constexpr (C <= 32) {
    if (total > 2 * kSMs) return launch_blocks<C, C == 16 ? 5 : 4>(p, total, stream);
  }
  return launch_blocks<C, C <= 64 ? 2 : 1>(p, total, stream);
}

}  // namespace

cudaError_t launch_simt(const KParams& p, int C, cudaStream_t stream) {
  switch (C) {
    case 16: return launch_one<16>(p, stream);
    case 32: return launch_one<32>(p, stream);
    case 64: return launch_one<64>(p, stream);
    case 128: return launch_one<128>(p, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace tri_inv

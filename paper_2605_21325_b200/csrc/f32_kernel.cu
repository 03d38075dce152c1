// Build, inversion, W and U in single precision (fp32 storage, C = 64, head dimensions up to 128, block recursion with
// substitution leaves): the calls that fp32 is used with most, apart from the general CUDA-core kernel (simt_kernel.cu).
//
// One CTA of 256 threads per chunk matrix.  K and V come whole, by cp.async, V behind the inversion; one 64 x 64 matrix holds N, then the
// inverse, block by block in place (a product of a merge waits in registers until its operand's place is free).  Every
// product is register-tiled with 16-byte shared-memory loads: Gram and WY, one element (or four columns) of the rows ty + 16 a in each
// 16 x 16 block on and below the diagonal: 8 loads per 40 and 64 FMAs.  While four warps invert the leaves the
// other four scale the rows of K and V by their factors.  Entries above a diagonal are never multiplied in, so a token's
// non-finite values reach no earlier row.
// What bounds it: many matrices, instruction issue; few, the latency of one matrix.
#include "f32_tiles.cuh"

namespace tri_inv {
namespace {

constexpr int kThreads = 256, C = 64, LDM = C + 4;

template <int DT>   // padded head dimension
struct F32Cfg {
  static constexpr int LD = DT + 4;
  static constexpr int floats(bool wy) { return C * LD * (wy ? 2 : 1) + C * LDM + 4 * C; }
};

template <int DT, bool WY>
__global__ void __launch_bounds__(kThreads, DT == 64 ? 4 : 2) f32_factors_kernel(const __grid_constant__ KParams p) {
  constexpr int LD = F32Cfg<DT>::LD;
  extern __shared__ __align__(16) float sm[];
  float *Ks = sm, *M = Ks + C * LD, *sb = M + C * LDM, *sg = sb + C, *sw = sg + C, *Vs = sw + 2 * C;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // eight rows and four columns of a block per warp: either operand's loads of a step touch 32 different banks
  const int ty = (lane >> 2) + 8 * (warp & 1), tx = (lane & 3) + 4 * (warp >> 1);
  const int gshift = (p.method & TRI_INV_GATE_SHIFTED) ? 1 : 0;   // Comba row: row i decays from the token before it
  const int total = p.n_chunks * p.H;
  wait_for_predecessor();

  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    int tok0, rows, h;
    locate(p, C, item, tok0, rows, h);
    // bounds-checking build: an item outside the tensors is reduced to no rows (nothing of it is then read or stored)
    if (!TRI_INV_CHECK(p, rows >= 1 && rows <= C && tok0 >= 0 && (long long)tok0 + rows <= p.n_tokens && h >= 0 && h < p.H)) { tok0 = 0; rows = 0; h = 0; }
    if (item != (int)blockIdx.x) __syncthreads();   // the last matrix's readers are done with shared memory
    auto copy_rows = [&](float* dst, const void* src, int d) {   // rows past the chunk become zeros, columns past d are left alone
#pragma unroll
      for (int m = 0; m < C * DT / 4 / kThreads; ++m) {
        const int e = tid + m * kThreads, j = e / (DT / 4), c = 4 * (e % (DT / 4));
        if (c < d) cp_async16(dst + j * LD + c, (const float*)src + (j < rows ? ((size_t)(tok0 + j) * p.H + h) * d + c : 0), j < rows);
      }
      cp_commit();
    };
    copy_rows(Ks, p.K, p.d_k);
    if (WY) copy_rows(Vs, p.V, p.d_v);
    if (tid < 2 * C) {   // beta, then g
      const int i = tid & (C - 1);
      (tid < C ? sb : sg)[i] = i < rows ? (tid < C ? p.beta : p.g)[(size_t)(tok0 + i) * p.H + h] : 0.f;
    }
    cp_wait<WY ? 1 : 0>();
    __syncthreads();
    // ---- Gram matrix and gate: N where i > j, in the blocks on and below the diagonal
    {
      float acc[4][4] = {};
      if (rows <= 16) {   // one block only
        for (int k = 0; k < p.d_k; k += 4) {
          const float4 q = ld4(Ks + ty * LD + k), kv = ld4(Ks + tx * LD + k);
          acc[0][0] = fmaf(q.w, kv.w, fmaf(q.z, kv.z, fmaf(q.y, kv.y, fmaf(q.x, kv.x, acc[0][0]))));
        }
      } else
#pragma unroll 2
      for (int k = 0; k < p.d_k; k += 4) {
        float4 q[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) q[a] = ld4(Ks + (ty + 16 * a) * LD + k);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float4 kv = ld4(Ks + (tx + 16 * b) * LD + k);
#pragma unroll
          for (int a = 0; a < 4; ++a)
            if (a >= b) acc[a][b] = fmaf(q[a].w, kv.w, fmaf(q[a].z, kv.z, fmaf(q[a].y, kv.y, fmaf(q[a].x, kv.x, acc[a][b]))));
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
          const int i = ty + 16 * a, j = tx + 16 * b;
          // select, never multiply an overflowed exp by zero; i > j >= 0, so i - 1 is in the chunk
          M[i * LDM + j] = (j < i && i < rows) ? sb[i] * acc[a][b] * expf(sg[i - gshift] - sg[j]) : 0.f;
        }
    }
    if (WY) cp_wait<0>();
    __syncthreads();
    if (warp < 4) {
      // ---- leaves by forward substitution: 16 x 16, lane = column (Sec. 3.1), in place
      float* blk = M + 16 * warp * LDM + 16 * warp;
      const int j = lane & 15;
      float x[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        float s = 0.f;
#pragma unroll
        for (int k4 = 0; k4 < (i + 3) / 4; ++k4) {
          const float4 n = ld4(blk + i * LDM + 4 * k4);
          if (4 * k4 < i && 4 * k4 >= j) s = fmaf(n.x, x[4 * k4], s);
          if (4 * k4 + 1 < i && 4 * k4 + 1 >= j) s = fmaf(n.y, x[4 * k4 + 1], s);
          if (4 * k4 + 2 < i && 4 * k4 + 2 >= j) s = fmaf(n.z, x[4 * k4 + 2], s);
          if (4 * k4 + 3 < i && 4 * k4 + 3 >= j) s = fmaf(n.w, x[4 * k4 + 3], s);
        }
        x[i] = i < j ? 0.f : (i == j ? 1.f : -s);
      }
      __syncwarp();
      if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) blk[i * LDM + j] = x[i];
      }
    } else if (WY) {
      // ---- meanwhile: row j of K times beta_j (times exp g_j for the decay-weighted W), row j of V times beta_j
      for (int e = tid - 128; e < C * DT / 4; e += 128) {
        const int j = e / (DT / 4), c = 4 * (e % (DT / 4));
        if (j >= rows) break;
        const float b = sb[j], f = (p.ops & kWDecay) ? b * ((gshift && j == 0) ? 1.f : expf(sg[j - gshift])) : b;
        float4* kp = reinterpret_cast<float4*>(Ks + j * LD + c);
        float4* vp = reinterpret_cast<float4*>(Vs + j * LD + c);
        const float4 k = *kp, v = *vp;
        *kp = make_float4(f * k.x, f * k.y, f * k.z, f * k.w);
        *vp = make_float4(b * v.x, b * v.y, b * v.z, b * v.w);
      }
    }
    __syncthreads();
    // ---- merges X21 = -(X22 N21) X11, both products into registers and then over N21 (none where the rows are padding)
    if (rows > 16) {
      // blocks of 16: two pairs, a thread has two neighbouring elements of a row
      const int r0 = 32 * (tid >> 7) + 16, c0 = r0 - 16, i = (tid >> 3) & 15, j = 2 * (tid & 7);
      float* out = M + (r0 + i) * LDM + c0 + j;
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int k4 = 0; k4 < 16; k4 += 4) {
        const float4 x4 = ld4(M + (r0 + i) * LDM + r0 + k4);
        const float x[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 n = *reinterpret_cast<const float2*>(M + (r0 + k4 + q) * LDM + c0 + j);
          if (k4 + q <= i) { s0 = fmaf(x[q], n.x, s0); s1 = fmaf(x[q], n.y, s1); }
        }
      }
      __syncthreads();
      *reinterpret_cast<float2*>(out) = make_float2(s0, s1);
      __syncthreads();
      s0 = s1 = 0.f;
#pragma unroll
      for (int k4 = 0; k4 < 16; k4 += 4) {
        const float4 t4 = ld4(M + (r0 + i) * LDM + c0 + k4);
        const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 x = *reinterpret_cast<const float2*>(M + (c0 + k4 + q) * LDM + c0 + j);
          if (k4 + q >= j) s0 = fmaf(t[q], x.x, s0);
          if (k4 + q >= j + 1) s1 = fmaf(t[q], x.y, s1);
        }
      }
      __syncthreads();
      *reinterpret_cast<float2*>(out) = make_float2(-s0, -s1);
      __syncthreads();
    }
    if (rows > 32) {
      // blocks of 32: one pair, four neighbouring elements of a row
      const int i = tid >> 3, j = 4 * (tid & 7);
      float* out = M + (32 + i) * LDM + j;
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int k4 = 0; k4 < 32; k4 += 4) {
        const float4 x = ld4(M + (32 + i) * LDM + 32 + k4);
        const float* n = M + (32 + k4) * LDM + j;
        const float4 n0 = ld4(n), n1 = ld4(n + LDM), n2 = ld4(n + 2 * LDM), n3 = ld4(n + 3 * LDM);
        if (k4 <= i) fma4(s, x.x, n0);
        if (k4 + 1 <= i) fma4(s, x.y, n1);
        if (k4 + 2 <= i) fma4(s, x.z, n2);
        if (k4 + 3 <= i) fma4(s, x.w, n3);
      }
      __syncthreads();
      *reinterpret_cast<float4*>(out) = make_float4(s[0], s[1], s[2], s[3]);
      __syncthreads();
      s[0] = s[1] = s[2] = s[3] = 0.f;
#pragma unroll 4
      for (int k4 = 0; k4 < 32; k4 += 4) {
        const float4 t = ld4(M + (32 + i) * LDM + k4);
        const float tq[4] = {t.x, t.y, t.z, t.w};
        const float* x = M + k4 * LDM + j;
        if (k4 > j) {
#pragma unroll
          for (int q = 0; q < 4; ++q) fma4(s, tq[q], ld4(x + q * LDM));
        } else if (k4 == j) {   // the rows that the columns' diagonals cross
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 xv = ld4(x + q * LDM);
            s[0] = fmaf(tq[q], xv.x, s[0]);
            if (q >= 1) s[1] = fmaf(tq[q], xv.y, s[1]);
            if (q >= 2) s[2] = fmaf(tq[q], xv.z, s[2]);
            if (q >= 3) s[3] = fmaf(tq[q], xv.w, s[3]);
          }
        }
      }
      __syncthreads();
      *reinterpret_cast<float4*>(out) = make_float4(-s[0], -s[1], -s[2], -s[3]);
      __syncthreads();
    }
    // ---- A: the strict lower part as computed, constants on and above the diagonal
    if ((p.ops & kStoreA) && p.A) {
#pragma unroll
      for (int m = 0; m < C * C / 4 / kThreads; ++m) {
        const int e = tid + m * kThreads, i = e >> 4, j = 4 * (e & 15);
        if (i < rows && TRI_INV_CHECK(p, (long long)tok0 + i < p.n_tokens)) {
          float4 v = ld4(M + i * LDM + j);
          v.x = j < i ? v.x : (j == i ? 1.f : 0.f);
          v.y = j + 1 < i ? v.y : (j + 1 == i ? 1.f : 0.f);
          v.z = j + 2 < i ? v.z : (j + 2 == i ? 1.f : 0.f);
          v.w = j + 3 < i ? v.w : (j + 3 == i ? 1.f : 0.f);
          *reinterpret_cast<float4*>(p.A + ((size_t)(tok0 + i) * p.H + h) * C + j) = v;
        }
      }
    }
    // ---- W = A (scaled K), U = A (scaled V): rows ty + 16 a, four columns
    if constexpr (WY) {
#pragma unroll 1
      for (int part = 0; part < 2 * DT / 64; ++part) {
        const bool second = part >= DT / 64;
        const int c = 64 * (part % (DT / 64)) + 4 * tx, d = second ? p.d_v : p.d_k;
        const float* tile = (second ? Vs : Ks) + c;
        float o[4][4] = {};
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (16 * b >= rows) break;
          const float *t0 = tile + 16 * b * LD, *a0 = M + ty * LDM + 16 * b;
#pragma unroll 2
          for (int j = 0; j < 16; j += 4) {
            const float4 u0 = ld4(t0 + j * LD), u1 = ld4(t0 + (j + 1) * LD), u2 = ld4(t0 + (j + 2) * LD), u3 = ld4(t0 + (j + 3) * LD);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              if (a == b) {
                const float4 v = ld4(a0 + 16 * a * LDM + j);
                if (j <= ty) fma4(o[a], v.x, u0);
                if (j + 1 <= ty) fma4(o[a], v.y, u1);
                if (j + 2 <= ty) fma4(o[a], v.z, u2);
                if (j + 3 <= ty) fma4(o[a], v.w, u3);
              } else if (a > b) {
                const float4 v = ld4(a0 + 16 * a * LDM + j);
                fma4(o[a], v.x, u0); fma4(o[a], v.y, u1); fma4(o[a], v.z, u2); fma4(o[a], v.w, u3);
              }
            }
          }
        }
        float* dst = (float*)(second ? p.U : p.W);
        if (c < d) {
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const int r = ty + 16 * a;
            if (r < rows && TRI_INV_CHECK(p, (long long)tok0 + r < p.n_tokens))
              *reinterpret_cast<float4*>(dst + ((size_t)(tok0 + r) * p.H + h) * d + c) = make_float4(o[a][0], o[a][1], o[a][2], o[a][3]);
          }
        }
      }
    }
  }
}

template <int DT, bool WY>
cudaError_t launch_one(const KParams& p, cudaStream_t stream) {
  const int bytes = F32Cfg<DT>::floats(WY) * (int)sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(f32_factors_kernel<DT, WY>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  const long long total = (long long)p.n_chunks * p.H;
  if (total == 0) return cudaSuccess;
  const int grid = (int)(total < (1 << 20) ? total : (1 << 20));
  return launch_early(f32_factors_kernel<DT, WY>, dim3(grid), kThreads, bytes, stream, p);
}

}  // namespace

bool f32_factors_fit(const KParams& p, int chunk) {
  return p.kv_dtype == TRI_INV_F32 && chunk == C && p.method == (p.method & TRI_INV_GATE_SHIFTED) && !(p.ops & (kLoadA | kRaw | kKda)) && p.d_k <= 128 &&
         (!(p.ops & kDoWY) || (p.V && p.W && p.U && p.d_v <= 128));
}

cudaError_t launch_f32_factors(const KParams& p, cudaStream_t stream) {
  const bool wy = (p.ops & kDoWY) != 0, wide = p.d_k > 64 || (wy && p.d_v > 64);
  if (wide) return wy ? launch_one<128, true>(p, stream) : launch_one<128, false>(p, stream);
  return wy ? launch_one<64, true>(p, stream) : launch_one<64, false>(p, stream);
}

}  // namespace tri_inv

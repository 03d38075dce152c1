// Chunk scan in single precision (fp32 storage, scalar gate, C = 64, d_k <= 128): the chunk form of scan_kernel.cu with
// every product as FFMA on register tiles, in two kernels, so that only what the state depends on runs chunk after chunk:
//   scan_f32_chain    one CTA per (sequence, head, slice of NS value columns) walks the chunks:
//                       U~ = U - W S,   S <- gamma_last S + K^T (exp(g_last - g) U~),
//                     and leaves U~ and the state that ENTERS each chunk in scratch memory.
//   scan_f32_output   one CTA per (sequence, head, chunk, 64 value columns), all chunks at once:
//                       P = (Q K^T) decay,   O = scale (gamma Q S + P U~).
// (Sequences of one chunk take one kernel, scan_f32_one_chunk.)
// The scratch of a call is bounded (kScratchBytes): longer inputs go through in segments of chunks, a pair of launches each,
// the state carried in scratch between them.
//
// What bounds the chain: latency.  Its two products are 64 x NS x d_k and d_k x NS x 64 (32 K FMAs each at 8 columns, d_k = 64);
// a thread holds a 4 x 4 tile of the result for one of KS parts of the summed index and the parts are joined by a
// reduce-scatter of shuffles, so that all 256 threads work on so small a result.  16-byte shared-memory loads (8 per 64 FMAs), the
// eight lanes of a load step in different banks (W and K by their tiles' 128-byte swizzle, S and U~ by padding); W and K come by TMA one
// or two chunks ahead, U and g into registers one chunk ahead; the thread's part of S stays in registers beside its shared copy.
// The output kernel is bound by FFMA issue and shared-memory loads (8 per 64 FMAs).
// Measured (ncu, B = 2, T = 2048, H = 8, d = 64: 16 pairs of 32 chunks): 44 + 27 us (50 + 28 with the chain's tiles by cp.async); 213 us as one kernel per slice of 16 columns that also
// formed P and O on the way (P again in each slice, all of it on the chain, 64 CTAs).
#include "f32_tiles.cuh"
#include "tc_device.cuh"

namespace tri_inv {
namespace {

constexpr int kThreads = 256, kC = 64, kLdP = kC + 4, kNV = 64;   // kNV: value columns of an output CTA
constexpr size_t kScratchBytes = (size_t)128 << 20;

struct F32Args {
  const float *Q, *K, *W, *U;
  int d_k, d_v;
  float* slots;          // per (pair, chunk of the segment): the state that enters the chunk [d_k][d_v], then U~ [64][d_v]
  float* carry;          // per pair: the state between segments [d_k][d_v]; unused with one segment
  int c0, n_seg;         // this segment: chunks c0 .. c0 + n_seg - 1 of every sequence
};
__device__ __forceinline__ size_t slot_floats(const F32Args& a) { return (size_t)(a.d_k + kC) * a.d_v; }

// rows of a [tokens, H, d] tensor into a tile of row length LD; rows past the sequence's end and columns past d become zeros
template <int DK, int LD>
__device__ __forceinline__ void copy_rows(float* dst, const float* src, int tok0, int rows, int H, int h, int d, int tid) {
  constexpr int Q4 = DK / 4;
#pragma unroll
  for (int m = 0; m < kC * Q4 / kThreads; ++m) {
    const int e = tid + m * kThreads, j = e / Q4, c = 4 * (e % Q4);
    const bool ok = j < rows && c < d;
    cp_async16(dst + j * LD + c, src + (ok ? ((size_t)(tok0 + j) * H + h) * d + c : 0), ok);
  }
}

// The sum of v over KS neighbouring lanes, scattered: each lane keeps 16 / KS consecutive ones of the 16 values, from the
// returned index on.
template <int KS>
__device__ __forceinline__ int reduce_scatter(float (&v)[16], int ks) {
  int base = 0;
#pragma unroll
  for (int m = KS / 2, n = 8; m >= 1; m >>= 1, n >>= 1) {
    const bool up = ks & m;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i < n) {
        const float give = up ? v[i] : v[n + i], keep = up ? v[n + i] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, m);
      }
    }
    base += up ? n : 0;
  }
  return base;
}

template <int DK, int NS>
struct Chain {
  static constexpr int BOX = kC * 32;                     // floats in a box of 32 features x 64 tokens, 128-byte swizzle
  static constexpr int NG = NS / 4;                       // groups of four columns
  static constexpr int KA = kThreads / (kC / 4 * NG);     // parts of the summed index: of W S (features) ...
  static constexpr int KB = kThreads / (DK / 4 * NG);     // ... and of K^T U~ (tokens)
  static_assert(KA >= 2 && KB >= 2 && KA <= 8 && KB <= 8, "a tile's parts lie in one warp");
  static constexpr int S_BLK = 4 * NS + (NS == 8 ? 4 : 8);   // four features of S and padding: neighbouring parts in different banks
  static constexpr int LDU = KB == 8 ? 12 : KB == 4 ? 24 : 16;   // row length of the decayed U~, for the same reason
  static_assert(LDU >= NS, "a row of U~");
  static constexpr int kStages = DK == 64 ? 3 : 2;
  static constexpr int TILE = kC * DK;
  static constexpr int floats = kStages * 2 * TILE + (DK / 4) * S_BLK + kC * LDU + 2 * kStages;   // the last: mbarriers
  static_assert(((kStages * 2 * TILE + (DK / 4) * S_BLK + kC * LDU) & 1) == 0, "mbarriers on 8 bytes");
  static constexpr size_t bytes = floats * sizeof(float);
};

template <int DK, int NS>
__global__ void __launch_bounds__(kThreads, DK == 64 ? 2 : 1) scan_f32_chain(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ ScanParams p, const __grid_constant__ F32Args a) {
  using cfg = Chain<DK, NS>;
  constexpr int KA = cfg::KA, KB = cfg::KB, NG = cfg::NG, VA = 16 / KA, VB = 16 / KB;
  extern __shared__ __align__(1024) float sm[];
  const uint32_t bars = smem_u32(sm + cfg::floats - 2 * cfg::kStages);
  float *tiles = sm, *S = sm + cfg::kStages * 2 * cfg::TILE, *Ud = S + (DK / 4) * cfg::S_BLK;
  const int tid = threadIdx.x;
  const int n_slices = (a.d_v + NS - 1) / NS;
  const int slice = blockIdx.x % n_slices, pair = blockIdx.x / n_slices, h = pair % p.H, s = pair / p.H;
  wait_for_predecessor();
  const int beg = p.seq_off ? p.seq_off[s] : s * p.T;
  const int end = p.seq_off ? p.seq_off[s + 1] : (s + 1) * p.T;
  const int n_all = (end - beg + kC - 1) / kC;
  const int n_chunks = n_all - a.c0 < a.n_seg ? n_all - a.c0 : a.n_seg;   // of this segment
  if (n_chunks <= 0 && a.c0 > 0) return;
  const int col0 = slice * NS;
  const size_t state_base = (size_t)pair * a.d_k * a.d_v;

  // this thread's results: VA neighbouring columns of a row of U~, VB neighbouring columns of a feature of S
  const int ka = tid & (KA - 1), cga = (tid / KA) % NG, rg = tid / (KA * NG);
  const int kb = tid & (KB - 1), cgb = (tid / KB) % NG, fg = tid / (KB * NG);
  auto base_of = [](int ks, int KS) {   // as reduce_scatter returns it
    int b = 0;
    for (int m = KS / 2, n = 8; m >= 1; m >>= 1, n >>= 1) b += (ks & m) ? n : 0;
    return b;
  };
  const int ba = base_of(ka, KA), bb = base_of(kb, KB);
  const int row = 4 * rg + ba / 4, ucol = 4 * cga + (ba & 3);       // VA = 2 or 4 columns from ucol on (VA = 8 does not occur)
  const int feat = 4 * fg + bb / 4, scol = 4 * cgb + (bb & 3);      // VB = 8: two features of four columns
  static_assert(VA <= 4 && VB <= 8, "layout of a thread's results");
  const bool ucol_in = col0 + ucol < a.d_v, scol_in = col0 + scol < a.d_v;

  float Sr[VB];
  auto for_state = [&](auto&& f) {   // (value, feature, column of the slice)
#pragma unroll
    for (int i = 0; i < VB; ++i) f(Sr[i], feat + i / 4, VB == 8 ? scol + (i & 3) : scol + i);
  };
  const float* src = a.c0 > 0 ? a.carry : p.S0;
  for_state([&](float& x, int k, int n) { x = (src && k < a.d_k && scol_in) ? src[state_base + (size_t)k * a.d_v + col0 + n] : 0.f; });
  auto put_state = [&](float* dst) {   // to a [d_k][d_v] matrix in global memory
    for_state([&](float& x, int k, int n) { if (k < a.d_k && scol_in) dst[(size_t)k * a.d_v + col0 + n] = x; });
  };
  if (n_chunks <= 0) {
    if (p.S_out) put_state(p.S_out + state_base);
    return;
  }
  auto share_state = [&]() {
    for_state([&](float& x, int k, int n) { S[(k >> 2) * cfg::S_BLK + (k & 3) * NS + n] = x; });
  };
  auto rows_of = [&](int c) { const int left = end - beg - (a.c0 + c) * kC; return left < kC ? left : kC; };
  int requested = -1;   // thread 0: the last chunk whose tiles it asked for
  auto copy_tiles = [&](int c) {   // by one thread; features past d_k are filled with zeros, rows past the sequence's end hold what follows
    requested = c;
    const int st = c % cfg::kStages, tok0 = beg + (a.c0 + c) * kC;
    const uint32_t dst = smem_u32(tiles + st * 2 * cfg::TILE), bar = bars + 8 * st;
    const int boxes = (a.d_k + 31) / 32;
    mbar_expect_tx(bar, 2 * boxes * cfg::BOX * 4);
#pragma unroll
    for (int b = 0; b < DK / 32; ++b) {
      if (b >= boxes) break;
      tma_load_3d(dst + b * cfg::BOX * 4, &tmW, bar, 32 * b, h, tok0);
      tma_load_3d(dst + (cfg::TILE + b * cfg::BOX) * 4, &tmK, bar, 32 * b, h, tok0);
    }
  };
  bool bad = (smem_u32(sm) & 1023u) != 0;   // a wait has run out: this thread walks on without waiting
  if (tid == 0) {
    for (int st = 0; st < cfg::kStages; ++st) mbar_init(bars + 8 * st, 1);
    fence_mbar_init();
    if (!bad)
      for (int c = 0; c < cfg::kStages - 1 && c < n_chunks; ++c) copy_tiles(c);
  }
  // this thread's elements of U and its row's decay exp(g_last - g_row), and gamma_last, of a chunk
  float u_next[VA], g_row, g_last;
  const size_t tok_first = (size_t)(beg + a.c0 * kC);
  const float* u_at = a.U + ((tok_first + row) * p.H + h) * a.d_v + col0 + ucol;
  const float* g_at = p.g + tok_first * p.H + h;
  auto fetch = [&](int c) {
    const int rows = rows_of(c);
#pragma unroll
    for (int i = 0; i < VA; ++i) u_next[i] = (row < rows && ucol_in) ? u_at[i] : 0.f;
    g_row = g_at[(row < rows ? row : rows - 1) * p.H];
    g_last = g_at[(rows - 1) * p.H];
    u_at += (size_t)kC * p.H * a.d_v;
    g_at += (size_t)kC * p.H;
  };
  // where a load step finds its 16 bytes of W (rows 4 rg + q, features 4 ka ..) and of K (token kb, features 4 fg ..) in the swizzled boxes
  int w_at[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) w_at[q] = (4 * rg + q) * 32 + ((ka ^ ((4 * rg + q) & 7)) << 2);
  const int k_at = (fg >> 3) * cfg::BOX + kb * 32, k_chunk = (fg & 7) ^ kb;
  fetch(0);
  share_state();
  float* slot = a.slots + (size_t)pair * a.n_seg * slot_floats(a);
  put_state(slot);
  for (int c = 0; c < n_chunks; ++c) {
    const int rows = rows_of(c);
    const float* Ws = tiles + (c % cfg::kStages) * 2 * cfg::TILE;
    const float* Ks = Ws + cfg::TILE;
    float u[VA];
#pragma unroll
    for (int i = 0; i < VA; ++i) u[i] = u_next[i];
    const float f = expf(g_last - g_row), gl = expf(g_last);
    __syncthreads();   // S in place; the last chunk's tiles have been read (and, before the first chunk, the barriers are initialised)
    if (tid == 0 && c + cfg::kStages - 1 < n_chunks && !bad) copy_tiles(c + cfg::kStages - 1);
    if (c + 1 < n_chunks) fetch(c + 1);
    if (!bad) bad = !mbar_wait_bounded(bars + 8 * (c % cfg::kStages), (uint32_t)(c / cfg::kStages) & 1u, p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs);
    if (rows < kC) {   // the sequence's last chunk: a neighbour's keys must not meet even a zero
      float* kt = tiles + (c % cfg::kStages) * 2 * cfg::TILE + cfg::TILE;
      for (int e = tid; e < (kC - rows) * DK; e += kThreads) kt[(e / 32 % (kC - rows) + rows) * 32 + (e / 32 / (kC - rows)) * cfg::BOX + e % 32] = 0.f;
    }
    // ---- U~ = U - W S
    {
      float acc[4][4] = {};
      const float* s0 = S + ka * cfg::S_BLK + 4 * cga;
#pragma unroll
      for (int i = 0; i < DK / 4 / KA; ++i) {
        if (4 * KA * i >= a.d_k) break;
        // features 4 (ka + KA i) ..: box (ka + KA i) / 8, chunk (ka + KA i) % 8 of its rows
        const float* wb = Ws + (KA * i / 8) * cfg::BOX;
        constexpr int kFlip = KA == 4 ? 16 : 0;
        const int f = (i & 1) * kFlip;
        const float4 x0 = ld4(wb + (w_at[0] ^ f)), x1 = ld4(wb + (w_at[1] ^ f)), x2 = ld4(wb + (w_at[2] ^ f)), x3 = ld4(wb + (w_at[3] ^ f));
        const float* sb = s0 + KA * i * cfg::S_BLK;
        const float4 y0 = ld4(sb), y1 = ld4(sb + NS), y2 = ld4(sb + 2 * NS), y3 = ld4(sb + 3 * NS);
        fma4(acc[0], x0.x, y0); fma4(acc[1], x1.x, y0); fma4(acc[2], x2.x, y0); fma4(acc[3], x3.x, y0);
        fma4(acc[0], x0.y, y1); fma4(acc[1], x1.y, y1); fma4(acc[2], x2.y, y1); fma4(acc[3], x3.y, y1);
        fma4(acc[0], x0.z, y2); fma4(acc[1], x1.z, y2); fma4(acc[2], x2.z, y2); fma4(acc[3], x3.z, y2);
        fma4(acc[0], x0.w, y3); fma4(acc[1], x1.w, y3); fma4(acc[2], x2.w, y3); fma4(acc[3], x3.w, y3);
      }
      float v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = acc[i / 4][i & 3];
      reduce_scatter<KA>(v, ka);
      float* ut = slot + (size_t)a.d_k * a.d_v + (size_t)row * a.d_v + col0 + ucol;
#pragma unroll
      for (int i = 0; i < VA; ++i) {
        const float x = row < rows ? u[i] - v[i] : 0.f;
        if (ucol_in) ut[i] = x;
        Ud[row * cfg::LDU + ucol + i] = x * f;
      }
    }
    __syncthreads();   // U~ in place; S has been read
    // ---- S
    {
      float acc[4][4] = {};
      const float *k0 = Ks + k_at, *u0 = Ud + kb * cfg::LDU + 4 * cgb;
      if (4 * fg < a.d_k)
#pragma unroll 8
      for (int i = 0; i < kC / KB; ++i) {
        // token kb + KB i: its row's chunks are exchanged by its last three bits
        const float4 kv = ld4(k0 + KB * i * 32 + ((k_chunk ^ ((KB * i) & 7)) << 2)), uv = ld4(u0 + KB * i * cfg::LDU);
        fma4(acc[0], kv.x, uv); fma4(acc[1], kv.y, uv); fma4(acc[2], kv.z, uv); fma4(acc[3], kv.w, uv);
      }
      float v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = acc[i / 4][i & 3];
      reduce_scatter<KB>(v, kb);
#pragma unroll
      for (int i = 0; i < VB; ++i) Sr[i] = fmaf(gl, Sr[i], v[i]);
    }
    slot += slot_floats(a);
    if (c + 1 < n_chunks) {
      share_state();
      put_state(slot);
    }
  }
  if (bad) {   // the copies still on their way get a bounded chance to land before the CTA's shared memory is given up
    atomicMax(p.status, TRI_INV_ERR_DEVICE_TIMEOUT);
    if (tid == 0 && (smem_u32(sm) & 1023u) == 0)
      for (int c = requested >= cfg::kStages ? requested - cfg::kStages + 1 : 0; c <= requested; ++c)   // the last of each stage
        mbar_wait_bounded(bars + 8 * (c % cfg::kStages), (uint32_t)(c / cfg::kStages) & 1u, p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs);
  }
  if (a.c0 + n_chunks < n_all) put_state(a.carry + state_base);
  else if (p.S_out) put_state(p.S_out + state_base);
}

template <int DK>
struct Output {
  static constexpr int LD = DK + 4, LDV = kNV + 4;
  static constexpr int P_FLOATS = kC * (kLdP > LD ? kLdP : LD);   // P takes the place of K
  static constexpr int floats = kC * LD + P_FLOATS + DK * LDV + kC * LDV + kC;
  static constexpr size_t bytes = floats * sizeof(float);
};

template <int DK>
__global__ void __launch_bounds__(kThreads, DK == 64 ? 3 : 1) scan_f32_output(ScanParams p, F32Args a) {
  using cfg = Output<DK>;
  constexpr int LD = cfg::LD, LDV = cfg::LDV;
  extern __shared__ __align__(16) float sm[];
  float *Qs = sm, *Ks = Qs + kC * LD, *P = Ks, *Ss = Ks + cfg::P_FLOATS, *Ut = Ss + DK * LDV, *sg = Ut + kC * LDV;
  const int tid = threadIdx.x;
  const int n_slices = (a.d_v + kNV - 1) / kNV;
  const int slice = blockIdx.x % n_slices, at = blockIdx.x / n_slices, lc = at % a.n_seg, pair = at / a.n_seg, h = pair % p.H, s = pair / p.H;
  wait_for_predecessor();
  const int beg = p.seq_off ? p.seq_off[s] : s * p.T;
  const int end = p.seq_off ? p.seq_off[s + 1] : (s + 1) * p.T;
  const int tok0 = beg + (a.c0 + lc) * kC;
  if (tok0 >= end) return;
  const int rows = end - tok0 < kC ? end - tok0 : kC;
  const int col0 = slice * kNV;
  const float* slot = a.slots + (size_t)at * slot_floats(a);

  copy_rows<DK, LD>(Qs, a.Q, tok0, rows, p.H, h, a.d_k, tid);
  copy_rows<DK, LD>(Ks, a.K, tok0, rows, p.H, h, a.d_k, tid);
  cp_commit();
#pragma unroll
  for (int m = 0; m < (DK + kC) * (kNV / 4) / kThreads; ++m) {   // the state [d_k][d_v], then U~ [64][d_v]
    const int e = tid + m * kThreads, k = e / (kNV / 4), n = 4 * (e % (kNV / 4));
    const bool in_state = k < DK, ok = col0 + n < a.d_v && (!in_state || k < a.d_k);
    cp_async16(Ss + k * LDV + n, slot + (ok ? (size_t)(in_state ? k : a.d_k + k - DK) * a.d_v + col0 + n : 0), ok);
  }
  cp_commit();
  if (tid < kC) sg[tid] = p.g[(size_t)(tok0 + (tid < rows ? tid : rows - 1)) * p.H + h];   // rows past the end take the last real row's
  // eight rows and four columns (groups of four columns) per warp: either operand's loads of a step touch 32 different banks
  const int ty = ((tid & 31) >> 2) + 8 * ((tid >> 5) & 1), tx = (tid & 3) + 4 * (tid >> 6);
  cp_wait<1>();
  __syncthreads();
  // ---- P: element (ty, tx) of the ten 16 x 16 blocks on and below the diagonal
  {
    float acc[4][4] = {};
#pragma unroll 2
    for (int k = 0; k < a.d_k; k += 4) {
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
    cp_wait<0>();
    __syncthreads();   // K has been read; S and U~ have landed
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j) {
        const int ri = ty + 16 * i, cj = tx + 16 * j;
        P[ri * kLdP + cj] = cj <= ri ? acc[i][j] * expf(sg[ri] - sg[cj]) : 0.f;
      }
  }
  // ---- O: rows ty + 16 i, four columns
  float o[4][4] = {};
  {
    const float* sc = Ss + 4 * tx;
#pragma unroll 2
    for (int k = 0; k < a.d_k; k += 4) {
      const float4 s0 = ld4(sc + k * LDV), s1 = ld4(sc + (k + 1) * LDV), s2 = ld4(sc + (k + 2) * LDV), s3 = ld4(sc + (k + 3) * LDV);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 q = ld4(Qs + (ty + 16 * i) * LD + k);
        fma4(o[i], q.x, s0); fma4(o[i], q.y, s1); fma4(o[i], q.z, s2); fma4(o[i], q.w, s3);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float gam = expf(sg[ty + 16 * i]);
#pragma unroll
      for (int n = 0; n < 4; ++n) o[i][n] *= gam;
    }
  }
  __syncthreads();   // P in place
#pragma unroll
  for (int b = 0; b < 4; ++b) {   // tokens 16 b .. + 15 of the sum: rows of the blocks i >= b
    const float *uc = Ut + 16 * b * LDV + 4 * tx, *pc = P + ty * kLdP + 16 * b;
#pragma unroll 2
    for (int j = 0; j < 16; j += 4) {
      const float4 u0 = ld4(uc + j * LDV), u1 = ld4(uc + (j + 1) * LDV), u2 = ld4(uc + (j + 2) * LDV), u3 = ld4(uc + (j + 3) * LDV);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i == b) {   // the diagonal's block: a later token's U~ is not multiplied in, not even by zero
          const float4 pv = ld4(pc + 16 * i * kLdP + j);
          if (j <= ty) fma4(o[i], pv.x, u0);
          if (j + 1 <= ty) fma4(o[i], pv.y, u1);
          if (j + 2 <= ty) fma4(o[i], pv.z, u2);
          if (j + 3 <= ty) fma4(o[i], pv.w, u3);
        } else if (i > b) {
          const float4 pv = ld4(pc + 16 * i * kLdP + j);
          fma4(o[i], pv.x, u0); fma4(o[i], pv.y, u1); fma4(o[i], pv.z, u2); fma4(o[i], pv.w, u3);
        }
      }
    }
  }
  if (col0 + 4 * tx < a.d_v) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 16 * i;
      if (r < rows)
        *reinterpret_cast<float4*>((float*)p.O + ((size_t)(tok0 + r) * p.H + h) * a.d_v + col0 + 4 * tx) =
            make_float4(p.scale * o[i][0], p.scale * o[i][1], p.scale * o[i][2], p.scale * o[i][3]);
    }
  }
}

// Sequences of at most one chunk: nothing is walked, so both steps in one kernel, without scratch.  One CTA per (sequence, head, 16 value
// columns).  Measured (graph of calls, B = 1, H = 20, d = 64): 8.8 us, 13.0 as two kernels; T = 1: 7.3 and 12.0.
constexpr int kNS1 = 16, kLdU1 = 24;
template <int DK>
struct OneChunk {
  static constexpr int LD = DK + 4;
  static constexpr int JG = DK == 64 ? 4 : 2;                 // token groups of the state's product: (DK / 4) x 4 x JG threads
  static constexpr int floats = 3 * kC * LD + DK * kNS1 + 2 * kC * kLdU1 + kC * kLdP + kC;
  static constexpr size_t bytes = floats * sizeof(float);
};

template <int DK>
__global__ void __launch_bounds__(kThreads, DK == 64 ? 2 : 1) scan_f32_one_chunk(const __grid_constant__ ScanParams p, const __grid_constant__ F32Args a) {
  using cfg = OneChunk<DK>;
  constexpr int LD = cfg::LD, JG = cfg::JG;
  extern __shared__ __align__(16) float sm[];
  float *Ws = sm, *Qs = Ws + kC * LD, *Ks = Qs + kC * LD, *S = Ks + kC * LD, *Ut = S + DK * kNS1, *Ud = Ut + kC * kLdU1, *P = Ud + kC * kLdU1, *sg = P + kC * kLdP;
  const int tid = threadIdx.x;
  const int n_slices = (a.d_v + kNS1 - 1) / kNS1;
  const int slice = blockIdx.x % n_slices, pair = blockIdx.x / n_slices, h = pair % p.H, s = pair / p.H;
  wait_for_predecessor();
  const int beg = p.seq_off ? p.seq_off[s] : s * p.T;
  const int rows = (p.seq_off ? p.seq_off[s + 1] : (s + 1) * p.T) - beg;   // 0 .. 64
  const int col0 = slice * kNS1;
  const size_t state_base = (size_t)pair * a.d_k * a.d_v;
  if (rows > 0) {
    copy_rows<DK, LD>(Ws, a.W, beg, rows, p.H, h, a.d_k, tid);
    copy_rows<DK, LD>(Qs, a.Q, beg, rows, p.H, h, a.d_k, tid);
    cp_commit();
    copy_rows<DK, LD>(Ks, a.K, beg, rows, p.H, h, a.d_k, tid);
    cp_commit();
    if (tid < kC) sg[tid] = p.g[(size_t)(beg + (tid < rows ? tid : rows - 1)) * p.H + h];   // rows past the end take the last real row's
  }
  // state slice: rows past d_k and columns past d_v stay zero throughout
  for (int e = tid; e < DK * kNS1; e += kThreads) {
    const int k = e / kNS1, n = e % kNS1;
    S[e] = (p.S0 && k < a.d_k && col0 + n < a.d_v) ? p.S0[state_base + (size_t)k * a.d_v + col0 + n] : 0.f;
  }
  if (rows > 0) {
    const int nq = tid & 3, r = tid >> 2;
    const int ty = ((tid & 31) >> 2) + 8 * ((tid >> 5) & 1), tx = (tid & 3) + 4 * (tid >> 6);
    const bool col_in = col0 + 4 * nq < a.d_v;
    const float4 u = (r < rows && col_in) ? ld4(a.U + ((size_t)(beg + r) * p.H + h) * a.d_v + col0 + 4 * nq) : make_float4(0.f, 0.f, 0.f, 0.f);
    cp_wait<1>();
    __syncthreads();
    // ---- W S and Q S: row r, four columns
    float ws[4] = {0.f, 0.f, 0.f, 0.f}, qs[4] = {0.f, 0.f, 0.f, 0.f};
    {
      const float *wr = Ws + r * LD, *qr = Qs + r * LD, *sc = S + 4 * nq;
      if (p.S0)
#pragma unroll 4
      for (int k = 0; k < a.d_k; k += 4) {
        const float4 w = ld4(wr + k), q = ld4(qr + k);
        const float4 s0 = ld4(sc + k * kNS1), s1 = ld4(sc + (k + 1) * kNS1), s2 = ld4(sc + (k + 2) * kNS1), s3 = ld4(sc + (k + 3) * kNS1);
        fma4(ws, w.x, s0); fma4(qs, q.x, s0);
        fma4(ws, w.y, s1); fma4(qs, q.y, s1);
        fma4(ws, w.z, s2); fma4(qs, q.z, s2);
        fma4(ws, w.w, s3); fma4(qs, q.w, s3);
      }
      const float f = expf(sg[rows - 1] - sg[r]);
      float4 t = make_float4(u.x - ws[0], u.y - ws[1], u.z - ws[2], u.w - ws[3]);
      if (r >= rows) t = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(Ut + r * kLdU1 + 4 * nq) = t;
      *reinterpret_cast<float4*>(Ud + r * kLdU1 + 4 * nq) = make_float4(t.x * f, t.y * f, t.z * f, t.w * f);
    }
    cp_wait<0>();
    __syncthreads();
    // ---- P: element (ty, tx) of the 16 x 16 blocks on and below the diagonal
    {
      float acc[4][4] = {};
#pragma unroll 2
      for (int k = 0; k < a.d_k; k += 4) {
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
          P[ri * kLdP + cj] = cj <= ri ? acc[i][j] * expf(sg[ri] - sg[cj]) : 0.f;
        }
    }
    __syncthreads();
    // ---- O
    if (r < rows && col_in) {
      const float gam = expf(sg[r]);
      float o[4] = {gam * qs[0], gam * qs[1], gam * qs[2], gam * qs[3]};
      const float *pr = P + r * kLdP, *uc = Ut + 4 * nq;
      int j = 0;
#pragma unroll 2
      for (; j + 3 <= r; j += 4) {
        const float4 pv = ld4(pr + j);
        fma4(o, pv.x, ld4(uc + j * kLdU1));
        fma4(o, pv.y, ld4(uc + (j + 1) * kLdU1));
        fma4(o, pv.z, ld4(uc + (j + 2) * kLdU1));
        fma4(o, pv.w, ld4(uc + (j + 3) * kLdU1));
      }
      for (; j <= r; ++j) fma4(o, pr[j], ld4(uc + j * kLdU1));
      *reinterpret_cast<float4*>((float*)p.O + ((size_t)(beg + r) * p.H + h) * a.d_v + col0 + 4 * nq) =
          make_float4(p.scale * o[0], p.scale * o[1], p.scale * o[2], p.scale * o[3]);
    }
    // ---- S: four features x four columns, tokens split over JG lanes
    const int jg = tid % JG, n4 = (tid / JG) & 3, kq = tid / (4 * JG);
    float v[16] = {};
#pragma unroll 4
    for (int i = 0; i < kC / JG; ++i) {
      const int j = (i >> 1) * 2 * JG + 2 * jg + (i & 1);   // two neighbouring tokens per lane group: their rows lie in different banks
      const float4 kv = ld4(Ks + j * LD + 4 * kq), uv = ld4(Ud + j * kLdU1 + 4 * n4);
      const float k4[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        v[4 * f] = fmaf(k4[f], uv.x, v[4 * f]); v[4 * f + 1] = fmaf(k4[f], uv.y, v[4 * f + 1]);
        v[4 * f + 2] = fmaf(k4[f], uv.z, v[4 * f + 2]); v[4 * f + 3] = fmaf(k4[f], uv.w, v[4 * f + 3]);
      }
    }
    const int base = reduce_scatter<JG>(v, jg);
    const float gl = expf(sg[rows - 1]);
#pragma unroll
    for (int i = 0; i < 16 / JG; ++i) {
      float* sp = S + (4 * kq + (base + i) / 4) * kNS1 + 4 * n4 + ((base + i) & 3);
      *sp = fmaf(gl, *sp, v[i]);
    }
  }
  if (p.S_out) {
    __syncthreads();
    for (int e = tid; e < DK * kNS1; e += kThreads) {
      const int k = e / kNS1, n = e % kNS1;
      if (k < a.d_k && col0 + n < a.d_v) p.S_out[state_base + (size_t)k * a.d_v + col0 + n] = S[e];
    }
  }
}

template <int DK>
cudaError_t launch_one_chunk(const ScanParams& p, const F32Args& a, cudaStream_t stream) {
  constexpr int bytes = (int)OneChunk<DK>::bytes;
  cudaError_t e = cudaFuncSetAttribute(scan_f32_one_chunk<DK>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  const long long grid = (long long)p.n_seqs * p.H * ((a.d_v + kNS1 - 1) / kNS1);
  if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
  e = launch_early(scan_f32_one_chunk<DK>, dim3((unsigned)grid), kThreads, bytes, stream, p, a);
  return e == cudaSuccess ? launched() : e;
}

template <int DK, int NS>
cudaError_t launch_chain(const CUtensorMap& tmW, const CUtensorMap& tmK, const ScanParams& p, const F32Args& a, long long pairs, cudaStream_t stream) {
  constexpr int bytes = (int)Chain<DK, NS>::bytes;
  cudaError_t e = cudaFuncSetAttribute(scan_f32_chain<DK, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  const long long grid = pairs * ((a.d_v + NS - 1) / NS);
  if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
  e = launch_early(scan_f32_chain<DK, NS>, dim3((unsigned)grid), kThreads, bytes, stream, tmW, tmK, p, a);
  return e == cudaSuccess ? launched() : e;
}

// 3-D view [tokens, H, d] of an fp32 tensor, one box = 32 features (128 bytes, swizzled) of one head x 64 tokens; features past d are
// outside the tensor and read as zeros.
bool make_tmap_heads(CUtensorMap* tm, const float* base, long long tokens, int H, int d) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)H, (cuuint64_t)tokens};
  cuuint64_t strides[2] = {(cuuint64_t)d * 4, (cuuint64_t)H * d * 4};
  cuuint32_t box[3] = {32, 1, (cuuint32_t)kC};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DK>
cudaError_t launch_segments(const ScanParams& p, F32Args a, int max_chunks, long long tokens, cudaStream_t stream) {
  CUtensorMap tmW, tmK;
  if (!make_tmap_heads(&tmW, a.W, tokens, p.H, a.d_k) || !make_tmap_heads(&tmK, a.K, tokens, p.H, a.d_k)) return cudaErrorUnknown;
  constexpr int out_bytes = (int)Output<DK>::bytes;
  cudaError_t e = cudaFuncSetAttribute(scan_f32_output<DK>, cudaFuncAttributeMaxDynamicSharedMemorySize, out_bytes);
  if (e != cudaSuccess) return e;
  const long long pairs = (long long)p.n_seqs * p.H;
  // eight columns a CTA while that is no more than two CTAs for each SM: half the work on the chain; beyond it the wider slice reads
  // W and K half as often
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const bool wide = pairs * ((a.d_v + 7) / 8) > 2 * sms;
  for (a.c0 = 0; a.c0 < max_chunks; a.c0 += a.n_seg) {
    e = wide ? launch_chain<DK, 16>(tmW, tmK, p, a, pairs, stream) : launch_chain<DK, 8>(tmW, tmK, p, a, pairs, stream);
    if (e != cudaSuccess) return e;
    const long long grid = pairs * a.n_seg * ((a.d_v + kNV - 1) / kNV);
    if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
    e = launch_early(scan_f32_output<DK>, dim3((unsigned)grid), kThreads, out_bytes, stream, p, a);
    if (e != cudaSuccess || (e = launched()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

// Chunks per segment and the scratch of a call: slots for every (pair, chunk) of a segment, and the carried state.
size_t chunk_scan_f32_scratch(long long pairs, int max_chunks, int d_k, int d_v, int* n_seg) {
  const size_t slot = (size_t)(d_k + kC) * d_v * sizeof(float), state = (size_t)d_k * d_v * sizeof(float);
  long long n = (long long)(kScratchBytes / (slot * (size_t)pairs));
  n = n < 1 ? 1 : n > max_chunks ? (max_chunks < 1 ? 1 : max_chunks) : n;
  *n_seg = (int)n;
  if (max_chunks <= 1) return 0;
  return (size_t)pairs * ((size_t)n * slot + (n < max_chunks ? state : 0));
}

cudaError_t launch_chunk_scan_f32(const ScanParams& p, const void* Q, const void* K, const void* W, int d_k, int d_v, int max_chunks,
                                  long long tokens, void* scratch, int n_seg, cudaStream_t stream) {
  F32Args a{(const float*)Q, (const float*)K, (const float*)W, (const float*)p.U, d_k, d_v, (float*)scratch, nullptr, 0, n_seg};
  if (max_chunks <= 1) return d_k <= 64 ? launch_one_chunk<64>(p, a, stream) : launch_one_chunk<128>(p, a, stream);
  a.carry = a.slots + (size_t)p.n_seqs * p.H * n_seg * (size_t)(d_k + kC) * d_v;
  return d_k <= 64 ? launch_segments<64>(p, a, max_chunks, tokens, stream) : launch_segments<128>(p, a, max_chunks, tokens, stream);
}

}  // namespace tri_inv

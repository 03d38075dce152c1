// One Gated-DeltaNet layer in one kernel (bf16, d_k = d_v = 128, C = 64, block recursion): build, inversion, W and U of every
// chunk, and the chunk scan that consumes them, side by side.
//
// The scan walks a (sequence, head) pair's chunks one after the other and uses as many SMs as there are pairs (or slices of their
// value columns); the factors of different chunks do not depend on one another.  As two launches the second starts when the
// first has ended, and with few pairs leaves most of the chip idle.  Here a CTA (one per SM, 512 threads) takes one of two roles:
//   factors  four groups of four warps work on a chunk matrix each, as the fused kernel's CTAs do (tc_kernel.cuh): K and V by TMA,
//            Gram product, gate, leaves, merges, W = A diag(beta exp g) K and U = A diag(beta) V; the group's warps then add
//            one each to the chunk's word in `ready` once their stores have completed.  Matrices are numbered in the order in which
//            the scans will want them, chunk by chunk across the pairs that are walked at the same time.
//   scan     scan_walk, whose copy warp waits for a chunk's word before it requests W and U.
// Roles go by SM: the scans have the SMs from a number on to themselves (the two roles' code is too much for the instruction caches
// that neighbouring SMs share: with roles dealt out at random single scans took up to 1.5 times as long while factors were being
// built, and the slowest scan is the kernel's time).  A CTA that scans first builds one matrix (there is nothing to scan yet), and
// goes on building if no factor CTA has come by then; factor CTAs scan when no matrix is left.  Every matrix is drawn by a
// group that is running, and nothing that group does waits for another CTA, so whatever part of the grid is resident (other
// kernels may hold the rest of the SMs, another call of this one among them), the words that a scan waits for are on their
// way.  A CTA scans one task at most, so the grid has one for each: a loop over tasks would keep more in registers than the walk of
// all 128 columns has.  All waits are bounded.
//
// The kernel has every SM, with all of its registers, until the factors are built: a small call on another stream waits that long, which it
// did not behind the fused kernel and the scan as launches of their own.  A decode step of 8 x 16 pairs put on a second stream right behind 32
// pairs x 512 chunks ends after 384 us (behind the two calls 178, alone 25), behind 64 x 64 after 95 us (27, 25); 333 tokens of 16 heads after
// 406 (211, 50) and 111 (106, 50).  The large call itself is the faster one: 566 and 766 us, 150 and 149.  (Before the scan's half products 377 (180), 92 (28), 394 (196) and 108 (114): the
// scans, which are faster now, leave the factors built beside them a smaller share; and a layer kernel whose blocks are placed early takes SMs from the scan that follows the fused call, where it runs with
// more of its blocks on fewer SMs: 199 instead of 211 if it is launched the ordinary way, which costs the call of 333 tokens by itself 2.5 us of 18.)
//
// W and U pass through scratch memory of the call; a scan reads a chunk microseconds after it was written, so mostly from L2.
// Part of scan_kernel.cu, whose scan_walk it calls.
#pragma once
#include <algorithm>
#include <cmath>
#include <mutex>

#include "kda_operands.cuh"

namespace tri_inv {
namespace {

constexpr int kGroups = 4, kLayerThreads = kGroups * 128;
constexpr int kGroupBytes = 51200;     // shared memory of a group
constexpr int OFF_V = 16384, OFF_X = 32768, LDX = C + 4, OFF_AP = OFF_X, OFF_AW = OFF_X + C * C * 2, OFF_BG = OFF_X + C * LDX * 4, OFF_CTL = OFF_BG + 2 * C * 4;
static_assert(OFF_CTL + 64 <= kGroupBytes && kGroupBytes % 1024 == 0 && OFF_X % 1024 == 0 && OFF_AW % 1024 == 0, "a group's tiles");
static_assert(2 * C * C * 2 <= C * LDX * 4, "both operands lie where the matrix was");

struct LayerEntry { int32_t tok0, rows, slot, pad; };   // packed sequences: a chunk of tokens; slot = tok0 / 64 + sequence

struct LayerParams {
  const float *beta, *g;
  __nv_bfloat16 *W, *U;
  const LayerEntry* tab;    // packed sequences, in build order; else null
  uint32_t* ready;          // [slots][H]
  int* counters;            // {arrivals, matrices, scans}
  int* status;
  int H, T, pairs, chunks;  // chunks: per sequence (dense)
  int wave;                 // pairs walked at the same time (dense)
  int total;                // matrices
  int factor_ctas, scan_tasks;   // the first arrivals build factors as long as there are any
  int sms;
  int groups;                    // of these CTAs: four each
  unsigned long long wait_limit_ns;
  int test_stall;           // self-test: the first matrix (per-channel scan: the first chunk) is never announced
};

struct Place { int tok0, rows, h, slot; };
__device__ __forceinline__ Place place_of(const LayerParams& p, int item) {
  int tok0, rows, h, slot;
  if (p.tab) {
    const unsigned e = (unsigned)item / (unsigned)p.H;
    h = (int)((unsigned)item - e * (unsigned)p.H);
    const LayerEntry x = p.tab[e];
    tok0 = x.tok0; rows = x.rows; slot = x.slot;
  } else {
    const unsigned per = (unsigned)p.wave * (unsigned)p.chunks, w = (unsigned)item / per, r = (unsigned)item - w * per;
    const unsigned first = w * (unsigned)p.wave, n = min((unsigned)p.wave, (unsigned)p.pairs - first);
    const unsigned c = r / n, pair = first + (r - c * n), s = pair / (unsigned)p.H;
    h = (int)(pair - s * (unsigned)p.H);
    tok0 = (int)(s * (unsigned)p.T + c * C);
    rows = min(C, p.T - (int)c * C);
    slot = tok0 / C + (int)s;
  }
  return Place{tok0, rows, h, slot};
}

// The matrices of one group: `item` (or, if that is negative, one drawn here), then drawn ones; `once`: only the first.  With more
// matrices than there are groups the next one is drawn while its predecessor is worked on, so that its tiles can come early;
// with fewer that would keep matrices from groups that have none.  False when a wait has run out.
__device__ __forceinline__ bool build_factors(const CUtensorMap& tmK, const CUtensorMap& tmV, const CUtensorMap& tmW, const CUtensorMap& tmU,
                                              const LayerParams& p, uint8_t* sm, uint32_t tmem, int group, int item, bool once) {
  float* sX = reinterpret_cast<float*>(sm + OFF_X);
  float* sBeta = reinterpret_cast<float*>(sm + OFF_BG);
  float* sG = sBeta + C;
  volatile int* s_next = reinterpret_cast<volatile int*>(sm + OFF_CTL + 32);
  volatile int* s_gave_up = s_next + 1;
  int4* s_place = reinterpret_cast<int4*>(sm + OFF_CTL + 48);   // where the drawn matrix lies: one thread's divisions
  const uint32_t sK = smem_u32(sm), sV = sK + OFF_V, sAp = sK + OFF_AP, sAw = sK + OFF_AW;
  const uint32_t bar_k = sK + OFF_CTL, bar_v = bar_k + 8, bar_mma = bar_k + 16, bar_exit = bar_k + 24;
  const int tid = threadIdx.x & 127, warp_u = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5) & 3, 0), warp = warp_u, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const uint32_t tmem_rows = tmem + ((uint32_t)(32 * warp) << 16);
  auto sync = [group]() { asm volatile("bar.sync %0, 128;" ::"r"(group + 1) : "memory"); };
  constexpr int kTidL2 = 32, kTidK = 64, kTidV = 96;
  // Give-up protocol as in tc_kernel.cuh: a thread whose wait has run out goes on without waiting, and the whole group leaves at the
  // top of its next matrix.
  bool bad = false;
  uint32_t n_issue = 0;
  auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
    if (bad) return false;
    bad = !mbar_wait_bounded(bar, parity, p.wait_limit_ns);
    return !bad;
  };
  auto wait_warp = [&](uint32_t bar, uint32_t parity) -> bool {
    wait(bar, parity);
    bad = __any_sync(0xffffffffu, bad);
    return !bad;
  };
  auto issue_tile = [&](uint32_t dst, const CUtensorMap& tm, uint32_t bar, int tok0, int h) {
    if (bad) return;
    ++n_issue;
    fence_proxy_async();
    mbar_expect_tx(bar, 16384u);
    tma_load_2d(dst, &tm, bar, h * D, tok0);
    tma_load_2d(dst + 8192, &tm, bar, h * D + 64, tok0);
  };
  auto fetch_bg = [&](int tok0, int rows, int h) -> float {
    const int i = tid & 63;
    return i < rows ? (tid < C ? p.beta : p.g)[(size_t)(tok0 + i) * p.H + h] : 0.f;
  };
  const int total = p.total;
  const bool ahead = !once && total > p.groups;
  Place at{0, 0, 0, 0}, nx{0, 0, 0, 0};   // of this matrix and the next
  float bg_next = 0.f;
  auto leave = [&](int x) {   // by one thread: a drawn matrix and its place for the group
    *s_next = x;
    if (x < total) {
      const Place q = place_of(p, x);
      *s_place = make_int4(q.tok0, q.rows, q.h, q.slot);
    }
  };
  auto take = [&](Place& q) -> int {   // behind a barrier
    const int4 v = *s_place;
    q = Place{v.x, v.y, v.z, v.w};
    return *s_next;
  };
  auto draw = [&](Place& q, int x) -> int {   // x < 0: from the counter
    if (tid == kTidL2) leave(x < 0 ? atomicAdd(p.counters + 1, 1) : x);
    sync();
    x = take(q);
    sync();
    return x;
  };
  auto start = [&]() {   // the first copies and loads of `item`
    if (tid == kTidK) issue_tile(sK, tmK, bar_k, at.tok0, at.h);
    if (tid == kTidV) issue_tile(sV, tmV, bar_v, at.tok0, at.h);
    bg_next = fetch_bg(at.tok0, at.rows, at.h);
  };
  if (tid == 0) {
    *s_gave_up = 0;
    mbar_init(bar_k, 1);
    mbar_init(bar_v, 1);
    mbar_init(bar_mma, 1);
    mbar_init(bar_exit, 1);
    fence_mbar_init();
  }
  item = draw(at, item);
  if (item < total) start();
  int nx_item = ahead && item < total ? draw(nx, -1) : total;
  uint32_t ph = 0, ph_mma = 0;
  bool gram_early = false;
  auto issue_gram = [&]() {
    constexpr uint32_t idesc = umma_idesc(C, C, 0);
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
      const uint64_t dk = umma_desc(sK + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024);
      umma_bf16(tmem, dk, dk, idesc, ks > 0);
    }
    umma_commit(bar_mma);
  };
  auto issue_wy = [&](uint32_t a_op, uint32_t b_tile) {
    constexpr uint32_t idesc = umma_idesc(C, D, 1);
#pragma unroll
    for (int ks = 0; ks < C / 16; ++ks)
      umma_bf16(tmem, umma_desc(a_op + ks * 32, 16, 1024), umma_desc(b_tile + ks * 2048, 8192, 1024), idesc, ks > 0);
    umma_commit(bar_mma);
  };
  bool partial = false;
  uint32_t* signal = nullptr;   // lane 0 of each warp: the word of the last matrix, whose stores may still be on their way
  auto publish = [&]() {
    if (lane == 0 && signal) {
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // this warp's stores have completed
      if (partial) asm volatile("fence.proxy.async;" ::: "memory");   // rows of a short chunk went out as ordinary stores
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(signal) : "memory");
    }
    signal = nullptr;
  };

  while (item < total) {
    const int tok0 = at.tok0, rows = at.rows, h = at.h;
    // ---- 1. beta and g (times log2 e) of this matrix; the next one's tiles into L2
    sBeta[tid] = bg_next * (tid < C ? 1.f : kLog2e);   // beta, g: adjacent
    const bool has_next = nx_item < total;
    const int nx_tok0 = nx.tok0, nx_rows = nx.rows, nx_h = nx.h;
    if (has_next) {
      const int i = tid & 63;
      if (i < nx_rows) asm volatile("prefetch.global.L2 [%0];" ::"l"((tid < C ? p.beta : p.g) + (size_t)(nx_tok0 + i) * p.H + nx_h));
      if (tid == kTidL2) {
#pragma unroll
        for (int bx = 0; bx < 2; ++bx) {
          tma_prefetch_l2_2d(&tmK, nx_h * D + 64 * bx, nx_tok0);
          tma_prefetch_l2_2d(&tmV, nx_h * D + 64 * bx, nx_tok0);
        }
      }
    }
    if (rows < C) {   // rows past the sequence's end hold a neighbour's tokens (or zero fill): cleared before any product
      wait(bar_k, ph);
      wait(bar_v, ph);
      for (int e = tid; e < (C - rows) * 32; e += 128) {
        const int r = rows + (e >> 5), q = e & 31;   // 8 pieces of 16 bytes in each of the four boxes
        *reinterpret_cast<uint4*>(sm + (q >> 3) * 8192 + r * 128 + (q & 7) * 16) = make_uint4(0, 0, 0, 0);
      }
      fence_proxy_async();
    }
    if (lane == 0) bulk_wait_read();   // this warp's last stores have read their staging tile, which lies in the matrix's space
    if (bad) *s_gave_up = 1;
    sync();
    if (*s_gave_up) break;
    int ticket = 0;
    if (tid == kTidL2 && has_next) ticket = atomicAdd(p.counters + 1, 1);   // the matrix after the next
    // ---- 2. Gram S = K K^T
    if (warp_u == 0 && !gram_early && wait_warp(bar_k, ph)) {
      tc_fence_after();
      issue_gram();
    }
    gram_early = false;
    wait(bar_mma, ph_mma);
    ph_mma ^= 1;
    tc_fence_after();
    // ---- 3. gate and mask on this warp's 16 rows, N -> shared memory
    const int ra = 16 * warp + g, rbw = ra + 8;
    {
      const float ba = sBeta[ra], bb = sBeta[rbw], g_a = sG[ra], g_b = sG[rbw];
      float sacc[8][4];
      tmem_ld_16x64(sacc, tmem_rows);
      tmem_wait_ld();
      float2 gcs[8];   // before the first store to the matrix: a load behind one would wait for it
#pragma unroll
      for (int q = 0; q < 8; ++q) gcs[q] = *reinterpret_cast<const float2*>(sG + 8 * q + 2 * t);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int c = 8 * nt + 2 * t;
        float2 va = make_float2(0.f, 0.f), vb = va;   // blocks above the diagonal: exact zeros
        if (nt / 2 <= warp) {
          va.x = ba * sacc[nt][0] * ex2_approx(g_a - gcs[nt].x);
          va.y = ba * sacc[nt][1] * ex2_approx(g_a - gcs[nt].y);
          vb.x = bb * sacc[nt][2] * ex2_approx(g_b - gcs[nt].x);
          vb.y = bb * sacc[nt][3] * ex2_approx(g_b - gcs[nt].y);
          if (nt / 2 == warp) {
            va.x = (c < ra) ? va.x : 0.f;
            va.y = (c + 1 < ra) ? va.y : 0.f;
            vb.x = (c < rbw) ? vb.x : 0.f;
            vb.y = (c + 1 < rbw) ? vb.y : 0.f;
          }
        }
        *reinterpret_cast<float2*>(sX + ra * LDX + c) = va;
        *reinterpret_cast<float2*>(sX + rbw * LDX + c) = vb;
      }
    }
    __syncwarp();
    // ---- 4. leaves and merges
    leaf_substitution<LDX>(sX + 16 * warp * LDX + 16 * warp, lane);
    sync();
    merge_level<C, 16>(sX, warp, lane, sync);
    merge_level<C, 32>(sX, warp, lane, sync);
    // ---- 5. A' = A diag(beta) and A'' = A diag(beta exp g), bf16 operands over the matrix's space
    {
      float4 xv[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) xv[m] = *reinterpret_cast<const float4*>(sX + ((tid >> 4) + 8 * m) * LDX + 4 * (tid & 15));
      const float4 b = *reinterpret_cast<const float4*>(sBeta + 4 * (tid & 15)), gj = *reinterpret_cast<const float4*>(sG + 4 * (tid & 15));
      const float4 bw = make_float4(b.x * ex2_approx(gj.x), b.y * ex2_approx(gj.y), b.z * ex2_approx(gj.z), b.w * ex2_approx(gj.w));
      if (tid == kTidL2) leave(has_next ? ticket : total);
      tc_fence_before();
      sync();
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int i = (tid >> 4) + 8 * m, j = 4 * (tid & 15);
        const uint32_t off = (uint32_t)(i * 128 + (((j >> 3) ^ (i & 7)) << 4) + (j & 7) * 2);
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(sAp + off), "r"(pack_bf16(xv[m].x * b.x, xv[m].y * b.y)), "r"(pack_bf16(xv[m].z * b.z, xv[m].w * b.w)) : "memory");
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(sAw + off), "r"(pack_bf16(xv[m].x * bw.x, xv[m].y * bw.y)), "r"(pack_bf16(xv[m].z * bw.z, xv[m].w * bw.w)) : "memory");
      }
      fence_proxy_async();
      sync();
    }
    if (has_next) bg_next = fetch_bg(nx_tok0, nx_rows, nx_h);
    // ---- 6. W, then U through the same columns of tensor memory
    if (warp_u == 0 && wait_warp(bar_k, ph)) { tc_fence_after(); issue_wy(sAw, sK); }
    publish();   // the last matrix's stores have long completed, and the release is hidden behind the product
    wait(bar_mma, ph_mma);
    ph_mma ^= 1;
    tc_fence_after();
    const int row0 = 16 * warp, left = rows - row0;
    const size_t stride = (size_t)p.H * D, out = ((size_t)(tok0 + row0) * p.H + h) * D;
    const uint32_t stage = sAw + warp * 2048;   // A'' has been read
    float f0[8][4], f1[8][4];
    tmem_ld_16x64(f0, tmem_rows);
    tmem_ld_16x64(f1, tmem_rows + 64);
    tmem_wait_ld();
    tc_fence_before();
    sync();   // every warp holds its rows of W: U may overwrite the columns
    if (warp_u == 0 && wait_warp(bar_v, ph)) { tc_fence_after(); issue_wy(sAp, sV); }
    if (tid == kTidK && has_next) issue_tile(sK, tmK, bar_k, nx_tok0, nx_h);
    store_frag_piece_bf16(f0, stage, lane, p.W + out, stride, left, &tmW, h * D, tok0 + row0);
    store_frag_piece_bf16(f1, stage, lane, p.W + out + 64, stride, left, &tmW, h * D + 64, tok0 + row0);
    wait(bar_mma, ph_mma);
    ph_mma ^= 1;
    tc_fence_after();
    tmem_ld_16x64(f0, tmem_rows);
    tmem_ld_16x64(f1, tmem_rows + 64);
    tmem_wait_ld();
    tc_fence_before();
    sync();   // tiles, A' and tensor memory are free
    ph ^= 1;
    if (tid == kTidV && has_next) issue_tile(sV, tmV, bar_v, nx_tok0, nx_h);
    if (warp_u == 0 && has_next && nx_rows == C && __all_sync(0xffffffffu, mbar_try_wait(bar_k, ph))) {
      tc_fence_after();
      issue_gram();
      gram_early = true;
    }
    store_frag_piece_bf16(f0, stage, lane, p.U + out, stride, left, &tmU, h * D, tok0 + row0);
    store_frag_piece_bf16<1>(f1, sAp + warp * 2048, lane, p.U + out + 64, stride, left, &tmU, h * D + 64, tok0 + row0);
    partial = rows < C;
    signal = (bad || (p.test_stall && item == 0)) ? nullptr : p.ready + ((size_t)at.slot * p.H + h);
    item = nx_item;
    at = nx;
    nx_item = take(nx);   // left there before the operands' barriers
    if (!ahead) {
      sync();
      // a CTA that scans first builds on only if no other CTA has come to do it
      item = draw(at, once && *(volatile int*)(p.counters + 3) > 0 ? total : -1);
      nx_item = total;
      if (item < total) start();
    }
  }
  publish();
  if (lane == 0) bulk_wait_read();
  if (bad) *s_gave_up = 1;
  sync();
  const bool gave_up = *s_gave_up != 0;
  if (gave_up) {   // what is still in flight gets a bounded chance to finish
    atomicMax(p.status, TRI_INV_ERR_DEVICE_TIMEOUT);
    if (tid == kTidK && n_issue) mbar_wait_bounded(bar_k, (n_issue - 1) & 1, p.wait_limit_ns);
    if (tid == kTidV && n_issue) mbar_wait_bounded(bar_v, (n_issue - 1) & 1, p.wait_limit_ns);
    if (warp_u == 0) { umma_commit(bar_exit); mbar_wait_bounded(bar_exit, 0, p.wait_limit_ns); }
  }
  sync();
  if (tid == 0)
    for (int b = 0; b < 4; ++b) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar_k + 8 * b) : "memory");
  tc_fence_before();
  return !gave_up;
}

template <int DVS>
struct LayerCfg {
  static constexpr int SCAN = ScanCfg<DVS, false>::OFF_BAR + 192, BUILD = kGroups * kGroupBytes;
  static constexpr int SMEM = (SCAN > BUILD ? SCAN : BUILD) + 16;   // + the CTA's own words
};
static_assert(LayerCfg<128>::SMEM <= 232448, "one CTA per SM");

template <int DVS>
__global__ void __launch_bounds__(kLayerThreads, 1)
layer_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
             const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmU,      // boxes of 64 tokens
             const __grid_constant__ CUtensorMap tmWs, const __grid_constant__ CUtensorMap tmUs,    // boxes of 16 tokens: a warp's stores
             const __grid_constant__ CUtensorMap tmO,
             const __grid_constant__ LayerParams p, const __grid_constant__ ScanParams sp) {
  constexpr int NS = D / DVS;
  extern __shared__ __align__(1024) uint8_t smem[];
  int* s_word = reinterpret_cast<int*>(smem + LayerCfg<DVS>::SMEM - 16);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  if (smem_u32(smem) & 1023u) {   // never expected; the swizzle pattern would not match the copies
    if (threadIdx.x == 0) atomicMax(p.status, TRI_INV_ERR_DEVICE_TIMEOUT);
    return;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_word + 1)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  wait_for_predecessor();
  if (threadIdx.x == 32) {
    s_word[2] = atomicAdd(p.counters + 1, 1);   // the first group's first matrix: with few of them, one per CTA
    *s_word = atomicAdd(p.counters, 1);
    prefetch_tmap(&tmK); prefetch_tmap(&tmV); prefetch_tmap(&tmWs); prefetch_tmap(&tmUs);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_word[1], 0);
  const int arrival = __shfl_sync(0xffffffffu, *s_word, 0);
  const int group = warp >> 2;
  unsigned smid;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
  const bool scans_first = arrival >= p.sms || (int)smid >= p.factor_ctas;
  if (!scans_first && threadIdx.x == 0) atomicAdd(p.counters + 3, 1);
  bool ok = true;
  if (!scans_first || group == 0)
    ok = build_factors(tmK, tmV, tmWs, tmUs, p, smem + group * kGroupBytes, tmem + 128 * group, group, group == 0 ? s_word[2] : -1, scans_first);
  fence_proxy_async();   // what this thread wrote to or read from shared memory comes before the scans' copies into it
  ok = __syncthreads_and(ok);
  tc_fence_after();
  if (threadIdx.x == 0) *s_word = ok ? atomicAdd(p.counters + 2, 1) : p.scan_tasks;
  __syncthreads();
  const int task = __shfl_sync(0xffffffffu, *s_word, 0);
  if (task < p.scan_tasks) {
    const int slice = task % NS, pair = task / NS;
    scan_walk<DVS, false, true>(tmW, tmQ, tmK, tmU, tmO, sp, smem, pair / p.H, pair % p.H, slice, false, p.ready, tmem);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ---------------------------------------------------------------- the per-channel scan beside the preparation of its operands
// The same split of the chip for tri_inv_chunk_scan_kda: instead of matrices the groups prepare chunks (Q+, K- and the three vectors,
// as kda_scan_prep_kernel does: kda_operands.cuh), bound by the bytes they move.
struct KdaOperands {
  const __nv_bfloat16 *Q, *K;
  const float* G;
  __nv_bfloat16 *Qp, *Km;   // [slots][64][H][128]
  float *EL, *ER, *EX;
};

// The chunks of one group, drawn one ahead; `once`: one, and more only if no other CTA has come to prepare them.
__device__ __forceinline__ void prepare_chunks(const LayerParams& p, const KdaOperands& a, int4* words, int group, bool once) {
  const int tid = threadIdx.x & 127, r0 = tid >> 4, f0 = 8 * (tid & 15);
  auto sync = [group]() { asm volatile("bar.sync %0, 128;" ::"r"(group + 1) : "memory"); };
  int turn = 0;   // two slots in turn: a slow thread may still read the one while the next draw is left in the other
  auto leave = [&](int x) {
    Place q{0, 0, 0, 0};
    if (x < p.total) q = place_of(p, x);
    words[2 * (turn & 1)] = make_int4(q.tok0, q.rows, q.h, q.slot);
    words[2 * (turn & 1) + 1].x = x;
  };
  auto take = [&](Place& q) -> int {
    const int4 v = words[2 * (turn & 1)];
    q = Place{v.x, v.y, v.z, v.w};
    const int x = words[2 * (turn & 1) + 1].x;
    ++turn;
    return x;
  };
  Place at, nx;
  if (tid == 0) leave(atomicAdd(p.counters + 1, 1));
  sync();
  int item = take(at);
  if (tid == 0) leave(once ? p.total : atomicAdd(p.counters + 1, 1));
  sync();
  int nx_item = take(nx);
  while (item < p.total) {
    int ticket = p.total;
    // (one thread decides for the group: it reads a word that other CTAs write)
    if (tid == 0 && (nx_item < p.total || (once && *(volatile int*)(p.counters + 3) == 0))) ticket = atomicAdd(p.counters + 1, 1);
    const size_t row0 = ((size_t)at.tok0 * p.H + at.h) * D + f0, stride = (size_t)p.H * D, out0 = ((size_t)at.slot * C * p.H + at.h) * D + f0;
    DecayRefs refs;
    load_decay_row(refs.ref, a.G + row0 + (size_t)(at.rows >> 1) * stride);
    if (r0 == 0) {   // the chunk's vectors, ahead of the rows: with the last row's values kept beside the rows of the loop, 128 registers are not enough (48 to 84 bytes spilled; 56 pairs x 256 chunks 493 -> 471 us, 37 x 256 376 -> 364)
      const size_t v = ((size_t)at.slot * p.H + at.h) * D + f0;
      load_decay_row(refs.last, a.G + row0 + (size_t)(at.rows - 1) * stride);
      store_decay_vectors(a.EL + v, a.ER + v, a.EX + v, refs);
    }
#pragma unroll 1
    for (int r4 = r0; r4 < at.rows; r4 += 32) {
      // four rows' loads first, without a branch between them (rows past the chunk: the last one again)
      uint4 qv[4], kv[4];
      float4 gv[4][2];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const size_t idx = row0 + (size_t)min(r4 + 8 * m, at.rows - 1) * stride;
        qv[m] = *reinterpret_cast<const uint4*>(a.Q + idx);
        kv[m] = *reinterpret_cast<const uint4*>(a.K + idx);
        gv[m][0] = *reinterpret_cast<const float4*>(a.G + idx);
        gv[m][1] = *reinterpret_cast<const float4*>(a.G + idx + 4);
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        uint4 qo, ko;
        decay_operands(qv[m], kv[m], gv[m][0], gv[m][1], refs, qo, ko);
        if (r4 + 8 * m < at.rows) {
          const size_t idx = out0 + (size_t)(r4 + 8 * m) * stride;
          *reinterpret_cast<uint4*>(a.Qp + idx) = qo;
          *reinterpret_cast<uint4*>(a.Km + idx) = ko;
        }
      }
    }
    // the scan's state product multiplies the rows past the sequence's end by zeros, and may not find Inf or NaN there
    for (int r = at.rows + r0; r < C; r += 8) *reinterpret_cast<uint4*>(a.Km + out0 + (size_t)r * stride) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async;" ::: "memory");   // ordinary stores, read by the scans' tile copies
    if (tid == 0) leave(ticket);
    sync();
    if (tid == 0 && !(p.test_stall && item == 0)) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p.ready + ((size_t)at.slot * p.H + at.h)), "r"(kReady) : "memory");
    item = nx_item;
    at = nx;
    nx_item = take(nx);
    if (once && item >= p.total) {   // not one ahead: the chunk just drawn, if any, is the next
      item = nx_item;
      at = nx;
      nx_item = p.total;
    }
  }
}

// as many threads as the walk has warps; every four of them prepare as a group (the fourth: 313 -> 306 us at 32 pairs x 256 chunks)
constexpr int kKdaThreads = kThreadsScan, kKdaGroups = kKdaThreads / 128;
template <int DVS>
struct KdaScanCfg {
  static constexpr int OFF_WORDS = (ScanCfg<DVS, true>::OFF_BAR + 192 + 15) / 16 * 16;
  static constexpr int SMEM = OFF_WORDS + kKdaGroups * 64 + 16;
};
static_assert(KdaScanCfg<128>::SMEM <= 232448, "one CTA per SM");

template <int DVS>
__global__ void __launch_bounds__(kKdaThreads, 1)
kda_scan_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmW,
                const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmO, const __grid_constant__ LayerParams p, const __grid_constant__ KdaOperands a,
                const __grid_constant__ ScanParams sp) {
  constexpr int NS = D / DVS;
  extern __shared__ __align__(1024) uint8_t smem[];
  int* s_word = reinterpret_cast<int*>(smem + KdaScanCfg<DVS>::SMEM - 16);
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_word + 1)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  wait_for_predecessor();
  if (threadIdx.x == 32) *s_word = atomicAdd(p.counters, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_word[1], 0);
  const int arrival = __shfl_sync(0xffffffffu, *s_word, 0);
  unsigned smid;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
  const bool scans_first = arrival >= p.sms || (int)smid >= p.factor_ctas;
  if (!scans_first && threadIdx.x == 0) atomicAdd(p.counters + 3, 1);
  if (warp < 4 * kKdaGroups)
    prepare_chunks(p, a, reinterpret_cast<int4*>(smem + KdaScanCfg<DVS>::OFF_WORDS) + 4 * (warp >> 2), warp >> 2, scans_first);
  __syncthreads();
  if (threadIdx.x == 0) *s_word = atomicAdd(p.counters + 2, 1);
  __syncthreads();
  const int task = __shfl_sync(0xffffffffu, *s_word, 0);
  if (task < p.scan_tasks) {
    const int slice = task % NS, pair = task / NS;
    scan_walk<DVS, true, true>(tmW, tmQ, tmK, tmU, tmO, sp, smem, pair / p.H, pair % p.H, slice, false, p.ready, tmem);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// Before the layer kernel: its words at zero, and for packed sequences the chunks in build order and the device copy of cu_seqlens.
// Sequences go in groups of `group` (those walked at the same time), and within a group chunk by chunk.
constexpr int kMostSeqs = 960;   // packed sequences of a call: their offsets are kernel parameters
struct PrepArgs {
  uint32_t* words;
  long long n_words;
  LayerEntry* tab;
  int* seq_off;
  int n, group;
  int32_t cu[kMostSeqs + 1];
};
__global__ void __launch_bounds__(256) layer_prep_kernel(const __grid_constant__ PrepArgs a) {
  let_successor_start();
  wait_for_predecessor();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < a.n_words; i += (long long)gridDim.x * blockDim.x) a.words[i] = 0u;
  auto chunks = [&](int s) { return (a.cu[s + 1] - a.cu[s] + C - 1) / C; };
  __shared__ int part[8];
  for (int s = blockIdx.x; s < a.n; s += gridDim.x) {
    const int g0 = s / a.group * a.group, g1 = min(g0 + a.group, a.n);
    int sum = 0;
    for (int q = threadIdx.x; q < g0; q += blockDim.x) sum += chunks(q);
    for (int m = 16; m >= 1; m >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, m);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    int base = 0;
    for (int q = 0; q < 8; ++q) base += part[q];
    const int len = a.cu[s + 1] - a.cu[s], n = chunks(s);
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      int at = base;
      for (int q = g0; q < g1; ++q) {
        const int nq = chunks(q);
        at += min(nq, c) + (q < s && nq > c ? 1 : 0);
      }
      const int tok0 = a.cu[s] + c * C;
      a.tab[at] = LayerEntry{tok0, min(C, len - c * C), tok0 / C + s, 0};
    }
    if (threadIdx.x == 0) {
      a.seq_off[s] = a.cu[s];
      if (s == a.n - 1) a.seq_off[a.n] = a.cu[a.n];
    }
  }
}

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

struct Layout { size_t words, tab, seq, w, u, bytes; long long n_words, entries; };
Layout layout_of(const tri_inv_desc* d) {
  Layout l{};
  const long long tokens = d->cu_seqlens ? (long long)d->T : (long long)d->B * d->T, seqs = d->cu_seqlens ? d->n_seqs : d->B;
  l.n_words = 64 + (tokens / C + seqs + 1) * d->H;
  if (d->cu_seqlens)
    for (int s = 0; s < d->n_seqs; ++s) l.entries += (d->cu_seqlens[s + 1] - d->cu_seqlens[s] + C - 1) / C;
  else
    l.entries = seqs * ((d->T + C - 1) / C);
  size_t at = 0;
  l.words = at; at = align_up(at + (size_t)l.n_words * 4);
  l.tab = at; if (d->cu_seqlens) at = align_up(at + (size_t)l.entries * sizeof(LayerEntry));
  l.seq = at; if (d->cu_seqlens) at = align_up(at + (size_t)(seqs + 1) * 4);
  const size_t tensor = align_up((size_t)tokens * d->H * D * 2);
  l.w = at; at += tensor;
  l.u = at; at += tensor;
  l.bytes = at;
  return l;
}

// Which slices and how many CTAs for the scans, and whether this kernel is the better form at all: predicted times in us, from
// what was measured with each form and width forced (back to back; pairs x chunks: two calls / here in slices of 32, 64, 128 columns):
//   16 x 64: 82 / 78, 82, 109    32 x 64: 100 / -, 85, 109    48 x 64: 125 / -, 129, 116    64 x 64: 151 / -, -, 132    75 x 64: 176 / -, -, 167
//   100 x 64: 213 / -, -, 276    8 x 512: 527 / 478, 505, 704    32 x 512: 728 / -, 592, 718    64 x 256: 583 / -, -, 486    32 x 6: 19.7 / -, 21.0, 24
//   (before the scan's half products: 1024 x up to 32 chunks: 502 / 525; since: 474 / 503 .. 657 with 48 .. 96 SMs that scan)
// (Since kernels start early the two calls are also the faster form of short calls that the predictions leave here: 64 x 2 15.8 and 17.2 us, 64 x 16 42 and 46, 48 x 24 51 and 57, 16 x 6 17.2 and 17.8.)
// A scan here takes 1.56, 1.02 or 0.9 us a chunk in slices of 128, 64 or 32 columns (1.3, 0.98, 0.93 with the chip to itself), an SM
// builds half a matrix per us.  More tasks than scan CTAs never paid, but for the few matrices of a call that is all latency:
// both parts are then bound by bytes and power, which side by side save nothing.
struct Split { int dvs, scans; };   // scans 0: two launches
Split choose_split(long long pairs, int longest, long long entries, int H, int sms) {
  const struct { int dvs; float start_us, here_us, alone_us; } width[3] = {{128, 18.2f, 1.56f, 1.3f}, {64, 15.f, 1.02f, 0.98f}, {32, 15.f, 0.9f, 0.93f}};
  const float items = (float)entries * (float)H;
  const auto& alone = width[pairs * 8 <= sms ? 2 : pairs * 2 <= sms ? 1 : 0];
  const float waves = std::max(1.f, std::ceil((float)pairs / (float)sms)), mean = pairs > 0 ? items / (float)pairs : 0.f;
  float best_us = 18.f + items / (0.55f * (float)sms) + std::max((float)longest * alone.alone_us, waves > 1.f ? waves * (4.f + mean * alone.alone_us) : 0.f);
  Split best{0, 0};
  for (const auto& w : width) {
    const long long tasks = pairs * (D / w.dvs);
    const bool few = w.dvs == 128 && items <= (float)(kGroups * sms) && tasks <= sms;
    if (tasks > sms * 3 / 4 && !few) continue;
    const int n = (int)std::min<long long>(tasks, sms * 3 / 4);
    const float start_us = items <= (float)(kGroups * sms) ? 15.f : w.start_us;   // (where every matrix has a group at once)
    const float us = std::max(start_us + (float)longest * w.here_us, 12.f + items / (0.5f * (float)(sms - n)));
    if (us < best_us) { best_us = us; best = Split{w.dvs, n}; }
  }
  return best;
}

// The same for the per-channel scan, each form and width forced, back to back on three sets of inputs; two launches / here in slices of 32, 64, 128 columns:
//   16 x 32: 40.8 / 48.0, 51, 66    16 x 64: 79 / 81, 87, 116    16 x 96: 115 / 110, 119, 162    8 x 128: 135 / 137, 149, 205    8 x 512: 520 / 488, 532, 752
//   24 x 64: 93 / 84, 89, 116    32 x 16: 28.6 / -, 35.9, 44    32 x 32: 54 / -, 57, 71    32 x 48: 78 / -, 74, 93    32 x 64: 99 / -, 92, 116    32 x 512: 764 / -, 649, 761
//   40 x 64: 109 / -, 113, 117    40 x 256: 430 / -, 431, 412    48 x 64: 121 / -, 156, 121    48 x 128: 241 / -, 307, 226    56 x 64: 134 / -, -, 138
//   56 x 256: 531 / -, -, 508    64 x 64: 148 / -, -, 159    64 x 256: 581 / -, -, 596    75 x 64: 181 / -, -, 199    100 x 128: 433 / -, -, 704    16 x 6: 17.3 / 19.6, 20, 24
// (of 60 such points the predictions miss the faster form in three, by 1.6 % at most)
// Two launches: the preparation takes 79 chunks a us, a scan 0.95, 1.07 or 1.8 us a chunk at its own widths (launch_chunk_scan), in slices of 64 columns more with each pair beyond 32: bytes
// and power.  Here: 0.89, 1.02 or 1.41 us a chunk, and an SM's four groups prepare 0.39 chunks a us (0.36 beside slices of 128), all of them 25.5 (28.5) at most: a group's chunk is a
// chain of latencies of about 9 us, so the gain is where the scan's chain is long.
Split choose_kda_split(long long pairs, int longest, long long entries, int H, int sms) {
  const struct { int dvs; float start_us, here_us, per_sm, most; } width[3] = {{128, 27.f, 1.41f, 0.36f, 28.5f}, {64, 23.f, 1.02f, 0.39f, 25.5f}, {32, 20.f, 0.89f, 0.39f, 25.5f}};
  const float items = (float)entries * (float)H;
  const float alone_us = pairs * 8 <= sms ? 0.95f : pairs * 2 <= sms ? 1.07f + 0.0115f * (float)std::max(0LL, pairs - 32) : 1.8f;
  float best_us = 3.f + items / 79.f + (float)longest * alone_us;   // (only compared where all scans run at the same time)
  Split best{0, 0};
  for (const auto& w : width) {
    const long long tasks = pairs * (D / w.dvs);
    if (tasks > sms * 3 / 4) continue;
    const float us = std::max(w.start_us + (float)longest * w.here_us, 12.f + items / std::min(w.per_sm * (float)(sms - tasks), w.most));
    if (us < best_us) { best_us = us; best = Split{w.dvs, (int)tasks}; }
  }
  return best;
}

int longest_of(const tri_inv_desc* d) {
  int n = d->T;
  if (d->cu_seqlens) {
    n = 0;
    for (int s = 0; s < d->n_seqs; ++s) n = std::max(n, d->cu_seqlens[s + 1] - d->cu_seqlens[s]);
  }
  return (n + C - 1) / C;
}

Split split_of(const tri_inv_desc* d, const Layout& l, int sms) {
  return choose_split((long long)(d->cu_seqlens ? d->n_seqs : d->B) * d->H, longest_of(d), l.entries, d->H, sms);
}

// What both kernels' roles go by.
void fill_params(LayerParams& p, const tri_inv_desc* d, const Layout& l, char* ws, const ScanParams& sp, const Split& split, int sms) {
  p.counters = reinterpret_cast<int*>(ws + l.words);
  p.ready = reinterpret_cast<uint32_t*>(ws + l.words) + 64;
  p.status = sp.status;
  p.H = d->H; p.T = d->T;
  p.pairs = sp.n_seqs * d->H;
  p.chunks = (d->T + C - 1) / C;
  p.total = (int)(l.entries * d->H);
  p.wait_limit_ns = sp.wait_limit_ns ? sp.wait_limit_ns : kWaitLimitNs;
  p.test_stall = sp.test_stall;
  p.factor_ctas = sms - split.scans;
  p.sms = sms;
  p.groups = kGroups * p.factor_ctas;
  p.scan_tasks = p.pairs * (D / split.dvs);
  p.wave = std::max(1, split.scans / (D / split.dvs));
}

// The words, the table and the offsets of a call's workspace (the last two for packed sequences); p.tab and sp.seq_off point to them.
cudaError_t launch_prep(const tri_inv_desc* d, const Layout& l, char* ws, int sms, LayerParams& p, ScanParams& sp, cudaStream_t stream) {
  PrepArgs a;
  a.words = reinterpret_cast<uint32_t*>(p.counters);
  a.n_words = l.n_words;
  a.tab = nullptr; a.seq_off = nullptr; a.n = 0; a.group = 1;
  int blocks = (int)std::min<long long>(sms, (l.n_words + 255) / 256);
  if (d->cu_seqlens) {
    p.tab = a.tab = reinterpret_cast<LayerEntry*>(ws + l.tab);
    sp.seq_off = a.seq_off = reinterpret_cast<int*>(ws + l.seq);
    a.group = std::max(1, (p.wave + d->H - 1) / d->H);
    a.n = d->n_seqs;
    for (int q = 0; q <= a.n; ++q) a.cu[q] = d->cu_seqlens[q];
    blocks = std::max(blocks, std::min(a.n, sms));
  }
  return launch_early(layer_prep_kernel, dim3(blocks), 256, 0, stream, a);
}

template <int DVS>
cudaError_t launch_width(const CUtensorMap (&tm)[7], const LayerParams& p, const ScanParams& sp, long long tokens, int grid, int dev, cudaStream_t stream) {
  static std::mutex mu;
  static bool ready[64] = {false};
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!ready[dev]) {
      cudaError_t e;
      if ((e = cudaFuncSetAttribute(layer_kernel<DVS>, cudaFuncAttributeMaxDynamicSharedMemorySize, LayerCfg<DVS>::SMEM)) != cudaSuccess) return e;
      if ((e = cudaFuncSetAttribute(layer_kernel<DVS>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared)) != cudaSuccess) return e;
      ready[dev] = true;
    }
  }
  CUtensorMap tmO;
  if (!make_tmap_out<DVS>(&tmO, sp.O, tokens, p.H)) return cudaErrorUnknown;
  const cudaError_t e = launch_early(layer_kernel<DVS>, dim3(grid), kLayerThreads, LayerCfg<DVS>::SMEM, stream, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], tmO, p, sp);
  return e == cudaSuccess ? launched() : e;
}

}  // namespace

bool layer_fits(const tri_inv_desc* d, size_t* workspace_bytes) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
  const Layout l = layout_of(d);
  if (l.entries * d->H > 0x7fffffffLL || d->n_seqs > kMostSeqs || split_of(d, l, sms).scans == 0) return false;   // matrices are numbered in 32 bits
  *workspace_bytes = l.bytes;
  return true;
}

cudaError_t launch_layer(const void* Q, const void* K, const void* V, const float* beta, const float* g, const ScanParams& scan,
                         void* workspace, const tri_inv_desc* d, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const Layout l = layout_of(d);
  char* ws = reinterpret_cast<char*>(workspace);
  const long long tokens = std::max(1LL, d->cu_seqlens ? (long long)d->T : (long long)d->B * d->T);
  ScanParams sp = scan;
  LayerParams p{};
  p.beta = beta; p.g = g;
  p.W = reinterpret_cast<__nv_bfloat16*>(ws + l.w); p.U = reinterpret_cast<__nv_bfloat16*>(ws + l.u);
  sp.U = p.U;
  const Split split = split_of(d, l, sms);
  if (split.scans == 0) return cudaErrorInvalidValue;
  fill_params(p, d, l, ws, sp, split, sms);

  CUtensorMap tm[7];
  if (!make_tmap(&tm[0], Q, tokens, d->H, D, C) || !make_tmap(&tm[1], K, tokens, d->H, D, C) || !make_tmap(&tm[2], V, tokens, d->H, D, C) ||
      !make_tmap(&tm[3], p.W, tokens, d->H, D, C) || !make_tmap(&tm[4], p.U, tokens, d->H, D, C) ||
      !make_tmap(&tm[5], p.W, tokens, d->H, D, 16) || !make_tmap(&tm[6], p.U, tokens, d->H, D, 16))
    return cudaErrorUnknown;

  if ((e = launch_prep(d, l, ws, sms, p, sp, stream)) != cudaSuccess) return e;
  const int grid = std::max(sms, p.scan_tasks);   // a CTA walks once
  switch (split.dvs) {
    case 32: return launch_width<32>(tm, p, sp, tokens, grid, dev, stream);
    case 64: return launch_width<64>(tm, p, sp, tokens, grid, dev, stream);
    default: return launch_width<128>(tm, p, sp, tokens, grid, dev, stream);
  }
}

bool kda_scan_fits(const tri_inv_desc* d, size_t* control_bytes) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
  const Layout l = layout_of(d);
  if (l.entries * d->H > 0x7fffffffLL || d->n_seqs > kMostSeqs || choose_kda_split((long long)(d->cu_seqlens ? d->n_seqs : d->B) * d->H, longest_of(d), l.entries, d->H, sms).scans == 0)
    return false;
  *control_bytes = l.w;
  return true;
}

namespace {
template <int DVS>
cudaError_t launch_kda_width(const CUtensorMap (&tm)[4], const LayerParams& p, const KdaOperands& a, const ScanParams& sp, long long tokens, int grid, int dev, cudaStream_t stream) {
  static std::mutex mu;
  static bool ready[64] = {false};
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!ready[dev]) {
      cudaError_t e;
      if ((e = cudaFuncSetAttribute(kda_scan_kernel<DVS>, cudaFuncAttributeMaxDynamicSharedMemorySize, KdaScanCfg<DVS>::SMEM)) != cudaSuccess) return e;
      if ((e = cudaFuncSetAttribute(kda_scan_kernel<DVS>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared)) != cudaSuccess) return e;
      ready[dev] = true;
    }
  }
  CUtensorMap tmO;
  if (!make_tmap_out<DVS>(&tmO, sp.O, tokens, p.H)) return cudaErrorUnknown;
  const cudaError_t e = launch_early(kda_scan_kernel<DVS>, dim3(grid), kKdaThreads, KdaScanCfg<DVS>::SMEM, stream, tm[0], tm[1], tm[2], tm[3], tmO, p, a, sp);
  return e == cudaSuccess ? launched() : e;
}
}  // namespace

cudaError_t launch_kda_scan(const ScanParams& scan, const void* Q, const void* K, const void* W, void* Qp, void* Km, void* control,
                            const tri_inv_desc* d, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const Layout l = layout_of(d);
  char* ws = reinterpret_cast<char*>(control);
  ScanParams sp = scan;
  LayerParams p{};
  const Split split = choose_kda_split((long long)sp.n_seqs * d->H, longest_of(d), l.entries, d->H, sms);
  if (split.scans == 0) return cudaErrorInvalidValue;
  fill_params(p, d, l, ws, sp, split, sms);
  const KdaOperands a{(const __nv_bfloat16*)Q, (const __nv_bfloat16*)K, sp.G, (__nv_bfloat16*)Qp, (__nv_bfloat16*)Km,
                      const_cast<float*>(sp.EL), const_cast<float*>(sp.ER), const_cast<float*>(sp.EX)};
  const long long tokens = d->cu_seqlens ? (long long)d->T : (long long)d->B * d->T, rows = (tokens / C + sp.n_seqs + 1) * C;
  CUtensorMap tm[4];
  if (!make_tmap(&tm[0], Qp, rows, d->H, D, C) || !make_tmap(&tm[1], Km, rows, d->H, D, C) || !make_tmap(&tm[2], W, tokens, d->H, D, C) ||
      !make_tmap(&tm[3], sp.U, tokens, d->H, D, C))
    return cudaErrorUnknown;
  if ((e = launch_prep(d, l, ws, sms, p, sp, stream)) != cudaSuccess) return e;
  const int grid = std::max(sms, p.scan_tasks);
  switch (split.dvs) {
    case 32: return launch_kda_width<32>(tm, p, a, sp, tokens, grid, dev, stream);
    case 64: return launch_kda_width<64>(tm, p, a, sp, tokens, grid, dev, stream);
    default: return launch_kda_width<128>(tm, p, a, sp, tokens, grid, dev, stream);
  }
}

}  // namespace tri_inv

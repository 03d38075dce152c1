// Chunk scan: the consumer of W and U.  The chunk form of the layer's recurrence (the re-formulation that
// Sec. 1 refers to; (I+N)^{-1} enters through W and U), per sequence and head, chunk after chunk, with the
// state S [d_k x d_v] carried in registers:
//
//     U~ = U - W S                                   W = A diag(beta exp g) K (decay-weighted), U = A diag(beta) V
//     O  = scale * (diag(gamma) Q S + P U~)          gamma_i = exp(g_i),  P_ij = (q_i . k_j) gamma_i / gamma_j  (j <= i)
//     S <- gamma_last S + K^T diag(gamma_last / gamma) U~
//
// Columns of S (the d_v axis) never mix, so a CTA owns one (sequence, head, slice of DVS value columns) and walks
// the chunks in order.
//
// Everything that carries the state is kept transposed, value columns as rows: a row is a tensor-memory lane, and the
// two operands on the dependent chain, S^T and U~'^T (bf16), are A operands IN tensor memory.  They go there straight
// from the accumulator fragments that produced them (tcgen05.ld 16x256b -> arithmetic -> tcgen05.st 16x128b: the same
// lanes, pairs of columns packed), with no trip through shared memory, no transpose and no proxy fence.  The products
// of a chunk (the transposed ones with M = 128, or for a slice of 64 or 32 columns M = 64, rows 16 q .. + 15 in lanes 0 .. 15 of
// quadrant q: the same time per instruction, but the kernel runs at the power cap, where less work is a higher clock: 612 ->
// 583 us back to back on 32 pairs of 512 chunks):
//   P1 [DVS x 64]  = S^T . W^T                     the chain's
//   PQ [DVS x 64]  = S^T . Q^T                     right behind it, with a commit of its own
//   P3 [DVS x 128] = U~'^T . K                     U~' = decay-scaled U~; the K tile is read MN-major
//   QK [64 x 64]   = Q . K^T                       both K-major tiles; needs no state: one chunk ahead, behind P3
//   PU [DVS x 64]  = U~^T . P^T, on top of gamma_i (Q S)^T
// The dependent chain of a chunk is  P1 -> U~' -> P3 -> S^T.
//
// Warps 0..7 ("chain") work on tensor-memory lanes 32 (w & 3) .. + 31 and on half (w >> 2) of the columns: 32 tokens of
// U~, 64 features of S (fp32, in registers for the whole sequence).  The output warps form P (a chunk
// ahead of its use), the gamma-weighted start of PU, and write O one chunk behind.  The control warp issues every product; the
// gate warp brings g and its factors a chunk ahead and requests the tile copies two chunks ahead, into
// three stages of {[W ; Q], K, U}.  Hand-offs are mbarriers: commits from the products, one arrival per warp after its
// operand writes (U~' first: the product on the chain needs only that; U~ follows).  No compute warp issues a global load
// inside the loop: one in flight would make its next tensor-memory load wait for it too.
// What bounds it: with few (sequence, head) pairs the latencies of the chain (a chunk of 32 columns: P1 420 cycles, U~' 330, P3
// 410, S^T 310 and the hand-overs between them: about 1,850), with more pairs than SMs the bytes.  Measured (L2 flushed)
// against the form that kept the operands in shared memory, S as columns and issued from one lane, over several GPUs: B = 4, T = 4096,
// H = 16: 110 -> 78 .. 86 us; B = 1, T = 32768, H = 32: 743 -> 542 us; 64 packed sequences of up to 2048 tokens, H = 16: 416 -> 262 .. 290 us
// (0.82 .. 0.9 of the copy bandwidth on 82 KB per chunk and head).  Not kept, on the second shape in slices of 32 columns (505 us with L2
// flushed then): Q K^T as mma.sync in the output warps (they get what tcgen05.mma leaves: 810 us), K in P1's free lanes instead
// of a product of its own (the output warps become the bound: 689 us, before the issue by a whole warp), eight output warps
// (no gain, more contention: 532 us).
// Every mbarrier wait is bounded; on expiry the CTA raises the status word, frees its tensor memory and returns.
#include "tc_device.cuh"

namespace tri_inv {
namespace {

constexpr int C = 64, D = 128;
constexpr int kChainWarps = 8, kOutWarps = 4, kControl = kChainWarps + kOutWarps, kGate = kControl + 1, kCopy = kGate + 1, kThreadsScan = (kGate + 1) * 32;
constexpr int kStages = 3;
constexpr float kLog2e = 1.4426950408889634f;

// KDA: the per-channel form (one decay per key feature, the KDA row of Table 1).  Its decays are folded into the
// operands beforehand (kda_scan_prep_kernel, scan_kda_prep.cu): with G_ref the middle row of a chunk and G_last its last,
//     Q+ = Q exp(G - G_ref),  K- = K exp(G_ref - G),
// S^T . W^T needs no decay, (diag(exp G_ref) S)^T . Q+^T gives ((Q exp G) S)^T, Q+ K-^T is the decayed Q K^T; P3 = U~^T K-,
// scaled per column by exp(G_last - G_ref), is the state increment (K exp(G_last - G) = K- exp(G_last - G_ref): no second,
// decay-scaled copy of U~); S decays by exp(G_last) per feature.  The kernel then differs from the scalar-gate one only in
// where its operands come from and in a few scalings: S^T is put down a second time, scaled per column by exp(G_ref) of the
// coming chunk, as PQ's operand; P needs no decay; the state update has two per-column factors.  (A second S^T operand instead
// of W exp(-G_ref) from the preparation pass takes a quarter of that pass's traffic away, and a rounding of W: 180.6 -> 164 us
// for the call on B = 4, T = 4096, H = 16.)
// How many chunks from `word` on (one word per chunk, `stride` apart, at most n) have their factors in memory; polls until it is one
// at least, with a limit (0: it ran out).  A word counts one arrival per warp of the group that writes them.  A lane per chunk:
// a round trip to L2 and the fence behind it cost about 1,000 cycles, too much for each chunk of a chain whose factors lie ready.
constexpr uint32_t kReady = 4;
__device__ __noinline__ int wait_ready(const uint32_t* word, int stride, int n, int lane, unsigned long long limit_ns) {
  const uint32_t* mine = word + (size_t)(lane < n ? lane : 0) * stride;
  unsigned long long t0 = 0;
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(mine) : "memory");
    const uint32_t not_yet = __ballot_sync(0xffffffffu, lane >= n || v < kReady);
    if (!(not_yet & 1u)) {
      asm volatile("fence.proxy.async;" ::: "memory");   // the copies of these chunks (async proxy) come behind the loads above
      __syncwarp();
      return not_yet ? __ffs(not_yet) - 1 : 32;
    }
    if ((i & 63u) == 0) {
      const unsigned long long now = global_timer_ns();
      if (i == 0) t0 = now;
      else if (__any_sync(0xffffffffu, now - t0 > limit_ns)) return 0;
    }
  }
  return 0;
}

template <int DVS, bool KDA>
struct ScanCfg {
  static_assert(DVS == 128 || DVS == 64 || DVS == 32, "slices of value columns");
  static constexpr int LG = DVS == 128 ? 2 : 1;          // groups of 16 tensor-memory lanes per quadrant in use
  static constexpr int M = 64 * LG;                      // M = 64: lanes 0 .. 15 of each quadrant
  static constexpr int E = DVS == 32 ? 1 : 2;            // halves of a group of 16 lanes in use
  static constexpr int RPQ = DVS / 4;                    // value columns (rows here) per quadrant
  static constexpr int UBOX = DVS == 128 ? 2 : 1;        // 64-column boxes of U that hold the slice
  // a stage: [W ; Q] in two boxes (64 features each) of 128 rows x 128 B, K in two boxes of 64 rows, U in UBOX boxes of 64 rows
  static constexpr int WQ_BOX = 16384, K_BOX = 8192;
  static constexpr int OFF_KT = 2 * WQ_BOX, OFF_UT = OFF_KT + 2 * K_BOX, STAGE = OFF_UT + UBOX * 8192;
  static constexpr int OFF_P = kStages * STAGE;          // P, bf16 [64 tokens i][64 tokens j], K-major B operand of PU
  static constexpr int OFF_O = OFF_P + 8192;             // O on its way out: per output warp [64 tokens][RPQ columns] bf16
  static constexpr int O_WARP = C * RPQ * 2;
  static constexpr int OFF_G = OFF_O + kOutWarps * O_WARP;
  static constexpr int G_BYTES = KDA ? 9 * D * 4 : 2 * 4 * C * 4;   // per-channel: 3 vectors x 3 chunks; scalar: g, column factor, gamma_last / gamma, gamma of two chunks
  static constexpr int OFF_BAR = OFF_G + G_BYTES;
  // The 32-column slice asks for more than it uses.  Its registers and tiles would leave room on the SM for a CTA of the inversion
  // kernels (26.5 KB for the build at d = 64, 34.7 KB at d = 128), which would then sit in tcgen05.alloc with its first matrices
  // until the scan ends, because this kernel takes all of the tensor memory.  With 22 KB left they go to other
  // SMs (this kernel as a launch of its own; layer_kernel.cuh keeps other streams waiting): three builds of 2048 matrices on a second stream beside a scan of 8 pairs x 256 chunks (262 us) end after 120 us, 323 us
  // without (86 us alone).  The 64-column slice leaves them too few registers, the 128-column one too little shared memory.
  static constexpr int SMEM = DVS == 32 ? 208896 : OFF_BAR + 160;
  static_assert(SMEM >= OFF_BAR + 160, "everything up to the tensor-memory slot");
  // tensor-memory columns
  // (per-channel form: the accumulators of P1 and P3 share their columns -- the chain warps have read the one before the other
  // is issued, either way round -- and the scaled copy of S^T takes the room)
  static constexpr int TM_WS = 0, TM_DS = KDA ? 0 : 64, TM_QS = TM_DS + 128, TM_PU = TM_QS + 64, TM_QK = TM_PU + 64, TM_S = TM_QK + 64,
                       TM_SQ = KDA ? TM_S + 64 : TM_S, TM_UD = TM_SQ + 64, TM_UT = KDA ? TM_UD : TM_UD + 32;
  static_assert(TM_UT + 32 <= 512, "tensor memory");
  static constexpr int TMEM_COLS = 512;
};
static_assert(ScanCfg<128, true>::SMEM <= 232448, "one CTA per SM");

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// whether the phase is complete, without waiting
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// One arrival for the whole warp: every lane has made its operand writes visible (the caller's fences) before the lanes
// meet; lane 0 then arrives for all of them.
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& m0, uint32_t& m1, uint32_t& m2, uint32_t& m3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(m0), "=r"(m1), "=r"(m2), "=r"(m3) : "r"(addr) : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t m0, uint32_t m1, uint32_t m2, uint32_t m3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(m0), "r"(m1), "r"(m2), "r"(m3) : "memory");
}
// D (tensor memory) += A (tensor memory, one 32-bit column = two bf16 of the summed index) . B (shared memory); called by a
// whole warp, one lane issues
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Packed pairs of a 16-lane fragment (row g: r[2 n], row g + 8: r[2 n + 1], n-tile n = columns 4 n + t) into tensor memory
__device__ __forceinline__ void tmem_st_packed16(const uint32_t (&r)[8], uint32_t taddr) {   // 16 columns
  asm volatile("tcgen05.st.sync.aligned.16x128b.x4.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"
               ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st_packed32(const uint32_t (&r)[16], uint32_t taddr) {  // 32 columns
  asm volatile("tcgen05.st.sync.aligned.16x128b.x8.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};"
               ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                 "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr) : "memory");
}

// A bounded wait whose outcome all lanes of the warp agree on.  A lane that has seen the phase may poll it again: the next phase
// of every barrier of this kernel waits for something that each of its waiting warps does after its wait.  Not inlined: the
// first polls are (below), and with the timer's loop in every wait as well the 128-column instance was 2 to 6 % slower (a vote
// behind the per-lane wait: 1 to 6 % more); in this form calls of 1 .. 300 (sequence, head) pairs and 16 .. 512 chunks
// take between 0.97 and 1.02 of the per-lane waits' time.
__device__ __noinline__ bool wait_by_warp(uint32_t bar, uint32_t parity, unsigned long long limit_ns) {
  const unsigned long long t0 = global_timer_ns();
  for (uint32_t i = 1; i < kSpinLimit; ++i) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if ((i & 63u) == 0 && __any_sync(0xffffffffu, global_timer_ns() - t0 > limit_ns)) return false;
  }
  return false;
}

// Zeros into rows `rows` .. 63 of a tile of two boxes (128 bytes a row), by the output warps; then visible to the products.  Not inlined: once a
// sequence, and the 128-column walk has no register to spare.
__device__ __noinline__ void clear_rows(uint32_t tile, int box, int rows, int tid) {
  for (int e = tid; e < (C - rows) * 16; e += kOutWarps * 32)
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(tile + ((e >> 3) & 1) * box + (rows + (e >> 4)) * 128 + (e & 7) * 16), "r"(0) : "memory");
  fence_proxy_async();
}

// One (sequence, head, slice) by a whole CTA; true when a wait has run out in this thread.
// FED: W and U (per-channel form: Q+, K- and the chunks' vectors) are being written by other CTAs of the same launch (layer_kernel.cuh).  The tile copies are then requested by a warp
// of their own, kCopy, which first waits until the chunk's word in `ready` says that they are in memory (the gate warp does the same for the vectors); tensor memory
// is the caller's (`tmem`).  Otherwise the gate warp requests the copies and the CTA allocates (and frees) its tensor memory.
template <int DVS, bool KDA, bool FED>
__device__ __forceinline__ bool scan_walk(const CUtensorMap& tmW, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmU,
                                          const ScanParams& p, uint8_t* smem, int s, int h, int slice, bool first_block,
                                          const uint32_t* ready, uint32_t tmem) {
  using cfg = ScanCfg<DVS, KDA>;
  constexpr int LG = cfg::LG, E = cfg::E;
  float* sG = reinterpret_cast<float*>(smem + cfg::OFF_G);   // scalar gate: [2][4][64]: g log2e; 2^(g_ref(j) - g_j), g_ref(j) = g of the first token of j's block of eight; 2^(g_last - g_j); 2^g_j
  float* sEl = sG;                 // per-channel form: exp(G_last) [3][128], exp(G_ref) [3][128], exp(G_last - G_ref) [3][128]
  float* sEr = sG + 3 * D;
  float* sEx = sG + 6 * D;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + cfg::OFF_BAR + 128);
  const uint32_t s0 = smem_u32(smem), sP = s0 + cfg::OFF_P;
  // copies (TMA):            bar_full + 8 stage (W, Q, K, U of a chunk)
  // products done (commit):  bar_t1 (P1), bar_tq (PQ), bar_s (P3), bar_qk (QK), bar_pu (PU); a commit covers every product issued before it
  // operands written:        bar_sr (S^T by the chain warps, the chunk's factors by the gate warp), bar_ud (U~'), bar_ut (U~),
  //                          bar_ut again (P and the start of PU, output warps); one arrival per warp
  // bar_kz: the output warps have cleared the last chunk's key rows past the sequence's end (scalar gate)
  // bar_qr: the output warps have read QK;  bar_g: the gate warp has stored a chunk's factors (for the output warps, which need them early)
  const uint32_t bar_full = s0 + cfg::OFF_BAR, bar_exit = bar_full + 24, bar_t1 = bar_full + 32, bar_s = bar_full + 40, bar_pu = bar_full + 48,
                 bar_qk = bar_full + 56, bar_sr = bar_full + 64, bar_ud = bar_full + 72, bar_ut = bar_full + 80,
                 bar_kz = bar_full + 88, bar_qr = bar_full + 96, bar_g = bar_full + 104, bar_tq = bar_full + 112;
  const unsigned long long lim = p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs;   // every wait of the kernel gives up after this long
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform for the compiler
  const bool chain = warp < kChainWarps;
  const int quad = warp & 3, half = (warp >> 2) & 1;
  const int gq = lane >> 2, t = lane & 3, mi = lane >> 3, mr = lane & 7;

  const int beg = p.seq_off ? p.seq_off[s] : s * p.T;
  const int end = p.seq_off ? p.seq_off[s + 1] : (s + 1) * p.T;
  const int n_chunks = (end - beg + C - 1) / C;
  const int row0 = quad * cfg::RPQ;              // first value column of this warp's lanes, within the slice

  // State, transposed, in accumulator-fragment layout: S[lg][nt][2 e + q] = element (value column row0 + 16 lg + 8 e + gq,
  // feature 64 half + 8 nt + 2 t + q).
  float S[LG][8][2 * E];
  auto for_state = [&](auto&& f) {
#pragma unroll
    for (int lg = 0; lg < LG; ++lg)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
          for (int q = 0; q < 2; ++q)
            f(S[lg][nt][2 * e + q], (size_t)(64 * half + 8 * nt + 2 * t + q) * D + slice * DVS + row0 + 16 * lg + 8 * e + gq);
  };
  if (chain) {
    const float* src = p.S0 ? p.S0 + ((size_t)s * p.H + h) * D * D : nullptr;
    for_state([&](float& x, size_t at) { x = src ? src[at] : 0.f; });
  }
  auto store_state = [&]() {
    if (!p.S_out || !chain) return;
    float* dst = p.S_out + ((size_t)s * p.H + h) * D * D;
    for_state([&](float& x, size_t at) { dst[at] = x; });
  };
  if (n_chunks == 0) { store_state(); return false; }
  const bool misaligned = (s0 & 1023u) != 0;     // never expected; the swizzle pattern would not match the copies

  // every tile of chunk c, into stage c % 3
  auto issue_copies = [&](int c) {
    const int st = c % kStages;
    const uint32_t base = s0 + st * cfg::STAGE, bar = bar_full + 8 * st;
    const int tok0 = beg + c * C;
    // beside the preparation Q+ and K- have 64 rows for every chunk, zeros past the sequence's end in K-: rows of a neighbour would be
    // another group's, written maybe later
    const int qk0 = KDA && FED ? (beg / C + s + c) * C : tok0;
    mbar_expect_tx(bar, (uint32_t)cfg::STAGE);
    tma_load_2d(base, &tmW, bar, h * D, tok0);
    tma_load_2d(base + cfg::WQ_BOX, &tmW, bar, h * D + 64, tok0);
    tma_load_2d(base + 8192, &tmQ, bar, h * D, qk0);
    tma_load_2d(base + cfg::WQ_BOX + 8192, &tmQ, bar, h * D + 64, qk0);
    tma_load_2d(base + cfg::OFF_KT, &tmK, bar, h * D, qk0);
    tma_load_2d(base + cfg::OFF_KT + cfg::K_BOX, &tmK, bar, h * D + 64, qk0);
    tma_load_2d(base + cfg::OFF_UT, &tmU, bar, h * D + (slice * DVS) / 64 * 64, tok0);
    if constexpr (cfg::UBOX == 2) tma_load_2d(base + cfg::OFF_UT + 8192, &tmU, bar, h * D + 64, tok0);
  };
  auto full_parity = [](int c) { return (uint32_t)((c / kStages) & 1); };
  int requested = -1;   // lane 0 of the warp that requests the copies: the last chunk whose copies were requested
  auto drain_copies = [&]() {   // give-up path: the copies still on their way into this CTA's shared memory, with a limit
    for (int c = requested >= kStages ? requested - kStages + 1 : 0; c <= requested; ++c) mbar_wait_bounded(bar_full + 8 * (c % kStages), full_parity(c), lim);
  };
  // g of a chunk, by the gate warp (lane l: tokens l and l + 32).  Rows past the sequence end take the last real
  // row's g, so that every exponent stays a difference of real values.
  auto fetch_g = [&](int c, float (&gr)[2]) {
    const int tok0 = beg + c * C, rows = end - tok0 < C ? end - tok0 : C;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = lane + 32 * q < rows ? lane + 32 * q : rows - 1;
      gr[q] = p.g[(size_t)(tok0 + i) * p.H + h];
    }
  };
  // g * log2(e) of a chunk and its factors.  The decay 2^(g_i - g_j) of P is formed as 2^(g_i - g_ref) * 2^(g_ref - g_j) with
  // g_ref the first token of j's block of eight -- one exponential per (row, block) instead of one per element; the
  // second factor spans at most seven tokens of decay
  auto store_g = [&](int c, const float (&gr)[2]) {
    float* b = sG + (c & 1) * 4 * C;
    const float g_last = __shfl_sync(0xffffffffu, gr[1], 31) * kLog2e;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float gl2 = gr[q] * kLog2e;
      const float gref = __shfl_sync(0xffffffffu, gl2, lane & ~7);
      const int i = lane + 32 * q;
      b[i] = gl2;
      b[C + i] = ex2_approx(gref - gl2);
      b[2 * C + i] = ex2_approx(g_last - gl2);
      b[3 * C + i] = ex2_approx(gl2);
    }
  };
  // per-channel form: exp(G_last), exp(G_ref) and exp(G_last - G_ref) of a chunk (128 floats each, written by the preparation
  // kernel at the chunk's slot), by the gate warp: lane l brings features 4 l .. 4 l + 3 of each; three chunks' worth are kept in turn
  auto fetch_e = [&](int c, float4 (&ev)[3]) {
    const size_t slot = (size_t)((beg + c * C) / C + s);
    ev[0] = *reinterpret_cast<const float4*>(p.EL + (slot * p.H + h) * D + 4 * lane);
    ev[1] = *reinterpret_cast<const float4*>(p.ER + (slot * p.H + h) * D + 4 * lane);
    ev[2] = *reinterpret_cast<const float4*>(p.EX + (slot * p.H + h) * D + 4 * lane);
  };
  int vectors_known = 0;   // FED: the vectors of the chunks before this one are in memory
  auto wait_vectors = [&](int c) {   // by the whole gate warp; false: they did not come within the limit
    if (!FED || c < vectors_known) return true;
    const int more = wait_ready(ready + ((size_t)((beg + c * C) / C + s) * p.H + h), p.H, n_chunks - c, lane, lim);
    vectors_known = c + more;
    return more > 0;
  };
  auto store_e = [&](int c, const float4 (&ev)[3]) {
    *reinterpret_cast<float4*>(sEl + (c % 3) * D + 4 * lane) = ev[0];
    *reinterpret_cast<float4*>(sEr + (c % 3) * D + 4 * lane) = ev[1];
    *reinterpret_cast<float4*>(sEx + (c % 3) * D + 4 * lane) = ev[2];
  };
  float4 e_raw[3] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  float g_raw[2] = {0.f, 0.f};   // gate warp: g of the chunk it stores next
  bool gate_ok = true;
  if (warp == kGate) {
    if (lane == 0) {
      prefetch_tmap(&tmW); prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmU);
      for (int b = 0; b < 8; ++b) mbar_init(bar_full + 8 * b, 1);   // three stages, exit, t1, s, pu, qk
      mbar_init(bar_sr, kChainWarps + (FED ? 2 : 1));
      mbar_init(bar_ud, kChainWarps);
      mbar_init(bar_ut, kChainWarps + kOutWarps);
      mbar_init(bar_qr, kOutWarps);
      mbar_init(bar_kz, kOutWarps);
      mbar_init(bar_g, 1);
      mbar_init(bar_tq, 1);
      fence_mbar_init();
      if (!FED && !misaligned) {
        issue_copies(0);
        if (n_chunks > 1) issue_copies(1);
        requested = n_chunks > 1 ? 1 : 0;
      }
    }
    __syncwarp();
    if constexpr (KDA) {
      // the vectors of the first two chunks are in place before the loop starts, the third chunk's in registers
      gate_ok = wait_vectors(0);
      fetch_e(0, e_raw);
      store_e(0, e_raw);
      if (n_chunks > 1) { gate_ok = gate_ok && wait_vectors(1); fetch_e(1, e_raw); store_e(1, e_raw); }
      if (n_chunks > 2) { gate_ok = gate_ok && wait_vectors(2); fetch_e(2, e_raw); }
    } else {
      fetch_g(0, g_raw);
      store_g(0, g_raw);
      if (n_chunks > 1) fetch_g(1, g_raw);
    }
  }
  if (!FED && warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(cfg::TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();   // barriers initialised, tensor memory allocated, first factors in place
  tc_fence_after();
  if (!FED) tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const uint32_t tmem_w = tmem + ((uint32_t)(32 * quad) << 16);   // this warp's lanes, column 0
  bool failed = misaligned;
  // Every wait of the roles below is one of a whole warp (wait_by_warp): its lanes go on together or give up together.  What
  // follows a wait (tcgen05.ld / st, ldmatrix, stmatrix, __syncwarp) takes the full warp, and lanes that polled and read the timer
  // one by one could leave at the limit while others see the phase complete.
  auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return wait_by_warp(bar, parity, lim);
  };
  // S^T as the A operand of P1: this warp's lanes, its 64 features as 32 columns of packed pairs
  // (per-channel form: a second time for PQ, feature k times er[k], exp(G_ref) of the chunk that will read the operand)
  auto write_state_operand = [&](const float* er) {
#pragma unroll
    for (int lg = 0; lg < LG; ++lg) {
      const uint32_t at = tmem_w + ((uint32_t)(16 * lg) << 16) + 32 * half;
      uint32_t r[16];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        r[2 * nt] = pack_bf16(S[lg][nt][0], S[lg][nt][1]);
        r[2 * nt + 1] = 0u;
        if constexpr (E == 2) r[2 * nt + 1] = pack_bf16(S[lg][nt][2], S[lg][nt][3]);
      }
      tmem_st_packed32(r, at + cfg::TM_S);
      if constexpr (KDA) {
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const float2 f = *reinterpret_cast<const float2*>(er + 64 * half + 8 * nt + 2 * t);
          r[2 * nt] = pack_bf16(f.x * S[lg][nt][0], f.y * S[lg][nt][1]);
          if constexpr (E == 2) r[2 * nt + 1] = pack_bf16(f.x * S[lg][nt][2], f.y * S[lg][nt][3]);
        }
        tmem_st_packed32(r, at + cfg::TM_SQ);
      }
    }
    tmem_wait_st();
    tc_fence_before();
    warp_arrive(bar_sr, lane);
  };

  if (warp == kControl) {
    // ---------------------------------------------------------------- control warp: every tcgen05.mma of the CTA
    // The whole warp walks the loop and one elected lane issues: the operands of tcgen05.mma are uniform registers, and only
    // code that the compiler knows to be uniform keeps them there (issued by a branch of one lane, each instruction costs 67
    // cycles of moves into them, whatever its shape).
    if (!misaligned) {
      constexpr uint32_t idesc_p1 = umma_idesc(cfg::M, 64, 0);    // S^T, W or Q K-major
      constexpr uint32_t idesc_p3 = umma_idesc(cfg::M, 128, 1);   // U~'^T, K MN-major
      constexpr uint32_t idesc_qk = umma_idesc(64, 64, 0);     // Q, K K-major
      constexpr uint32_t idesc_pu = umma_idesc(cfg::M, 64, 0);    // U~^T, P K-major
      // descriptors differ from these bases only in the address field (bits 0..13, units of 16 bytes)
      const uint64_t dW = umma_desc(s0, 16, 1024), dQ = umma_desc(s0 + 8192, 16, 1024), dK = umma_desc(s0 + cfg::OFF_KT, 16, 1024),
                     dKm = umma_desc(s0 + cfg::OFF_KT, cfg::K_BOX, 1024), dP = umma_desc(sP, 16, 1024);
      auto seen = [&](uint32_t bar, uint32_t parity) { return (bool)__all_sync(0xffffffffu, mbar_test_wait(bar, parity)); };
      auto issue_qk = [&](int c) {
        const uint32_t st = (uint32_t)((c % kStages) * cfg::STAGE) >> 4;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          umma_bf16(tmem + cfg::TM_QK, dQ + st + (((ks >> 2) * cfg::WQ_BOX + (ks & 3) * 32) >> 4),
                    dK + st + (((ks >> 2) * cfg::K_BOX + (ks & 3) * 32) >> 4), idesc_qk, ks > 0);
        umma_commit(bar_qk);
      };
      auto issue_p1 = [&](uint32_t d_col, uint32_t a_col, uint64_t b) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          umma_bf16_ta(tmem + d_col, tmem + a_col + 8 * ks, b + (((ks >> 2) * cfg::WQ_BOX + (ks & 3) * 32) >> 4), idesc_p1, ks > 0);
      };
      const bool partial = ((end - beg) & (C - 1)) != 0;
      uint32_t ph = 0;
      if (wait(bar_full, 0)) issue_qk(0);
      else failed = true;
      for (int c = 0; c < n_chunks && !failed; ++c, ph ^= 1) {
        const uint32_t st = (uint32_t)((c % kStages) * cfg::STAGE) >> 4;
        TL(9);
        if (!wait(bar_sr, ph)) { failed = true; break; }   // (the chunk's tiles were waited for before its QK)
        tc_fence_after();
        TL(0);
        issue_p1(cfg::TM_WS, cfg::TM_S, dW + st);
        umma_commit(bar_t1);
        issue_p1(cfg::TM_QS, cfg::TM_SQ, dQ + st);
        umma_commit(bar_tq);
        TL(1);
        const bool last = c + 1 >= n_chunks;
        TL(2);
        if (!KDA && last && partial && !wait(bar_kz, 0u)) { failed = true; break; }
        if (!wait(bar_ud, ph)) { failed = true; break; }
        tc_fence_after();
        TL(3);
        // self-test (ScanParams::test_stall): the first CTA leaves out this product in its second chunk, so that the
        // waits for it, and then every other wait of the CTA, run out
        if (!(p.test_stall && first_block && c == 1)) {
#pragma unroll
          for (int ks = 0; ks < C / 16; ++ks)   // 16 tokens (8 columns of the A operand, 2048 bytes of the K tile) per step
            umma_bf16_ta(tmem + cfg::TM_DS, tmem + (KDA ? cfg::TM_UT : cfg::TM_UD) + 8 * ks, dKm + st + ((ks * 2048) >> 4), idesc_p3, ks > 0);
          umma_commit(bar_s);
        }
        TL(4);
        // the next chunk's QK, if its tiles have landed and this chunk's QK has been read; otherwise behind PU
        const bool early = !last && seen(bar_full + 8 * ((c + 1) % kStages), full_parity(c + 1)) && seen(bar_qr, ph);
        if (early) { tc_fence_after(); issue_qk(c + 1); }
        if (!wait(bar_ut, ph)) { failed = true; break; }   // U~ (chain warps) and P with the start of PU (output warps)
        tc_fence_after();
        TL(5);
#pragma unroll
        for (int ks = 0; ks < C / 16; ++ks)
          umma_bf16_ta(tmem + cfg::TM_PU, tmem + cfg::TM_UT + 8 * ks, dP + ((ks * 32) >> 4), idesc_pu, 1u);   // on top of gamma_i (Q S)^T
        umma_commit(bar_pu);
        TL(6);
        if (!last && !early) {
          if (!wait(bar_full + 8 * ((c + 1) % kStages), full_parity(c + 1)) || !wait(bar_qr, ph)) { failed = true; break; }
          tc_fence_after();
          issue_qk(c + 1);
        }
      }
      if (failed) {
        // A wait has run out and this CTA is about to give up its shared and tensor memory: every product issued so far is
        // waited for first, again with a limit (a commit on a spare barrier); the gate warp does the same for the copies.
        umma_commit(bar_exit);
        mbar_wait_bounded(bar_exit, 0u, lim);
      }
    }
  } else if (warp == kGate) {
    // ---------------------------------------------------------------- gate warp: tile copies of chunk c + 2, factors of chunk c + 1
    // Its arrival on bar_sr tells the control thread, and through the first product's commit every reader, that
    // the chunk's factors are in place (bar_g tells the output warps, which start on a chunk earlier).
    if (!misaligned) { warp_arrive(bar_sr, lane); if (lane == 0) mbar_arrive(bar_g); }   // the first chunk's (written before the CTA barrier above)
    failed |= !gate_ok;
    for (int c = 0; c + 1 < n_chunks && !misaligned && !failed; ++c) {
      // stage of c + 2 = that of c - 1: its readers (the products of chunk c - 1, the chain warps' U) were done before the
      // arrivals that open chunk c
      if (!wait(bar_sr, (uint32_t)(c & 1))) { failed = true; break; }
      if (!FED && lane == 0 && c + 2 < n_chunks) { issue_copies(c + 2); requested = c + 2; }
      __syncwarp();
      // the factors of c - 1 have no reader left once the first product of chunk c is complete (it was issued behind the
      // arrivals of every warp that read them); bar_qr also says that every output warp has seen bar_g of chunk c, which must not
      // run two phases ahead of a warp that still waits for it
      if (!wait(bar_t1, (uint32_t)(c & 1)) || !wait(bar_qr, (uint32_t)(c & 1))) { failed = true; break; }
      if constexpr (KDA) {
        // The vectors run one chunk further ahead than g: exp(G_ref) of chunk c + 1 is read at the end of chunk c (it
        // scales the S^T operand), so it has to be in place, and announced by an arrival, a chunk earlier.  Those of
        // c + 2 go where those of c - 1 were.
        if (c + 2 < n_chunks) store_e(c + 2, e_raw);
      } else {
        store_g(c + 1, g_raw);
      }
      warp_arrive(bar_sr, lane);
      if (lane == 0) mbar_arrive(bar_g);
      if constexpr (KDA) {
        if (c + 3 < n_chunks) {
          if (!wait_vectors(c + 3)) { failed = true; break; }
          fetch_e(c + 3, e_raw);
        }
      }
      else { if (c + 2 < n_chunks) fetch_g(c + 2, g_raw); }
    }
    if (!FED && failed && lane == 0) drain_copies();
  } else if (FED && warp == kCopy) {
    // ---------------------------------------------------------------- copy warp: tile copies of chunk c + 2, once W and U are there
    // It arrives on bar_sr itself, after its wait for the phase before: the barrier must not run two phases ahead of it while it
    // waits for another CTA.
    int known = 0;   // chunks before this one have their factors in memory
    auto request = [&](int c) -> bool {   // false: W and U did not come within the limit
      if (c >= known) {
        const int more = wait_ready(ready + ((size_t)((beg + c * C) / C + s) * p.H + h), p.H, n_chunks - c, lane, lim);
        if (!more) return false;
        known = c + more;
      }
      if (lane == 0) { issue_copies(c); requested = c; }
      __syncwarp();
      return true;
    };
    if (!misaligned) {
      warp_arrive(bar_sr, lane);
      failed = !request(0) || (n_chunks > 1 && !request(1));
    }
    for (int c = 0; c + 1 < n_chunks && !misaligned && !failed; ++c) {
      if (!wait(bar_sr, (uint32_t)(c & 1))) { failed = true; break; }
      warp_arrive(bar_sr, lane);
      if (c + 2 < n_chunks && !request(c + 2)) { failed = true; break; }
    }
    if (failed && lane == 0) drain_copies();
  } else if (chain) {
    // ---------------------------------------------------------------- chain warps
    if (!misaligned) write_state_operand(sEr);
    uint32_t ph = 0;
    for (int c = 0; c < n_chunks && !misaligned; ++c, ph ^= 1) {
      const int tok0 = beg + c * C;
      const int rows = end - tok0 < C ? end - tok0 : C;
      const float* fb = sG + (c & 1) * 4 * C;
      const uint32_t sU = s0 + (c % kStages) * cfg::STAGE + cfg::OFF_UT;
      TL(0);
      if (!wait(bar_full + 8 * (c % kStages), full_parity(c))) { failed = true; break; }   // landed long ago; U is read below
      TL(1);
      if (!wait(bar_t1, ph)) { failed = true; break; }
      tc_fence_after();
      TL(2);
      // ---- U~ = U - W S, transposed: first the decay-scaled U~' that the chain waits for (its own arrival), then U~ itself
      float v[LG][4][4];
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) tmem_ld_16x32(v[lg], tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_WS + 32 * half);
      // while those are in flight: U out of its tile, transposed on the way (matrices of 8 tokens x 8 columns), and the decays
      const int ushift = DVS == 32 ? (slice * DVS) & 32 : 0;   // a narrow slice: which half of the copied 64-column box is ours
      auto load_u = [&](int lg, uint32_t (&xu)[4][E]) {
        if constexpr (E == 2) {
#pragma unroll
          for (int nt = 0; nt < 4; nt += 2) {
            const int tok = 32 * half + 8 * (nt + (mi >> 1)) + mr, n = row0 + 16 * lg + 8 * (mi & 1);
            ldmatrix_x4_trans(sU + (n >> 6) * 8192 + tok * 128 + ((((n & 63) >> 3) ^ (tok & 7)) << 4), xu[nt][0], xu[nt][1], xu[nt + 1][0], xu[nt + 1][1]);
          }
        } else {
          const int tok = 32 * half + 8 * mi + mr, n = row0 + ushift;
          ldmatrix_x4_trans(sU + tok * 128 + (((n >> 3) ^ (tok & 7)) << 4), xu[0][0], xu[1][0], xu[2][0], xu[3][0]);
        }
      };
      uint32_t xu[4][E];
      load_u(0, xu);
      float2 dd[4];
      if constexpr (!KDA) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) dd[nt] = *reinterpret_cast<const float2*>(fb + 2 * C + 32 * half + 8 * nt + 2 * t);
      }
      const float gl = KDA ? 0.f : fb[3 * C + rows - 1];
      tmem_wait_ld();
      TL(3);
      uint32_t ut[LG][8];   // U~ packed
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) {
        if (lg > 0) load_u(lg, xu);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const uint32_t w = xu[nt][e];   // bf16 pair: low half = token 2 t
            v[lg][nt][2 * e] = __uint_as_float(w << 16) - v[lg][nt][2 * e];
            v[lg][nt][2 * e + 1] = __uint_as_float(w & 0xffff0000u) - v[lg][nt][2 * e + 1];
          }
        if (rows < C) {   // tokens past the sequence end count as zero
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            const int i = 32 * half + 8 * nt + 2 * t;
#pragma unroll
            for (int e = 0; e < E; ++e) {
              v[lg][nt][2 * e] = i < rows ? v[lg][nt][2 * e] : 0.f;
              v[lg][nt][2 * e + 1] = i + 1 < rows ? v[lg][nt][2 * e + 1] : 0.f;
            }
          }
        }
        if constexpr (!KDA) {
          uint32_t r[8];
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            r[2 * nt] = pack_bf16(v[lg][nt][0] * dd[nt].x, v[lg][nt][1] * dd[nt].y);
            r[2 * nt + 1] = E == 2 ? pack_bf16(v[lg][nt][2] * dd[nt].x, v[lg][nt][3] * dd[nt].y) : 0u;
          }
          tmem_st_packed16(r, tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_UD + 16 * half);
        }
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          ut[lg][2 * nt] = pack_bf16(v[lg][nt][0], v[lg][nt][1]);
          ut[lg][2 * nt + 1] = E == 2 ? pack_bf16(v[lg][nt][2], v[lg][nt][3]) : 0u;
        }
      }
      if constexpr (!KDA) {
        tmem_wait_st();
        tc_fence_before();
        warp_arrive(bar_ud, lane);
      }
      TL(4);
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) tmem_st_packed16(ut[lg], tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_UT + 16 * half);
      tmem_wait_st();
      tc_fence_before();
      if constexpr (KDA) warp_arrive(bar_ud, lane);   // U~ itself is the operand of both later products
      warp_arrive(bar_ut, lane);
      TL(5);
      // ---- state update and the bf16 operand for the next chunk
      if (!wait(bar_s, ph)) { failed = true; break; }
      tc_fence_after();
      TL(6);
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) {
        float ds[8][4];
        tmem_ld_16x64(ds, tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_DS + 64 * half);
        tmem_wait_ld();
        if (lg == 0) TL(10);
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          if constexpr (KDA) {
            const float2 el = *reinterpret_cast<const float2*>(sEl + (c % 3) * D + 64 * half + 8 * nt + 2 * t);
            const float2 ex = *reinterpret_cast<const float2*>(sEx + (c % 3) * D + 64 * half + 8 * nt + 2 * t);
#pragma unroll
            for (int e = 0; e < E; ++e) {
              S[lg][nt][2 * e] = fmaf(el.x, S[lg][nt][2 * e], ex.x * ds[nt][2 * e]);
              S[lg][nt][2 * e + 1] = fmaf(el.y, S[lg][nt][2 * e + 1], ex.y * ds[nt][2 * e + 1]);
            }
          } else {
#pragma unroll
            for (int q = 0; q < 2 * E; ++q) S[lg][nt][q] = fmaf(gl, S[lg][nt][q], ds[nt][q]);
          }
        }
      }
      TL(7);
      if (c + 1 < n_chunks) write_state_operand(sEr + ((c + 1) % 3) * D);   // its last reader was P1 of this chunk
      TL(8);
    }
    if (!failed) store_state();
  } else if (warp < kChainWarps + kOutWarps) {
    // ---------------------------------------------------------------- output warps
    uint32_t ph = 0;
    int o_tok0 = 0, o_rows = 0;
    uint8_t* stage = smem + cfg::OFF_O + (warp - kChainWarps) * cfg::O_WARP;
    const uint32_t stage_a = smem_u32(stage);
    constexpr int PP = cfg::RPQ / 8;   // 16-byte pieces per token in this warp's staging tile
    auto piece_at = [](int tok, int piece) {   // eight neighbouring tokens' pieces in different banks
      const int x = PP == 4 ? piece ^ ((tok >> 1) & 3) : PP == 2 ? piece ^ ((tok >> 2) & 1) : piece;
      return (uint32_t)(tok * PP * 16 + x * 16);
    };
    // O = scale * (gamma_i QS + P U~) of the previous chunk (the PU accumulator starts from gamma_i QS), while the next
    // chunk's first product runs: fragments -> [token][column] tile (stmatrix.trans) -> 16-byte stores
    auto write_output = [&]() {   // (behind the wait for that chunk's PU)
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) {
        float pu[8][4];
        tmem_ld_16x64(pu, tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_PU);
        tmem_wait_ld();
        if constexpr (E == 2) {
#pragma unroll
          for (int nt = 0; nt < 8; nt += 2)
            stmatrix_x4_trans(stage_a + piece_at(8 * (nt + (mi >> 1)) + mr, 2 * lg + (mi & 1)),
                              pack_bf16(p.scale * pu[nt][0], p.scale * pu[nt][1]), pack_bf16(p.scale * pu[nt][2], p.scale * pu[nt][3]),
                              pack_bf16(p.scale * pu[nt + 1][0], p.scale * pu[nt + 1][1]), pack_bf16(p.scale * pu[nt + 1][2], p.scale * pu[nt + 1][3]));
        } else {
#pragma unroll
          for (int nt = 0; nt < 8; nt += 4)
            stmatrix_x4_trans(stage_a + piece_at(8 * (nt + mi) + mr, 0),
                              pack_bf16(p.scale * pu[nt][0], p.scale * pu[nt][1]), pack_bf16(p.scale * pu[nt + 1][0], p.scale * pu[nt + 1][1]),
                              pack_bf16(p.scale * pu[nt + 2][0], p.scale * pu[nt + 2][1]), pack_bf16(p.scale * pu[nt + 3][0], p.scale * pu[nt + 3][1]));
        }
      }
      tc_fence_before();
      __syncwarp();
      __nv_bfloat16* Og = reinterpret_cast<__nv_bfloat16*>(p.O) + ((size_t)(o_tok0) * p.H + h) * D + slice * DVS + row0;
#pragma unroll
      for (int it = 0; it < 2 * PP; ++it) {
        const int tok = (32 * it + lane) / PP, piece = lane % PP;
        const uint4 w = *reinterpret_cast<const uint4*>(stage + piece_at(tok, piece));
        if (tok < o_rows) *reinterpret_cast<uint4*>(Og + (size_t)tok * p.H * D + 8 * piece) = w;
      }
      __syncwarp();   // the tile has been read
    };
    for (int c = 0; c < n_chunks && !misaligned; ++c, ph ^= 1) {
      const int tok0 = beg + c * C;
      const float* fb = sG + (c & 1) * 4 * C;
      TL(0);
      // ---- P = (Q K^T) * decay, lower triangle with its diagonal: rows 16 quad .. + 15 of this warp
      if (!wait(bar_g, ph) || !wait(bar_qk, ph)) { failed = true; break; }
      tc_fence_after();
      TL(1);
      if (!KDA && end - tok0 < C) {
        // The tile's rows past the sequence's end hold a neighbour's keys.  U~ is zero there, but zero times Inf or NaN is not: the state
        // product must find zeros.  QK, the tile's other reader, is done.  By these warps and not the chain's, whose loop got 1 % longer with
        // it (512 chunks, 32 pairs: 650 -> 655 us; here 654 and 653).  The per-channel form does without: clearing in either role cost it 1 to
        // 4 %; beside the preparation each chunk has rows of its own instead (issue_copies).
        clear_rows(s0 + (c % kStages) * cfg::STAGE + cfg::OFF_KT, cfg::K_BOX, end - tok0, tid - kChainWarps * 32);
        warp_arrive(bar_kz, lane);
      }
      uint32_t wa[8], wb[8];
      {
        float qk[8][4];
        tmem_ld_16x64(qk, tmem_w + cfg::TM_QK);
        tmem_wait_ld();
        tc_fence_before();
        warp_arrive(bar_qr, lane);
        const int ia = 16 * quad + gq, ib = ia + 8;
        const float g_a = KDA ? 0.f : fb[ia], g_b = KDA ? 0.f : fb[ib];
        // No branch around a block: entries right of a row's diagonal are masked by selection, and the exponent of
        // a row that lies above the whole block is not formed (its argument is replaced by zero).
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const int j0 = 8 * nt, j = j0 + 2 * t;
          float p0, p1, p2, p3;
          if constexpr (KDA) {   // the product carries its decay: only the mask is left
            p0 = j <= ia ? qk[nt][0] : 0.f; p1 = j + 1 <= ia ? qk[nt][1] : 0.f;
            p2 = j <= ib ? qk[nt][2] : 0.f; p3 = j + 1 <= ib ? qk[nt][3] : 0.f;
          } else {
            const float gref = fb[j0];
            const float2 cj = *reinterpret_cast<const float2*>(fb + C + j);
            const float ea = ex2_approx(j0 <= ia ? g_a - gref : 0.f), eb = ex2_approx(j0 <= ib ? g_b - gref : 0.f);
            p0 = j <= ia ? qk[nt][0] * ea * cj.x : 0.f; p1 = j + 1 <= ia ? qk[nt][1] * ea * cj.y : 0.f;
            p2 = j <= ib ? qk[nt][2] * eb * cj.x : 0.f; p3 = j + 1 <= ib ? qk[nt][3] * eb * cj.y : 0.f;
          }
          wa[nt] = pack_bf16(p0, p1);
          wb[nt] = pack_bf16(p2, p3);
        }
      }
      TL(2);
      // PU of the last chunk has completed: P's tile is free, O can be read.  P goes first (its fence would wait for O's stores):
      // K-major operand, row i, 16-byte pieces of eight tokens j, swizzled; x4 stores of the matrices (rows +0..7, block),
      // (rows +8..15, block), and the same of block + 1
      if (c > 0) {
        if (!wait(bar_pu, ph ^ 1)) { failed = true; break; }
        tc_fence_after();
      }
      {
        const int row = 16 * quad + 8 * (mi & 1) + mr;
#pragma unroll
        for (int nt = 0; nt < 8; nt += 2) stmatrix_x4(sP + row * 128 + (((nt + (mi >> 1)) ^ (row & 7)) << 4), wa[nt], wb[nt], wa[nt + 1], wb[nt + 1]);
        fence_proxy_async();
      }
      if (c > 0) write_output();
      TL(3);
      if (!wait(bar_tq, ph)) { failed = true; break; }
      tc_fence_after();
      TL(4);
      // ---- gamma_i (Q S)^T becomes the starting value of the PU accumulator (same lanes); in the per-channel form the
      // decay is inside the product already
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) {
        const uint32_t trow = tmem_w + ((uint32_t)(16 * lg) << 16);
        float qs[8][4];
        tmem_ld_16x64(qs, trow + cfg::TM_QS);
        tmem_wait_ld();
        if constexpr (!KDA) {
#pragma unroll
          for (int nt = 0; nt < 8; ++nt) {
            const float2 y = *reinterpret_cast<const float2*>(fb + 3 * C + 8 * nt + 2 * t);
            qs[nt][0] *= y.x; qs[nt][1] *= y.y; qs[nt][2] *= y.x; qs[nt][3] *= y.y;
          }
        }
#pragma unroll
        for (int b = 0; b < 8; b += 4) {
          const float q4[4][4] = {{qs[b][0], qs[b][1], qs[b][2], qs[b][3]}, {qs[b + 1][0], qs[b + 1][1], qs[b + 1][2], qs[b + 1][3]},
                                  {qs[b + 2][0], qs[b + 2][1], qs[b + 2][2], qs[b + 2][3]}, {qs[b + 3][0], qs[b + 3][1], qs[b + 3][2], qs[b + 3][3]}};
          tmem_st_16x32(q4, trow + cfg::TM_PU + 8 * b);
        }
      }
      tmem_wait_st();
      tc_fence_before();
      warp_arrive(bar_ut, lane);
      TL(5);
      o_tok0 = tok0;
      o_rows = end - tok0 < C ? end - tok0 : C;
    }
    if (!failed && !misaligned) {
      if (wait(bar_pu, ph ^ 1)) {
        tc_fence_after();
        write_output();
      } else {
        failed = true;
      }
    }
  }
  if (failed) atomicMax(p.status, TRI_INV_ERR_DEVICE_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if constexpr (!FED) {
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cfg::TMEM_COLS) : "memory");
  }
  return failed;
}

template <int DVS, bool KDA>
__global__ void __launch_bounds__(kThreadsScan, 1)
chunk_scan_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmQ,
                  const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmU, ScanParams p) {
  constexpr int NS = D / DVS;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int slice = blockIdx.x % NS, h = (blockIdx.x / NS) % p.H, s = blockIdx.x / (NS * p.H);
  scan_walk<DVS, KDA, false>(tmW, tmQ, tmK, tmU, p, smem, s, h, slice, blockIdx.x == 0, nullptr, 0u);
}

constexpr int kSeqsPerLaunch = 960;
struct OffsetBatch {
  int32_t cu[kSeqsPerLaunch + 1];
  int32_t n, first;
};
__global__ void __launch_bounds__(256) seq_offsets_kernel(int* out, const __grid_constant__ OffsetBatch b) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= b.n; i += gridDim.x * blockDim.x) out[b.first + i] = b.cu[i];
}

template <int DVS, bool KDA>
cudaError_t launch_scan_one(const ScanParams& p, const CUtensorMap& tmW, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                            const CUtensorMap& tmU, cudaStream_t stream) {
  using cfg = ScanCfg<DVS, KDA>;
  static std::mutex mu;
  static bool ready[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!ready[dev]) {
      if ((e = cudaFuncSetAttribute(chunk_scan_kernel<DVS, KDA>, cudaFuncAttributeMaxDynamicSharedMemorySize, cfg::SMEM)) != cudaSuccess) return e;
      if ((e = cudaFuncSetAttribute(chunk_scan_kernel<DVS, KDA>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared)) != cudaSuccess) return e;
      ready[dev] = true;
    }
  }
  const long long grid = (long long)p.n_seqs * p.H * (D / DVS);
  if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
  chunk_scan_kernel<DVS, KDA><<<(int)grid, kThreadsScan, cfg::SMEM, stream>>>(tmW, tmQ, tmK, tmU, p);
  return launched();
}

}  // namespace

// The device copy of cu_seqlens (n_seqs + 1 ints), written from kernel parameters: no host-to-device copy.
cudaError_t launch_seq_offsets(int* dev_out, const tri_inv_desc* d, cudaStream_t stream) {
  for (int s0 = 0; s0 <= d->n_seqs; s0 += kSeqsPerLaunch) {
    OffsetBatch b;
    b.first = s0;
    b.n = d->n_seqs - s0 < kSeqsPerLaunch ? d->n_seqs - s0 : kSeqsPerLaunch;
    for (int q = 0; q <= b.n; ++q) b.cu[q] = d->cu_seqlens[s0 + q];
    seq_offsets_kernel<<<(b.n + 256) / 256, 256, 0, stream>>>(dev_out, b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (s0 + kSeqsPerLaunch >= d->n_seqs) break;
  }
  return cudaSuccess;
}

// bf16 Q, K, W, U with d_k = d_v = 128 and C = 64.  One CTA per SM walks a (sequence, head) pair or a slice of its value
// columns.  A pair is cut into four slices of 32 columns while that takes half the SMs at most, into two of 64 while every
// slice gets an SM of its own: the steps between the products get shorter with the slice (512 chunks, 18 pairs, one launch:
// 498 us in slices of 32, 545 in slices of 64, 764 in one).  The first line keeps clear of the power cap, which 128 CTAs of 32 columns
// reach back to back (512 chunks, 32 pairs: one launch 529 against 541 us in slices of 64, back to back 574 at 1.78 GHz against
// 538 at 1.97 GHz; 37 pairs 612 against 541); from 19 to about 28 pairs the narrow slices do not reach it and would be 6 to 9 %
// faster than what is taken (24 pairs: 500 against 542).  With more pairs than half the SMs a CTA takes all 128 columns: the
// products take the same time at any slice width, so each further slice would repeat them in a second wave (64 chunks: 74 pairs
// 79.9 us in slices of 64, 113 in one; 75 pairs 148 and 113).
// kda selects the per-channel form: Q, K are then the prepared operands Q+, K- (scan_kda_prep.cu), with p.EL,
// p.ER, p.EX the per-chunk vectors.
cudaError_t launch_chunk_scan(const ScanParams& p, const void* Q, const void* K, const void* W, long long tokens,
                              cudaStream_t stream, bool kda) {
  CUtensorMap tmW, tmQ, tmK, tmU;
  if (!make_tmap(&tmW, W, tokens, p.H, D, C, 2) || !make_tmap(&tmQ, Q, tokens, p.H, D, C, 2) || !make_tmap(&tmK, K, tokens, p.H, D, C, 2) ||
      !make_tmap(&tmU, p.U, tokens, p.H, D, C, 2))
    return cudaErrorUnknown;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cudaErrorUnknown;
  const long long pairs = (long long)p.n_seqs * p.H;
  if (pairs * 8 <= sms) return kda ? launch_scan_one<32, true>(p, tmW, tmQ, tmK, tmU, stream) : launch_scan_one<32, false>(p, tmW, tmQ, tmK, tmU, stream);
  if (pairs * 2 <= sms) return kda ? launch_scan_one<64, true>(p, tmW, tmQ, tmK, tmU, stream) : launch_scan_one<64, false>(p, tmW, tmQ, tmK, tmU, stream);
  return kda ? launch_scan_one<128, true>(p, tmW, tmQ, tmK, tmU, stream) : launch_scan_one<128, false>(p, tmW, tmQ, tmK, tmU, stream);
}

}  // namespace tri_inv

#include "layer_kernel.cuh"   // the layer in one kernel walks with scan_walk as well

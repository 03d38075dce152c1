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
//   P1 [DVS x 64]  = S^T . W^T                     the chain's, as two products of 32 tokens with a commit each
//   PQ [DVS x 64]  = S^T . Q^T                     behind it
//   P3 [DVS x 128] = U~'^T . K                     U~' = decay-scaled U~; the K tile is read MN-major; two products of 64 features, a commit each
//   PU [DVS x 64]  = U~^T . P^T
//   QK [64 x 64]   = Q . K^T                       both K-major tiles; needs no state: one chunk ahead, behind PU
// The dependent chain of a chunk is  P1 -> U~' -> P3 -> S^T.
//
// Warps 0..7 ("chain") work on tensor-memory lanes 32 (w & 3) .. + 31 and on half (w >> 2) of the columns: 32 tokens of
// U~, 64 features of S (fp32, in registers for the whole sequence).  The halves have barriers of their own: a product's time goes by its columns
// (N / 2 cycles for 16 of the summed index, whatever M, and about 70 until its commit is seen), so the first half of the warps starts on the next
// step, and the next product on its first half of the summed index, 64 to 128 cycles before the whole product would be through.
// The output warps form P and put O one chunk behind into its tile (O = gamma_i Q S + P U~ is joined there and scaled, both in fp32); the store warp sends the
// tile on by the copy engine.  The control warp issues every product; the gate warp brings g (cp.async, two chunks ahead) and its factors a chunk
// ahead; the copy warp requests the tile copies two chunks ahead, into
// three stages of {[W ; Q], K, U}.  Hand-offs are mbarriers: commits from the products, one arrival per warp after its
// operand writes (U~' first: the product on the chain needs only that; U~ follows).  No compute warp issues a global load or store
// inside the loop: its next tensor-memory load, or the next fence for the asynchronous proxy, would wait for it.  That fence stands behind the barrier, with the
// warp that issues the product or the copy: in the output warps, behind their stores, it took up to 400 cycles.
// What bounds it: with few (sequence, head) pairs the chain (a chunk of 64 columns: P1 and P3 about 330 cycles each until the second half is
// seen, U~' 320, S^T 250, the hand-overs) and the output warps, which take nearly as long a chunk; with more pairs than SMs the bytes.  The warps slow
// each other down: code that does not fit the instruction caches (a second inlined copy of the O step: 95 -> 135 us at 100 pairs x 64 chunks), loads of tensor memory
// beside a product that nobody waits for yet (Q S, Q K^T).
// Measured back to back, us, (sequence, head) pairs x chunks; before: whole products, the start of PU put into tensor memory, O stored and g loaded by the
// warps that use them: 8 x 256: 252 -> 243, 32 x 64: 74.6 -> 70.4, 32 x 256: 277 -> 259, 64 x 64: 76.6 -> 70.8, 100 x 64: 125 -> 91.5, 148 x 64: 138 -> 128;
// per-channel form with its preparation: 8 x 256: 291 -> 266, 32 x 256: 339 -> 314, 64 x 64: 152 -> 140.  Not kept, of these (32 x 256): QK in two parts around P1 (260 .. 270), behind P1 (270), before
// PU (276); polls without a suspended wait (286) or with a suspension hint (308); O and P 32 columns at a time (267 .. 305).  Not kept before: Q K^T as
// mma.sync in the output warps (they get what tcgen05.mma leaves), K in P1's free lanes instead of a product of its own, eight output warps.
// Every mbarrier wait is bounded; on expiry the CTA raises the status word, frees its tensor memory and returns.
#include "tc_device.cuh"

namespace tri_inv {
namespace {

constexpr int C = 64, D = 128;
constexpr int kChainWarps = 8, kOutWarps = 4, kControl = kChainWarps + kOutWarps, kGate = kControl + 1, kCopy = kGate + 1, kStore = kCopy + 1, kThreadsScan = (kStore + 1) * 32;
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
  static constexpr int OFF_O = OFF_P + 8192;             // O on its way out, bf16: boxes of 64 columns (32: the narrow slice) x 64 tokens, swizzled
  static constexpr int OFF_G = OFF_O + C * DVS * 2;
  static constexpr int G_BYTES = (KDA ? 12 * D : 16 * C) * 4;   // per-channel: 3 vectors of four chunks; scalar: g and its three factors of three, and g as it comes of four
  static constexpr int OFF_BAR = OFF_G + G_BYTES;
  // The 32-column slice asks for more than it uses.  Its registers and tiles would leave room on the SM for a CTA of the inversion
  // kernels (26.5 KB for the build at d = 64, 34.7 KB at d = 128), which would then sit in tcgen05.alloc with its first matrices
  // until the scan ends, because this kernel takes all of the tensor memory.  With 22 KB left they go to other
  // SMs (this kernel as a launch of its own; layer_kernel.cuh keeps other streams waiting): three builds of 2048 matrices on a second stream beside a scan of 8 pairs x 256 chunks (262 us) end after 120 us, 323 us
  // without (86 us alone).  The 64-column slice leaves them too few registers, the 128-column one too little shared memory.
  static constexpr int SMEM = DVS == 32 ? 208896 : OFF_BAR + 192;
  static_assert(SMEM >= OFF_BAR + 192, "everything up to the tensor-memory slot");
  // Tensor-memory columns.  WS: P1 of the chunk's tokens 0 .. 31, then of 32 .. 63; the chain warps put U~ (UT) and the decay-scaled
  // U~' (UD), 16 columns of packed pairs each for 32 tokens, where they have read their accumulators (per-channel form: U~ only).
  // QS: two chunks in turn.  SQ: per-channel form, S^T scaled for PQ.
  static constexpr int TM_WS = 0, TM_UT = TM_WS, TM_UD = KDA ? TM_UT : TM_WS + 16, TM_DS = TM_WS + 64, TM_QS = TM_DS + 128, TM_PU = TM_QS + 128,
                       TM_QK = KDA ? TM_PU : TM_PU + 64, TM_S = TM_QK + 64, TM_SQ = KDA ? TM_S + 64 : TM_S;
  static_assert(TM_SQ + 64 <= 512, "tensor memory");
  static constexpr int TMEM_COLS = 512;
};
static_assert(ScanCfg<128, true>::SMEM <= 232448, "one CTA per SM");
template <int N> struct Width { static constexpr int value = N; };
__device__ __forceinline__ void tmem_ld_tokens(float (&r)[4][4], uint32_t taddr) { tmem_ld_16x32(r, taddr); }
__device__ __forceinline__ void tmem_ld_tokens(float (&r)[8][4], uint32_t taddr) { tmem_ld_16x64(r, taddr); }

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

// Two elements in one instruction, each rounded as by fmaf and by a multiplication
__device__ __forceinline__ void fma_pair(float& d0, float& d1, float2 a, float b0, float b1) {   // d += a b
  asm("{\n\t.reg .b64 d, a, b;\n\tmov.b64 d, {%0, %1};\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tfma.rn.f32x2 d, a, b, d;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "+f"(d0), "+f"(d1) : "f"(a.x), "f"(a.y), "f"(b0), "f"(b1));
}
__device__ __forceinline__ void mul_pair(float& d0, float& d1, float a) {
  asm("{\n\t.reg .b64 d, a;\n\tmov.b64 d, {%0, %1};\n\tmov.b64 a, {%2, %2};\n\tmul.rn.f32x2 d, d, a;\n\tmov.b64 {%0, %1}, d;\n\t}" : "+f"(d0), "+f"(d1) : "f"(a));
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
// FED: W and U (per-channel form: Q+, K- and the chunks' vectors) are being written by other CTAs of the same launch (layer_kernel.cuh).  The copy
// warp then waits until the chunk's word in `ready` says that they are in memory before it requests the chunk's tiles (the gate warp does the same for the
// vectors); tensor memory is the caller's (`tmem`).  Otherwise the first two chunks are requested ahead of the CTA's barrier, by the gate warp, and the CTA
// allocates (and frees) its tensor memory.
template <int DVS, bool KDA, bool FED>
__device__ __forceinline__ bool scan_walk(const CUtensorMap& tmW, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmU, const CUtensorMap& tmO,
                                          const ScanParams& p, uint8_t* smem, int s, int h, int slice, bool first_block,
                                          const uint32_t* ready, uint32_t tmem) {
  using cfg = ScanCfg<DVS, KDA>;
  constexpr int LG = cfg::LG, E = cfg::E;
  float* sG = reinterpret_cast<float*>(smem + cfg::OFF_G);   // scalar gate: [3][4][64]: g log2e; 2^(g_ref(j) - g_j), g_ref(j) = g of the first token of j's block of eight; 2^(g_last - g_j); 2^g_j
  float* sEl = sG;                 // per-channel form: exp(G_last) [4][128], exp(G_ref) [4][128], exp(G_last - G_ref) [4][128]
  float* sEr = sG + 4 * D;
  float* sEx = sG + 8 * D;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + cfg::OFF_BAR + 128);
  const uint32_t s0 = smem_u32(smem), sP = s0 + cfg::OFF_P;
  // copies (TMA):            bar_full + 8 stage (W, Q, K, U of a chunk)
  // products done (commit):  bar_t1 (P1), bar_s (P3), bar_qk (QK), bar_pu (PU); a commit covers every product issued before it
  // operands written:        bar_sr (S^T by the chain warps, the chunk's factors by the gate warp), bar_ud (U~'), bar_ut (U~),
  //                          bar_ut again (P, output warps); one arrival per warp
  // bar_t1, bar_s, bar_sr and bar_ud are the first half's (tokens 0 .. 31, features 0 .. 63); the second half's lie kSecond further on
  // bar_o: O's tile is full;  bar_of: it has been read
  // bar_kz: the output warps have cleared the last chunk's key rows past the sequence's end (scalar gate)
  // bar_qr: the output warps have read QK;  bar_g: the gate warp has stored a chunk's factors (for the output warps, which need them early)
  const uint32_t bar_full = s0 + cfg::OFF_BAR, bar_exit = bar_full + 24, bar_t1 = bar_full + 32, bar_s = bar_full + 40, bar_pu = bar_full + 48,
                 bar_qk = bar_full + 56, bar_sr = bar_full + 64, bar_ud = bar_full + 72, bar_ut = bar_full + 80,
                 bar_kz = bar_full + 88, bar_qr = bar_full + 96, bar_g = bar_full + 104, bar_o = bar_full + 112, bar_of = bar_full + 120,
                 kSecond = 104, bar_t1b = bar_t1 + kSecond, bar_sb = bar_s + kSecond, bar_srb = bar_sr + kSecond, bar_udb = bar_ud + kSecond;
  const unsigned long long lim = p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs;   // every wait of the kernel gives up after this long
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform for the compiler
  const bool chain = warp < kChainWarps;
  const int quad = warp & 3, half = (warp >> 2) & 1;
  const int gq = lane >> 2, t = lane & 3, mi = lane >> 3, mr = lane & 7;
  const uint32_t bars_half = bar_full + (half ? kSecond : 0);   // chain warps: where their half's barriers are counted from

  // uniform for the compiler as well: what the control warp's loop and its branches depend on
  const int beg = __shfl_sync(0xffffffffu, p.seq_off ? p.seq_off[s] : s * p.T, 0);
  const int end = __shfl_sync(0xffffffffu, p.seq_off ? p.seq_off[s + 1] : (s + 1) * p.T, 0);
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
  // g of a chunk into shared memory, by the gate warp (lane l: tokens l and l + 32), two chunks ahead of its use.  Rows past the sequence end take the last real
  // row's g, so that every exponent stays a difference of real values.  By cp.async: a load into registers would be waited for before
  // the next poll of a barrier, 1,400 cycles of a chunk's 2,100 with 128 CTAs at work.
  auto cp_async = [](float* dst, const float* src, auto bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(decltype(bytes)::value) : "memory");
  };
  auto fetch_g = [&](int c) {
    if (c < n_chunks) {
      const int tok0 = beg + c * C, rows = end - tok0 < C ? end - tok0 : C;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = lane + 32 * q < rows ? lane + 32 * q : rows - 1;
        cp_async(sG + (12 + (c & 3)) * C + lane + 32 * q, p.g + (size_t)(tok0 + i) * p.H + h, Width<4>{});
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // g * log2(e) of a chunk and its factors.  The decay 2^(g_i - g_j) of P is formed as 2^(g_i - g_ref) * 2^(g_ref - g_j) with
  // g_ref the first token of j's block of eight -- one exponential per (row, block) instead of one per element; the
  // second factor spans at most seven tokens of decay
  auto store_g = [&](int c) {   // behind the wait for the group; a lane reads what it copied itself
    float* b = sG + (c % 3) * 4 * C;
    const float gr[2] = {sG[(12 + (c & 3)) * C + lane], sG[(12 + (c & 3)) * C + lane + 32]};
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
  // kernel at the chunk's slot), by the gate warp: lane l brings features 4 l .. 4 l + 3 of each; four chunks' worth are kept in turn
  auto fetch_e = [&](int c) {
    if (c < n_chunks) {
      const size_t at = ((size_t)((beg + c * C) / C + s) * p.H + h) * D + 4 * lane;
      cp_async(sEl + (c & 3) * D + 4 * lane, p.EL + at, Width<16>{});
      cp_async(sEr + (c & 3) * D + 4 * lane, p.ER + at, Width<16>{});
      cp_async(sEx + (c & 3) * D + 4 * lane, p.EX + at, Width<16>{});
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto fetched = [](auto keep) { asm volatile("cp.async.wait_group %0;" ::"n"(decltype(keep)::value) : "memory"); };   // all but the last `keep`
  int vectors_known = 0;   // FED: the vectors of the chunks before this one are in memory
  auto wait_vectors = [&](int c) {   // by the whole gate warp; false: they did not come within the limit
    if (!FED || c < vectors_known) return true;
    const int more = wait_ready(ready + ((size_t)((beg + c * C) / C + s) * p.H + h), p.H, n_chunks - c, lane, lim);
    vectors_known = c + more;
    return more > 0;
  };
  bool gate_ok = true;
  if (warp == kGate) {
    if (lane == 0) {
      prefetch_tmap(&tmW); prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmU); prefetch_tmap(&tmO);
      for (int b = 0; b < 8; ++b) mbar_init(bar_full + 8 * b, 1);   // three stages, exit, t1, s, pu, qk
      mbar_init(bar_sr, kChainWarps / 2 + 2);   // and the gate and the copy warp
      mbar_init(bar_srb, kChainWarps / 2 + 2);
      mbar_init(bar_ud, kChainWarps / 2);
      mbar_init(bar_udb, kChainWarps / 2);
      mbar_init(bar_t1b, 1);
      mbar_init(bar_sb, 1);
      mbar_init(bar_ut, kChainWarps + kOutWarps);
      mbar_init(bar_qr, kOutWarps);
      mbar_init(bar_kz, kOutWarps);
      mbar_init(bar_g, 1);
      mbar_init(bar_o, kOutWarps);
      mbar_init(bar_of, 1);
      fence_mbar_init();
      if (!FED && !misaligned) {
        issue_copies(0);
        if (n_chunks > 1) issue_copies(1);
      }
    }
    __syncwarp();
    if constexpr (KDA) {
      // the vectors of the first two chunks are in place before the loop starts, the third chunk's on their way
      gate_ok = wait_vectors(0);
      fetch_e(0);
      if (n_chunks > 1) gate_ok = gate_ok && wait_vectors(1);
      fetch_e(1);
      if (n_chunks > 2) gate_ok = gate_ok && wait_vectors(2);
      fetch_e(2);
      fetched(Width<1>{});
    } else {
      fetch_g(0);
      fetch_g(1);
      fetched(Width<1>{});
      store_g(0);
      fetch_g(2);
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
    return __all_sync(0xffffffffu, wait_by_warp(bar, parity, lim));
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
    warp_arrive(bars_half + (bar_sr - bar_full), lane);
  };
  // the gate and copy warps' arrivals, on both halves' barriers
  auto arrive_sr = [&]() {
    __syncwarp();
    if (lane == 0) { mbar_arrive(bar_sr); mbar_arrive(bar_srb); }
  };

  if (warp == kControl) {
    // ---------------------------------------------------------------- control warp: every tcgen05.mma of the CTA
    // The whole warp walks the loop and one elected lane issues: the operands of tcgen05.mma are uniform registers, and only
    // code that the compiler knows to be uniform keeps them there (issued by a branch of one lane, each instruction costs 67
    // cycles of moves into them, whatever its shape).
    if (!misaligned) {
      constexpr uint32_t idesc_p1 = umma_idesc(cfg::M, 32, 0);    // S^T, half of W's tokens K-major
      constexpr uint32_t idesc_pq = umma_idesc(cfg::M, 64, 0);    // S^T, Q K-major
      constexpr uint32_t idesc_p3 = umma_idesc(cfg::M, 64, 1);    // U~'^T, half of K's features MN-major
      constexpr uint32_t idesc_qk = umma_idesc(64, 64, 0);     // Q, K K-major
      constexpr uint32_t idesc_pu = umma_idesc(cfg::M, 64, 0);    // U~^T, P K-major
      // descriptors differ from these bases only in the address field (bits 0..13, units of 16 bytes)
      const uint64_t dW = umma_desc(s0, 16, 1024), dQ = umma_desc(s0 + 8192, 16, 1024), dK = umma_desc(s0 + cfg::OFF_KT, 16, 1024),
                     dKm = umma_desc(s0 + cfg::OFF_KT, cfg::K_BOX, 1024), dP = umma_desc(sP, 16, 1024);
      auto issue_qk = [&](int c) {
        const uint32_t st = (uint32_t)((c % kStages) * cfg::STAGE) >> 4;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
          umma_bf16(tmem + cfg::TM_QK, dQ + st + (((ks >> 2) * cfg::WQ_BOX + (ks & 3) * 32) >> 4),
                    dK + st + (((ks >> 2) * cfg::K_BOX + (ks & 3) * 32) >> 4), idesc_qk, ks > 0);
        umma_commit(bar_qk);
      };
      auto seen = [&](uint32_t bar, uint32_t parity) { return (bool)__all_sync(0xffffffffu, mbar_test_wait(bar, parity)); };
      // half `fh` of the features (k-steps), into columns d_col
      auto issue_s = [&](uint32_t d_col, uint32_t a_col, uint64_t b, uint32_t idesc, int fh) {
#pragma unroll
        for (int ks = 4 * fh; ks < 4 * fh + 4; ++ks)
          umma_bf16_ta(tmem + d_col, tmem + a_col + 8 * ks, b + (((ks >> 2) * cfg::WQ_BOX + (ks & 3) * 32) >> 4), idesc, ks > 0);
      };
      // P3: tokens 32 th .. + 31 (k-steps of 16: 8 columns of the A operand, 2048 bytes of the K tile), features 64 fh .. + 63
      auto issue_p3 = [&](uint64_t b, int th, int fh) {
#pragma unroll
        for (int ks = 2 * th; ks < 2 * th + 2; ++ks)
          umma_bf16_ta(tmem + cfg::TM_DS + 64 * fh, tmem + cfg::TM_UD + 32 * th + 8 * (ks & 1), b + ((fh * cfg::K_BOX + ks * 2048) >> 4), idesc_p3, ks > 0);
      };
      const bool partial = ((end - beg) & (C - 1)) != 0;
      uint32_t ph = 0;
      bool early = false;   // this chunk's QK has been issued
      for (int c = 0; c < n_chunks && !failed; ++c, ph ^= 1) {
        const uint32_t st = (uint32_t)((c % kStages) * cfg::STAGE) >> 4;
        TL(9);
        // (P1 goes where U~ is, and QK where the output warps read the last chunk's)
        if (!early && (!wait(bar_full + 8 * (c % kStages), full_parity(c)) || (c > 0 && !wait(bar_qr, ph ^ 1)))) { failed = true; break; }
        if ((c > 0 && !wait(bar_pu, ph ^ 1)) || !wait(bar_sr, ph)) { failed = true; break; }
        tc_fence_after();
        TL(0);
        issue_s(cfg::TM_WS, cfg::TM_S, dW + st, idesc_p1, 0);
        if (!wait(bar_srb, ph)) { failed = true; break; }
        tc_fence_after();
        issue_s(cfg::TM_WS, cfg::TM_S, dW + st, idesc_p1, 1);
        umma_commit(bar_t1);
        issue_s(cfg::TM_WS + 32, cfg::TM_S, dW + st + (4096 >> 4), idesc_p1, 0);
        issue_s(cfg::TM_WS + 32, cfg::TM_S, dW + st + (4096 >> 4), idesc_p1, 1);
        umma_commit(bar_t1b);
        if (!early) issue_qk(c);
        const uint32_t qs = cfg::TM_QS + 64 * (c & 1);
        issue_s(qs, cfg::TM_SQ, dQ + st, idesc_pq, 0);
        issue_s(qs, cfg::TM_SQ, dQ + st, idesc_pq, 1);
        TL(1);
        const bool last = c + 1 >= n_chunks;
        TL(2);
        if (!KDA && last && partial && !wait(bar_kz, 0u)) { failed = true; break; }
        const bool stall = p.test_stall && first_block && c == 1;
        if (!wait(bar_ud, ph)) { failed = true; break; }
        tc_fence_after();
        TL(3);
        if (!stall) { issue_p3(dKm + st, 0, 0); issue_p3(dKm + st, 0, 1); }
        if (!wait(bar_udb, ph)) { failed = true; break; }
        tc_fence_after();
        // self-test (ScanParams::test_stall): the first CTA leaves out this product in its second chunk, so that the
        // waits for it, and then every other wait of the CTA, run out
        if (!stall) {
          issue_p3(dKm + st, 1, 0);
          umma_commit(bar_s);
          issue_p3(dKm + st, 1, 1);
          umma_commit(bar_sb);
        }
        TL(4);
        if (!wait(bar_ut, ph)) { failed = true; break; }   // U~ (chain warps) and P (output warps)
        fence_proxy_async();   // P was written by ordinary stores; the fence is on this side because the writers took up to 400 cycles for it
        tc_fence_after();
        TL(5);
#pragma unroll
        for (int ks = 0; ks < C / 16; ++ks)
          umma_bf16_ta(tmem + (KDA ? qs : (uint32_t)cfg::TM_PU), tmem + cfg::TM_UT + 32 * (ks >> 1) + 8 * (ks & 1), dP + ((ks * 32) >> 4), idesc_pu,
                       KDA || ks > 0);   // per-channel form: on top of (Q S)^T, which carries its decay
        umma_commit(bar_pu);
        TL(6);
        // the next chunk's QK, if its tiles have landed and this chunk's QK has been read; otherwise behind its P1
        early = !last && seen(bar_full + 8 * ((c + 1) % kStages), full_parity(c + 1)) && seen(bar_qr, ph);
        if (early) { tc_fence_after(); issue_qk(c + 1); }
        TL(11);
      }
      if (failed) {
        // A wait has run out and this CTA is about to give up its shared and tensor memory: every product issued so far is
        // waited for first, again with a limit (a commit on a spare barrier); the gate warp does the same for the copies.
        umma_commit(bar_exit);
        mbar_wait_bounded(bar_exit, 0u, lim);
      }
    }
  } else if (warp == kGate) {
    // ---------------------------------------------------------------- gate warp: factors of chunk c + 1
    // Its arrival on bar_sr tells the control thread, and through the first product's commit every reader, that
    // the chunk's factors are in place (bar_g tells the output warps, which start on a chunk earlier).
    if (!misaligned) { arrive_sr(); if (lane == 0) mbar_arrive(bar_g); }   // the first chunk's (written before the CTA barrier above)
    failed |= !gate_ok;
    for (int c = 0; c + 1 < n_chunks && !misaligned && !failed; ++c) {
      // the factors of c - 2 (per-channel form: the vectors of c - 1) have no reader left once the first product of chunk c is complete (it was issued behind the
      // arrivals of every warp that read them); bar_qr also says that every output warp has seen bar_g of chunk c, which must not
      // run two phases ahead of a warp that still waits for it
      if (!wait(bar_t1b, (uint32_t)(c & 1)) || !wait(bar_qr, (uint32_t)(c & 1))) { failed = true; break; }
      fetched(Width<KDA ? 0 : 1>{});
      // The vectors run one chunk further ahead than g: exp(G_ref) of chunk c + 1 is read at the end of chunk c (it
      // scales the S^T operand), so it has to be in place, and announced by an arrival, a chunk earlier.
      if constexpr (!KDA) store_g(c + 1);
      arrive_sr();
      if (lane == 0) mbar_arrive(bar_g);
      if constexpr (KDA) {
        if (c + 3 < n_chunks && !wait_vectors(c + 3)) { failed = true; break; }
        fetch_e(c + 3);
      } else {
        fetch_g(c + 3);
      }
    }
    if (failed) fetched(Width<0>{});   // give-up path: its copies too are through before the CTA gives up its shared memory
  } else if (warp == kCopy) {
    // ---------------------------------------------------------------- copy warp: tile copies of chunk c + 2 (FED: once W and U are there)
    // It arrives on bar_sr itself, after its wait for the phase before: the barrier must not run two phases ahead of it while it
    // waits for another CTA.
    int known = 0;   // chunks before this one have their factors in memory
    auto request = [&](int c) -> bool {   // false: W and U did not come within the limit
      if (FED && c >= known) {
        const int more = wait_ready(ready + ((size_t)((beg + c * C) / C + s) * p.H + h), p.H, n_chunks - c, lane, lim);
        if (!more) return false;
        known = c + more;
      }
      if (lane == 0) { issue_copies(c); requested = c; }
      __syncwarp();
      return true;
    };
    if (!misaligned) {
      arrive_sr();
      if constexpr (FED) failed = !request(0) || (n_chunks > 1 && !request(1));
      else requested = n_chunks > 1 ? 1 : 0;   // by the gate warp, before the CTA barrier
    }
    for (int c = 0; c + 1 < n_chunks && !misaligned && !failed; ++c) {
      if (!wait(bar_sr, (uint32_t)(c & 1)) || !wait(bar_srb, (uint32_t)(c & 1))) { failed = true; break; }
      arrive_sr();
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
      const float* fb = sG + (c % 3) * 4 * C;
      const uint32_t sU = s0 + (c % kStages) * cfg::STAGE + cfg::OFF_UT;
      TL(0);
      if (!wait(bar_full + 8 * (c % kStages), full_parity(c))) { failed = true; break; }   // landed long ago; U is read below
      TL(1);
      if (!wait(bars_half + (bar_t1 - bar_full), ph)) { failed = true; break; }
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
          tmem_st_packed16(r, tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_UD + 32 * half);
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
        warp_arrive(bars_half + (bar_ud - bar_full), lane);
      }
      TL(4);
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) tmem_st_packed16(ut[lg], tmem_w + ((uint32_t)(16 * lg) << 16) + cfg::TM_UT + 32 * half);
      tmem_wait_st();
      tc_fence_before();
      if constexpr (KDA) warp_arrive(bars_half + (bar_ud - bar_full), lane);   // U~ itself is the operand of both later products
      warp_arrive(bar_ut, lane);
      TL(5);
      // ---- state update and the bf16 operand for the next chunk
      if (!wait(bars_half + (bar_s - bar_full), ph)) { failed = true; break; }
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
            const float2 el = *reinterpret_cast<const float2*>(sEl + (c & 3) * D + 64 * half + 8 * nt + 2 * t);
            const float2 ex = *reinterpret_cast<const float2*>(sEx + (c & 3) * D + 64 * half + 8 * nt + 2 * t);
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
      if (c + 1 < n_chunks) write_state_operand(sEr + ((c + 1) & 3) * D);   // its last reader was P1 of this chunk
      TL(8);
    }
    if (!failed) store_state();
  } else if (warp < kChainWarps + kOutWarps) {
    // ---------------------------------------------------------------- output warps
    // 16 bytes (eight columns) of a token in O's tile: the swizzle that the copy engine undoes on the way out
    auto o_at = [&](int tok, int col) {
      if constexpr (DVS == 32) return s0 + cfg::OFF_O + tok * 64 + ((((col >> 3) ^ (tok >> 1)) & 3) << 4);
      else return s0 + cfg::OFF_O + (col >> 6) * 8192 + tok * 128 + ((((col >> 3) ^ tok) & 7) << 4);
    };
    // O = scale * (gamma_i QS + P U~) of a chunk out of tensor memory (behind the wait for its PU) into its tile, from where the store warp
    // sends it on.  Accumulator fragments -> [token][column] by stmatrix.trans.
    auto put_output = [&](int c) -> bool {
      if (c > 0 && !wait(bar_of, (uint32_t)((c - 1) & 1))) return false;   // the last chunk's store has read the tile
      const float* gam = sG + (c % 3) * 4 * C + 3 * C + 2 * t;
      constexpr int NC = 4;   // blocks of eight tokens at a time: what the registers of 128 columns allow, and faster for 64 (32768 tokens, 32 heads: 571 -> 545 us)
#pragma unroll
      for (int lg = 0; lg < LG; ++lg) {
#pragma unroll
        for (int n0 = 0; n0 < 8; n0 += NC) {
          const uint32_t at = tmem_w + ((uint32_t)(16 * lg) << 16) + 8 * n0;
          float pu[NC][4], qs[NC][4];
          tmem_ld_tokens(pu, at + (KDA ? cfg::TM_QS + 64 * (c & 1) : cfg::TM_PU));
          if constexpr (KDA) {
            tmem_wait_ld();
          } else {
            tmem_ld_tokens(qs, at + cfg::TM_QS + 64 * (c & 1));
            float2 y[NC];
#pragma unroll
            for (int nt = 0; nt < NC; ++nt) y[nt] = *reinterpret_cast<const float2*>(gam + 8 * (n0 + nt));
            tmem_wait_ld();
#pragma unroll
            for (int nt = 0; nt < NC; ++nt)
#pragma unroll
              for (int e = 0; e < E; ++e) fma_pair(pu[nt][2 * e], pu[nt][2 * e + 1], y[nt], qs[nt][2 * e], qs[nt][2 * e + 1]);
          }
          // The scale last, on the fp32 sum, and not in P's and gamma's factors: P is rounded to bf16, elsewhere with a scale in it (3.2e-3 of O).  In pairs it takes the
          // instructions that the join alone took (32768 tokens, 32 heads: 608 us, 608 with the scale in the factors, 614 one by one).
#pragma unroll
          for (int nt = 0; nt < NC; ++nt)
#pragma unroll
            for (int e = 0; e < E; ++e) mul_pair(pu[nt][2 * e], pu[nt][2 * e + 1], p.scale);
          if constexpr (E == 2) {
#pragma unroll
            for (int nt = 0; nt < NC; nt += 2)
              stmatrix_x4_trans(o_at(8 * (n0 + nt + (mi >> 1)) + mr, row0 + 16 * lg + 8 * (mi & 1)),
                                pack_bf16(pu[nt][0], pu[nt][1]), pack_bf16(pu[nt][2], pu[nt][3]), pack_bf16(pu[nt + 1][0], pu[nt + 1][1]), pack_bf16(pu[nt + 1][2], pu[nt + 1][3]));
          } else {
#pragma unroll
            for (int nt = 0; nt < NC; nt += 4)
              stmatrix_x4_trans(o_at(8 * (n0 + nt + mi) + mr, row0),
                                pack_bf16(pu[nt][0], pu[nt][1]), pack_bf16(pu[nt + 1][0], pu[nt + 1][1]), pack_bf16(pu[nt + 2][0], pu[nt + 2][1]), pack_bf16(pu[nt + 3][0], pu[nt + 3][1]));
          }
        }
      }
      tc_fence_before();
      return true;
    };
    // rows 16 quad .. + 15 of P's tile (K-major operand, row i, 16-byte pieces of eight tokens j, swizzled): the columns that form_p leaves out are zero
    for (int e = lane; e < 16 * 8; e += 32)
      asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sP + 2048 * quad + 16 * e), "r"(0) : "memory");
    __syncwarp();
    uint32_t ph = 0;
    // P = (Q K^T) * decay of chunk c, lower triangle with its diagonal: rows 16 quad .. + 15 and the first 8 NT columns.
    // Its factors first, while QK is on its way.  No branch around a block: entries right of a row's diagonal are masked by
    // selection, and the exponent of a row that lies above the whole block is not formed (its argument is replaced by zero).
    float f[8][4];
    const int ia = 16 * quad + gq, ib = ia + 8;
    auto form_factors = [&](auto width, const float* fb) {
      const float g_a = fb[ia], g_b = fb[ib];
#pragma unroll
      for (int nt = 0; nt < decltype(width)::value; ++nt) {
        const float gref = fb[8 * nt];
        const float2 cj = *reinterpret_cast<const float2*>(fb + C + 8 * nt + 2 * t);
        const float ea = ex2_approx(8 * nt <= ia ? g_a - gref : 0.f), eb = ex2_approx(8 * nt <= ib ? g_b - gref : 0.f);
        f[nt][0] = ea * cj.x; f[nt][1] = ea * cj.y;
        f[nt][2] = eb * cj.x; f[nt][3] = eb * cj.y;
      }
    };
    auto form_p = [&](auto width) {
      constexpr int NT = decltype(width)::value;
      float qk[NT][4];
      tmem_ld_tokens(qk, tmem_w + cfg::TM_QK);
      tmem_wait_ld();
      tc_fence_before();
      warp_arrive(bar_qr, lane);
      uint32_t wa[NT], wb[NT];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int j = 8 * nt + 2 * t;
        if constexpr (!KDA) {   // (per-channel form: the product carries its decay, only the mask is left)
#pragma unroll
          for (int q = 0; q < 4; ++q) qk[nt][q] *= f[nt][q];
        }
        wa[nt] = pack_bf16(j <= ia ? qk[nt][0] : 0.f, j + 1 <= ia ? qk[nt][1] : 0.f);
        wb[nt] = pack_bf16(j <= ib ? qk[nt][2] : 0.f, j + 1 <= ib ? qk[nt][3] : 0.f);
      }
      // x4 stores of the matrices (rows +0..7, block), (rows +8..15, block), and the same of block + 1
      const int row = 16 * quad + 8 * (mi & 1) + mr;
#pragma unroll
      for (int nt = 0; nt < NT; nt += 2) stmatrix_x4(sP + row * 128 + (((nt + (mi >> 1)) ^ (row & 7)) << 4), wa[nt], wb[nt], wa[nt + 1], wb[nt + 1]);
    };
    const bool narrow = quad < 2;   // nothing in the right half (and on the schedulers of the control and the gate warp)
    // Chunk c: its P, and the O of the chunk before (a last round has only that: one copy of each in the code, since the warps of a CTA run different
    // code and what does not fit the instruction caches slows all of them down)
    for (int c = 0; c <= n_chunks && !misaligned; ++c, ph ^= 1) {
      TL(0);
      const bool more = c < n_chunks;
      if (more) {
        // (per-channel form: waited for as well, so that bar_qr does not run two phases ahead of the gate warp)
        if (!wait(bar_g, ph)) { failed = true; break; }
        if constexpr (!KDA) {
          if (narrow) form_factors(Width<4>{}, sG + (c % 3) * 4 * C);
          else form_factors(Width<8>{}, sG + (c % 3) * 4 * C);
        }
      }
      if (c > 0) {   // PU of the chunk before has completed: its O can be read, and P's tile is free
        if (!wait(bar_pu, ph ^ 1)) { failed = true; break; }
        tc_fence_after();
        if (!put_output(c - 1)) { failed = true; break; }
      }
      if (more) {
        if (!wait(bar_qk, ph)) { failed = true; break; }
        tc_fence_after();
        TL(1);
        if (!KDA && end - beg - c * C < C) {
          // The tile's rows past the sequence's end hold a neighbour's keys.  U~ is zero there, but zero times Inf or NaN is not: the state
          // product must find zeros.  QK, the tile's other reader, is done.  By these warps and not the chain's, whose loop got 1 % longer with
          // it (512 chunks, 32 pairs: 650 -> 655 us; here 654 and 653).  The per-channel form does without: clearing in either role cost it 1 to
          // 4 %; beside the preparation each chunk has rows of its own instead (issue_copies).
          clear_rows(s0 + (c % kStages) * cfg::STAGE + cfg::OFF_KT, cfg::K_BOX, end - beg - c * C, tid - kChainWarps * 32);
          warp_arrive(bar_kz, lane);
        }
        if (narrow) form_p(Width<4>{});
        else form_p(Width<8>{});
        TL(2);
      }
      // (the fences between these ordinary stores and what reads them through the asynchronous proxy are the control and the store warp's)
      __syncwarp();
      if (lane == 0) {
        if (more) mbar_arrive(bar_ut);
        if (c > 0) mbar_arrive(bar_o);
      }
      TL(5);
    }
  } else if (warp == kStore) {
    // ---------------------------------------------------------------- store warp: O's tile to memory
    // By the copy engine, whose stores cost the output warps nothing and write whole rows of 128 bytes; the rows of a partial chunk by ordinary ones.
    for (int c = 0; c < n_chunks && !misaligned; ++c) {
      if (!wait(bar_o, (uint32_t)(c & 1))) { failed = true; break; }
      const int tok0 = beg + c * C;
      if (end - tok0 >= C) {
        if (lane == 0) {
          fence_proxy_async();   // the tile was written by ordinary stores
          tma_store_2d(&tmO, s0 + cfg::OFF_O, h * D + slice * DVS, tok0);
          if constexpr (DVS == 128) tma_store_2d(&tmO, s0 + cfg::OFF_O + 8192, h * D + 64, tok0);
          bulk_commit();
          bulk_wait_read();
        }
      } else {
        __nv_bfloat16* Og = reinterpret_cast<__nv_bfloat16*>(p.O) + ((size_t)tok0 * p.H + h) * D + slice * DVS;
        for (int e = lane; e < (end - tok0) * (DVS / 8); e += 32) {
          const int tok = e / (DVS / 8), pc = e % (DVS / 8);
          const int at = DVS == 32 ? tok * 64 + (((pc ^ (tok >> 1)) & 3) << 4) : (pc >> 3) * 8192 + tok * 128 + (((pc ^ tok) & 7) << 4);
          *reinterpret_cast<uint4*>(Og + (size_t)tok * p.H * D + 8 * pc) = *reinterpret_cast<const uint4*>(smem + cfg::OFF_O + at);
        }
      }
      warp_arrive(bar_of, lane);
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
                  const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmO, ScanParams p) {
  constexpr int NS = D / DVS;
  extern __shared__ __align__(1024) uint8_t smem[];
  wait_for_predecessor();   // (its successor starts when it is through: with a signal in the gate warp's loop 100 pairs x 64 chunks took 100 us, 95 without)
  const int slice = blockIdx.x % NS, h = (blockIdx.x / NS) % p.H, s = blockIdx.x / (NS * p.H);
  scan_walk<DVS, KDA, false>(tmW, tmQ, tmK, tmU, tmO, p, smem, s, h, slice, blockIdx.x == 0, nullptr, 0u);
}

constexpr int kSeqsPerLaunch = 960;
struct OffsetBatch {
  int32_t cu[kSeqsPerLaunch + 1];
  int32_t n, first;
};
__global__ void __launch_bounds__(256) seq_offsets_kernel(int* out, const __grid_constant__ OffsetBatch b) {
  let_successor_start();
  wait_for_predecessor();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= b.n; i += gridDim.x * blockDim.x) out[b.first + i] = b.cu[i];
}

// O as the scans store it: boxes of 64 tokens x 64 columns, or 32 of the narrow slice
template <int DVS>
bool make_tmap_out(CUtensorMap* tm, const void* base, long long tokens, int H) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)H * D, (cuuint64_t)tokens};
  cuuint64_t strides[1] = {(cuuint64_t)H * D * 2};
  cuuint32_t box[2] = {DVS == 32 ? 32 : 64, (cuuint32_t)C};
  cuuint32_t estr[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            DVS == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DVS, bool KDA>
cudaError_t launch_scan_one(const ScanParams& p, const CUtensorMap& tmW, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                            const CUtensorMap& tmU, long long tokens, cudaStream_t stream) {
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
  CUtensorMap tmO;
  if (!make_tmap_out<DVS>(&tmO, p.O, tokens, p.H)) return cudaErrorUnknown;
  e = launch_early(chunk_scan_kernel<DVS, KDA>, dim3((unsigned)grid), kThreadsScan, cfg::SMEM, stream, tmW, tmQ, tmK, tmU, tmO, p);
  return e == cudaSuccess ? launched() : e;
}

}  // namespace

// The device copy of cu_seqlens (n_seqs + 1 ints), written from kernel parameters: no host-to-device copy.
cudaError_t launch_seq_offsets(int* dev_out, const tri_inv_desc* d, cudaStream_t stream) {
  for (int s0 = 0; s0 <= d->n_seqs; s0 += kSeqsPerLaunch) {
    OffsetBatch b;
    b.first = s0;
    b.n = d->n_seqs - s0 < kSeqsPerLaunch ? d->n_seqs - s0 : kSeqsPerLaunch;
    for (int q = 0; q <= b.n; ++q) b.cu[q] = d->cu_seqlens[s0 + q];
    const cudaError_t e = launch_early(seq_offsets_kernel, dim3((b.n + 256) / 256), 256, 0, stream, dev_out, b);
    if (e != cudaSuccess) return e;
    if (s0 + kSeqsPerLaunch >= d->n_seqs) break;
  }
  return cudaSuccess;
}

// bf16 Q, K, W, U with d_k = d_v = 128 and C = 64.  One CTA per SM walks a (sequence, head) pair or a slice of its value
// columns.  A pair is cut into four slices of 32 columns while that takes half the SMs at most, into two of 64 while every
// slice gets an SM of its own: the steps between the products get shorter with the slice (512 chunks, 18 pairs, back to back: 473 us in slices of 32, 498 in
// slices of 64, 651 in one).  The first line keeps clear of the power cap, which 112 and more CTAs of 32 columns reach: 28 x 256 254 us in slices of 32 and 250 in slices of 64, 32 x 64 68 and 66,
// 32 x 512 532 to 558 and 499, 37 x 512 593 and 506.  Between the line and there (19 to 27 pairs) the narrow slices are 4 to 5 % faster by themselves (24 x 64: 62.5 and 65.2; 24 x 512: 472 and 497) and
// behind a fused call that is not long (24 x 64: 90 and 93, 24 x 128: 167 and 173), and slower behind a long one, which leaves the chip hot (24 x 512: 671 and 657); the layer call takes one kernel for these shapes.  With more
// slices of 64 than SMs a CTA takes all 128 columns: the
// products take the same time at any slice width, so each further slice would repeat them in a second wave (64 chunks: 74 pairs
// 76 us in slices of 64, 90 in one; 75 pairs 133 and 90).
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
  if (pairs * 8 <= sms) return kda ? launch_scan_one<32, true>(p, tmW, tmQ, tmK, tmU, tokens, stream) : launch_scan_one<32, false>(p, tmW, tmQ, tmK, tmU, tokens, stream);
  if (pairs * 2 <= sms) return kda ? launch_scan_one<64, true>(p, tmW, tmQ, tmK, tmU, tokens, stream) : launch_scan_one<64, false>(p, tmW, tmQ, tmK, tmU, tokens, stream);
  return kda ? launch_scan_one<128, true>(p, tmW, tmQ, tmK, tmU, tokens, stream) : launch_scan_one<128, false>(p, tmW, tmQ, tmK, tmU, tokens, stream);
}

}  // namespace tri_inv

#include "layer_kernel.cuh"   // the layer in one kernel walks with scan_walk as well

// Backward pass on the 5th-generation tensor cores, bf16, d = 64 or 128.
//
// Formulas (derivative of Eq. 1 with the permutation held constant; per branch x, with
// dO = g_x dY and Delta_i = g_x sum_c dY[i,c] Y_x[i,c]):
//   P_ij = exp(scale q_i.k_j - lse_i),  dP_ij = dY_i . v_j,
//   dS_ij = scale P_ij (g_x dP_ij - Delta_i),
//   dQ_i = sum_j dS_ij k_j,   dK_j = sum_i dS_ij q_i,   dV_j = sum_i g_x P_ij dY_i.
//
// prep_kernel first: Delta and lse of every row, in the order the kernels read them, the partial
// sums of the gate gradients, and (SA branch) copies of Q, dY, K, V in slot order.  A row is met by
// (128 + w) / 128 row tiles in each of the two launches, and gathering it every time holds the
// load/store unit for 28 cycles per 512 bytes (3600 cycles for a 128-row K + V tile pair, more than
// its products take), while the copy costs one pass at HBM speed, part of which the Delta sums
// need anyway.  Circular windows get the first and last h slots once more on the other side, so
// that every tile is one box.  The one-sided SWA branch, whose rows are consecutive tokens, is read
// in place.
//
// Then two launches per branch, neither of which needs an atomic, so results are run-to-run
// identical:
//   rows = queries: an item is 128 query slots of one head; it walks the K/V tiles of its
//                   band, and accumulates dQ;
//   rows = keys:    an item is 128 key slots of one KV head; it walks the query tiles that can
//                   see them for every query head of the group, and accumulates dK and dV.
// A persistent grid, one CTA per SM, walks the items.  One step (rows: Q, dY or K, V; a column
// tile of 128: K, V or Q, dY): S = R1 C1^T and dP = R2 C2^T into tensor memory, P and dS in
// registers, back to tensor memory as bf16, and from there times the column tiles into the
// accumulators.  All tiles come by TMA.
//
// Four threads share a row, 32 columns each (nothing is reduced along a row here), so that 16 warps
// hide one another's latencies.  A thread takes its scores out of tensor memory and keeps P in
// registers until dP is there, so the next step's scores go into the same columns S while this
// step is worked on.  With columns left for two dP buffers (all but rows = keys at d = 128) both
// score products of a step run ahead of the accumulation before it; P and dS are written over dP.
// Rows = keys at d = 128 have columns for one dP buffer: it is filled, answered and accumulated in
// two halves of 64 columns, so that one half's products run while the other is worked on.
//
// Bound: the tensor pipe (128-cycle-per-16-columns products in four groups, and ~180 cycles per
// commit) where windows are wide, HBM and the item's fixed latencies where they are narrow.
// Whole backward, us, gathering kernels with one item per CTA before / now: 32/8 heads of 128, n = 10007,
// w = 1024, gated 2166 / 1440; 8 x 12 heads of 64, n = 4096, w = 128, gated 687 / 515; SA alone, 16 x 16
// heads of 64, n = 2048, w = 256 810 / 479.
//
// Every mbarrier wait is bounded; on expiry the CTA records SA_ERR_TIMEOUT in the device status
// word, stops issuing work, drains what it started and returns.
#include <type_traits>

#include "sa_bwd_tc.cuh"
#include "sa_gemm_common.cuh"
#include "sa_tc_common.cuh"

namespace sa {
namespace {

constexpr int kTile = 128;
constexpr int kRowWarps = 16, kThreads = 32 * (kRowWarps + 4);
constexpr uint32_t kTmemCols = 512;

// Where a branch's rows live.  Copies: row `left + slot` of [B, H, ext, d]; in place: left = 0,
// ext = n.  Statistics and token lists: index `sleft + slot` with `spitch` per head (sequence).
struct Order {
  int left, ext, sleft, spitch;
  int circular;              // the window wraps, and the copies with it
};

struct BwdTcParams {
  const int32_t* perm;        // null for the SWA branch
  const int32_t* tok;         // [B, spitch]: token of every slot
  const float *lse2, *delta;  // [B, Hq, spitch] of this branch: lse log2(e) - log2(scale), Delta
  const float* gate_logit;    // null, or the [Hq] logits of this branch
  void *dq, *dk, *dv;
  int accumulate;             // add to what the outputs already hold
  // The launch before is a kernel of this pass that needs no wait but for what the outputs hold, and
  // it started behind prep_kernel, which wrote all that is read (past L1).  Then only the epilogue
  // waits for it, and these CTAs fill the SMs that its last round leaves idle.
  // Gated training pass, 8 x 12 heads of 64, n = 4096, w = 128: 788 -> 763 us; 32/8 heads of 128,
  // n = 10007, w = 1024: 2208 -> 2143.
  int late_wait;
  int* status;
  const int* abort_flag;
  int B, Hq, Hkv, G, n, w, h;
  int linear, one_sided, full_range;
  int n_tiles;
  int step_r0, step_h, step_b;   // from an item to the one gridDim.x later
  uint32_t magic_g;              // hr / G == umulhi(hr, magic_g)
  Order o;
  float scale, scale2;
  int64_t qs[3], ks[3];
};

// Columns (virtual slots) a row tile starting at slot r0 has to meet: T tiles from cstart on.
// rows_are_keys selects the transposed window of the one-sided rule.  For the symmetric windows
// cstart + h is a multiple of 128 (the statistics are loaded from 16-byte boundaries).
__device__ __forceinline__ void column_range(const BwdTcParams& p, int r0, bool rows_are_keys,
                                             int* cstart, int* T) {
  const int rl = min(r0 + kTile - 1, p.n - 1);
  int lo, hi;
  if (p.full_range) { lo = 0; hi = p.n - 1; }
  else if (p.one_sided) {
    if (rows_are_keys) { lo = r0; hi = min(rl + p.w - 1, p.n - 1); }
    else { lo = max(r0 - (p.w - 1), 0); hi = rl; }
  } else {
    lo = r0 - p.h;
    hi = rl + p.h;
    if (p.linear) {
      if (lo < 0) lo += -lo / kTile * kTile;
      hi = min(hi, p.n - 1);
    }
  }
  *cstart = lo;
  *T = (hi - lo + kTile) / kTile;
}

// KEYS: rows are keys (dK, dV), else queries (dQ).
template <int D, bool KEYS>
struct BCfg {
  static constexpr int kTileBytes = kTile * D * 2, kChunkBytes = kTile * 128;
  // Column tile slots.  A step's score products are wanted right behind the accumulations of the
  // step before last, and a tile takes 1000 cycles to come: at d = 128 a pair of two-slot rings
  // freed together idled the tensor pipe for 1300 of 3400 cycles a step.  Rows = queries: C1 (K)
  // is freed by the accumulation, three slots; C2 (V) by its dP product already, one slot.  Rows =
  // keys: C1 (Q) by dK, which goes first, C2 (dY) by dV behind it, two slots each.  At d = 64
  // three of each.
  static constexpr int kC1 = D == 64 ? 3 : KEYS ? 2 : 3, kC2 = D == 64 ? 3 : KEYS ? 2 : 1;
  static constexpr int kRBufs = D == 128 ? 1 : 2;               // row operand pairs
  static constexpr int kAccCols = (KEYS ? 2 : 1) * D;
  // dP buffers.  Rows = keys has room for one (at d = 128): it is worked on in two halves of 64
  // columns, so that the products of one half run while the row threads have the other.
  static constexpr int kNX = KEYS ? 1 : 2;
  static constexpr int kPArrivals = KEYS ? kRowWarps / 2 : kRowWarps;
  static constexpr int kAccBufs = D == 64 ? 2 : 1;
  static constexpr int kOffR = 0;
  static constexpr int kOffC = kRBufs * 2 * kTileBytes;
  static constexpr int kOffC2 = kOffC + kC1 * kTileBytes;
  // staging of the epilogue: rows of 64 bytes per row warp (half a warp's at a time where only
  // 16 KB are left)
  static constexpr int kStageRows = D == 128 && KEYS ? 16 : 32;
  static constexpr int kOffStage = kOffC2 + kC2 * kTileBytes;
  static constexpr int kOffVec = kOffStage + kRowWarps * kStageRows * 64;
  static constexpr int kVecTok = KEYS ? 2 * kTile : 0, kVec = kVecTok + kTile;  // (lse2, delta,) tokens
  static constexpr int kOffBar = kOffVec + kC1 * kVec * 4;
  static constexpr int kBarRFull = 0, kBarREmpty = kRBufs, kBarC1Full = 2 * kRBufs,
                       kBarC2Full = kBarC1Full + kC1, kBarC1Empty = kBarC2Full + kC2,
                       kBarVFull = kBarC1Empty + kC1, kBarSFull = kBarVFull + kC1, kBarSRead = kBarSFull + 1,
                       kBarDpFull = kBarSRead + 1, kBarPReady = kBarDpFull + 2,
                       kBarAccFull = kBarPReady + 2,
                       kBarAccFree = kBarAccFull + kAccBufs, kNumBars = kBarAccFree + kAccBufs;
  static constexpr int kOffMisc = kOffBar + kNumBars * 8;
  static constexpr int kBytes = kOffMisc + 16;
  // tensor memory: S, then the dP buffers (P and dS are written over them), then accumulators
  static constexpr uint32_t kColS = 0, kColX = 128, kColAcc = 128 + 128 * kNX;
  static_assert(kColAcc + kAccBufs * kAccCols <= kTmemCols, "tensor memory");
  static_assert(kBytes <= 232448, "shared memory");
};

// Four K steps of D (+)= A B with A (bf16 pairs) in tensor memory, 16 columns further on each step
// (8 of dS, then 8 of P), and B in shared memory, 16 rows further on each step.
__device__ __forceinline__ void mma_ts_rows_x4(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc,
                                               uint32_t acc0) {
  asm volatile(
      "{\n\t.reg .pred p0, p1;\n\t.reg .b64 b1, b2, b3;\n\t.reg .b32 a1, a2, a3;\n\t"
      "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 p1, %3, %3;\n\t"
      "add.u32 a1, %1, 16;\n\tadd.u64 b1, %2, 128;\n\t"
      "add.u32 a2, %1, 32;\n\tadd.u64 b2, %2, 256;\n\t"
      "add.u32 a3, %1, 48;\n\tadd.u64 b3, %2, 384;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a1], b1, %3, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a2], b2, %3, p1;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a3], b3, %3, p1;\n\t}"
      ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc0)
      : "memory");
}

// TOK: the token order decides which columns a row sees (causal, window in slot space).
template <int D, bool KEYS, bool TOK>
__global__ void __launch_bounds__(kThreads, 1)
bwd_tc_kernel(const __grid_constant__ BwdTcParams p, const __grid_constant__ CUtensorMap tm_q,
              const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
              const __grid_constant__ CUtensorMap tm_dy) {
  extern __shared__ __align__(1024) uint8_t smem[];
  using C = BCfg<D, KEYS>;
  constexpr bool kVec = KEYS || TOK;          // something travels with the column tiles
  constexpr int kMmaWarp = kRowWarps, kLoadWarp = kRowWarps + 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {
    if (threadIdx.x == 0) atomicCAS(p.status, SA_OK, SA_ERR_CUDA);
    return;
  }
  const uint32_t bar0 = sbase + C::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  volatile int* gave_up = reinterpret_cast<volatile int*>(smem + C::kOffMisc + 4);

  if (threadIdx.x == 0) {
    *gave_up = 0;
    for (int i = 0; i < C::kNumBars; ++i)
      mbar_init(bar(i), i >= C::kBarPReady && i < C::kBarAccFull ? C::kPArrivals
                        : i == C::kBarSRead || i >= C::kBarAccFree ? kRowWarps : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!p.late_wait) grid_dependency_wait(); // what earlier launches wrote may be read from here on
    note_skip(reinterpret_cast<volatile int*>(smem + C::kOffMisc + 8), p.status, p.abort_flag);
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dependents_launch();
  const uint32_t tmem = *tmem_slot;
  if (*reinterpret_cast<volatile int*>(smem + C::kOffMisc + 8)) grid_dependency_wait();
  SA_LEAVE_IF_SKIPPED(reinterpret_cast<volatile int*>(smem + C::kOffMisc + 8), kMmaWarp, tmem, kTmemCols)

  // An item: (batch, head of the row operand, row tile), the row tile innermost so that
  // neighbouring items meet the same column tiles in L2.
  const int H = KEYS ? p.Hkv : p.Hq;
  const int total = p.B * H * p.n_tiles;
  struct Item { int b, hr, hk, r0, cstart, T, iters; };
  auto span_of = [&](Item& i) {
    i.hk = KEYS || p.G == 1 ? i.hr : (int)__umulhi((uint32_t)i.hr, p.magic_g);
    column_range(p, i.r0, KEYS, &i.cstart, &i.T);
    i.iters = KEYS ? i.T * p.G : i.T;      // column tiles (times query heads of the group)
  };
  auto first_item = [&]() {
    Item i;
    const int bh = blockIdx.x / p.n_tiles;
    i.r0 = (blockIdx.x - bh * p.n_tiles) * kTile;
    i.b = bh / H;
    i.hr = bh - i.b * H;
    span_of(i);
    return i;
  };
  // gridDim.x items on (sixteen row warps would spend a thousand issue slots on the divisions)
  auto next_item = [&](Item i) {
    i.r0 += p.step_r0;
    i.hr += p.step_h;
    i.b += p.step_b;
    if (i.r0 >= p.n_tiles * kTile) { i.r0 -= p.n_tiles * kTile; ++i.hr; }
    if (i.hr >= H) { i.hr -= H; ++i.b; }
    span_of(i);
    return i;
  };

  // Registers move from the issuer and loading warps to the row threads.  Per lane over the 20
  // warps: 4 x 64 + 16 x 104 = 1920, all that the launch holds (20 x 96).  (The sum may never
  // exceed what the launch holds: a warpgroup asking for more waits for ever.)
  static_assert(4 * 64 + 16 * 104 == 20 * 96, "register split");
  if (warp >= kRowWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp == kLoadWarp && lane == 0) {
      // ------------------------------------------------------------- loads (one thread, TMA)
      // A tile is D / 64 boxes of 128 rows x 64 columns; rows outside the tensor read zeros and
      // are masked by the slot window.
      uint32_t u = 0, it = 0, r_on = 0, c1_on = 0, c2_on = 0;      // tiles started
      bool live = true;
      auto load_tile = [&](const CUtensorMap* tm, uint32_t dst, int row, int head, int b, uint32_t mb) {
#pragma unroll
        for (int c = 0; c < D / 64; ++c)
          tma_load_4d(dst + c * C::kChunkBytes, tm, 64 * c, row, head, b, mb);
      };
      Item i = first_item();
      for (int w_item = blockIdx.x; w_item < total && live; w_item += gridDim.x, ++it, i = next_item(i)) {
        const uint32_t rb = it % C::kRBufs;
        if (it >= (uint32_t)C::kRBufs)
          live = mbar_wait(bar(C::kBarREmpty + rb), (it / C::kRBufs - 1) & 1u, gave_up, p.status);
        if (!live) break;
        {
          const uint32_t dst = sbase + C::kOffR + rb * 2 * C::kTileBytes, mb = bar(C::kBarRFull + rb);
          mbar_expect_tx(mb, 2 * C::kTileBytes);
          load_tile(KEYS ? &tm_k : &tm_q, dst, p.o.left + i.r0, i.hr, i.b, mb);
          load_tile(KEYS ? &tm_v : &tm_dy, dst + C::kTileBytes, p.o.left + i.r0, i.hr, i.b, mb);
          r_on = it + 1;
        }
        int j = 0, hq = KEYS ? i.hk * p.G : i.hr;
        for (int x = 0; x < i.iters; ++x, ++u) {
          const uint32_t s = u % C::kC1, s2 = u % C::kC2;
          if (u >= (uint32_t)C::kC1)
            live = mbar_wait(bar(C::kBarC1Empty + s), (u / C::kC1 - 1) & 1u, gave_up, p.status);
          if (!live) break;
          const int col = i.cstart + j * kTile, hc = KEYS ? hq : i.hk;
          uint32_t mb = bar(C::kBarC1Full + s);
          mbar_expect_tx(mb, C::kTileBytes);
          load_tile(KEYS ? &tm_q : &tm_k, sbase + C::kOffC + s * C::kTileBytes, p.o.left + col, hc,
                    i.b, mb);
          c1_on = u + 1;
          if (kVec) {
            const uint32_t vb = bar(C::kBarVFull + s), vec = sbase + C::kOffVec + s * C::kVec * 4;
            mbar_expect_tx(vb, ((KEYS ? 2 : 0) + (TOK ? 1 : 0)) * kTile * 4);
            if (KEYS) {
              const size_t at = ((size_t)i.b * p.Hq + hq) * p.o.spitch + p.o.sleft + col;
              bulk_load(vec, p.lse2 + at, kTile * 4, vb);
              bulk_load(vec + kTile * 4, p.delta + at, kTile * 4, vb);
            }
            if (TOK)
              bulk_load(vec + C::kVecTok * 4, p.tok + (size_t)i.b * p.o.spitch + p.o.sleft + col,
                        kTile * 4, vb);
          }
          // (d = 64: C2's slot was freed together with C1's)
          // (from u = 1 on: a parity wait may not pass over a phase unseen)
          if (D == 128 && u > 0)
            live = KEYS ? mbar_wait(bar(C::kBarDpFull + 1), (u - 1) & 1u, gave_up, p.status)
                        : mbar_wait(bar(C::kBarSFull), (u - 1) & 1u, gave_up, p.status);
          if (!live) break;
          mb = bar(C::kBarC2Full + s2);
          mbar_expect_tx(mb, C::kTileBytes);
          load_tile(KEYS ? &tm_dy : &tm_v, sbase + C::kOffC2 + s2 * C::kTileBytes, p.o.left + col, hc,
                    i.b, mb);
          c2_on = u + 1;
          if (++j == i.T) { j = 0; ++hq; }
        }
      }
      // loads that were started but never consumed (only after a failed wait) must land before
      // the shared memory goes away: wait for them, again with a limit
      if (!live || *gave_up) {
        auto landed = [&](int index, uint32_t parity) {
          for (int tries = 0; tries < 100000; ++tries) {
            if (mbar_try(bar(index), parity)) break;
            __nanosleep(100);
          }
        };
        for (uint32_t x = r_on > (uint32_t)C::kRBufs ? r_on - C::kRBufs : 0u; x < r_on; ++x)
          landed(C::kBarRFull + x % C::kRBufs, (x / C::kRBufs) & 1u);
        for (uint32_t x = c1_on > (uint32_t)C::kC1 ? c1_on - C::kC1 : 0u; x < c1_on; ++x) {
          landed(C::kBarC1Full + x % C::kC1, (x / C::kC1) & 1u);
          if (kVec) landed(C::kBarVFull + x % C::kC1, (x / C::kC1) & 1u);
        }
        for (uint32_t x = c2_on > (uint32_t)C::kC2 ? c2_on - C::kC2 : 0u; x < c2_on; ++x)
          landed(C::kBarC2Full + x % C::kC2, (x / C::kC2) & 1u);
      }
    } else if (warp < kLoadWarp && lane == 0) {
      // ------------------------------------------------------------ MMA issuers (two threads)
      // Issuing runs at the pace of the products, and between two groups of products the issuing
      // thread spends some 300 cycles on waits and commits: one thread's fall into the other's
      // products.  Thread 0: the score products, one step ahead of the accumulations, across items
      // (rows = keys: S alone, whose columns are free once the row threads hold it).  Thread 1: the
      // accumulations (rows = keys: and dP of the next step behind them, over the P and dS that
      // they have read).
      constexpr uint32_t idesc_s = instr_desc(kTile, kTile, false), idesc_h = instr_desc(kTile, 64, false);
      constexpr uint32_t idesc_acc = instr_desc(kTile, D, true);
      constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
      constexpr uint32_t kLoK = (16u >> 4) << 16;                             // K-major operands
      constexpr uint32_t kLoMN = ((uint32_t)C::kChunkBytes >> 4) << 16;       // column tile as [k][n]
      constexpr uint32_t kBlock = C::kChunkBytes >> 4, kTileD = C::kTileBytes >> 4;
      const uint32_t r_lo = (sbase + C::kOffR) >> 4, c_lo = (sbase + C::kOffC) >> 4,
                     c2_lo = (sbase + C::kOffC2) >> 4;
      // X (128 x 128 or 64, fp32, tensor memory column col) = A B^T, both tiles K-major, K = D
      auto product = [&](uint32_t col, uint32_t a_lo, uint32_t b_lo, uint32_t idesc) {
        const uint64_t ad = desc64(a_lo | kLoK, kDescHi), bd = desc64(b_lo | kLoK, kDescHi);
        mma_ss_x4(tmem + col, ad, bd, idesc, 0u);
        if (D == 128) mma_ss_x4(tmem + col, ad + kBlock, bd + kBlock, idesc, 1u);
      };
      // acc (128 x D, tensor memory column col) += X (64 columns, from column xcol on) * 64 rows
      auto accumulate = [&](uint32_t col, uint32_t xcol, uint32_t b_lo, uint32_t acc0) {
        mma_ts_rows_x4(tmem + col, tmem + xcol, desc64(b_lo | kLoMN, kDescHi), idesc_acc, acc0);
      };
      bool ok = true;
      uint32_t u = 0, it = 0;                     // steps and items of this thread
      Item i = first_item();
      if (warp == kMmaWarp) {
        for (int w_item = blockIdx.x; w_item < total && ok; w_item += gridDim.x, ++it, i = next_item(i)) {
          const uint32_t rb = it % C::kRBufs;
          ok = mbar_wait(bar(C::kBarRFull + rb), (it / C::kRBufs) & 1u, gave_up, p.status);
          for (int x = 0; x < i.iters && ok; ++x, ++u) {
            const uint32_t s = u % C::kC1, s2 = u % C::kC2;
            ok = mbar_wait(bar(C::kBarC1Full + s), (u / C::kC1) & 1u, gave_up, p.status);
            if (ok && u > 0) ok = mbar_wait(bar(C::kBarSRead), (u - 1) & 1u, gave_up, p.status);
            if (!ok) break;
            tc_fence_after();
            product(C::kColS, r_lo + rb * 2 * kTileD, c_lo + s * kTileD, idesc_s);
            if (!KEYS) {
              // the dP buffer was read by the accumulation two steps ago, which freed C1
              if (u > 1)
                ok = mbar_wait(bar(C::kBarC1Empty + (u - 2) % C::kC1), ((u - 2) / C::kC1) & 1u, gave_up,
                               p.status);
              if (ok) ok = mbar_wait(bar(C::kBarC2Full + s2), (u / C::kC2) & 1u, gave_up, p.status);
              if (!ok) break;
              tc_fence_after();
              product(C::kColX + 128 * (u % 2), r_lo + (rb * 2 + 1) * kTileD, c2_lo + s2 * kTileD, idesc_s);
            }
            tc_commit(bar(C::kBarSFull));
          }
          // rows = keys: dP still reads the row operands, the other thread says when it is done
          if (!KEYS && ok) tc_commit(bar(C::kBarREmpty + rb));
        }
      } else if (!KEYS) {
        for (int w_item = blockIdx.x; w_item < total && ok; w_item += gridDim.x, ++it, i = next_item(i)) {
          const uint32_t ab = it % C::kAccBufs, acc = C::kColAcc + ab * C::kAccCols;
          if (it >= (uint32_t)C::kAccBufs)
            ok = mbar_wait(bar(C::kBarAccFree + ab), (it / C::kAccBufs - 1) & 1u, gave_up, p.status);
          for (int x = 0; x < i.iters && ok; ++x, ++u) {
            const uint32_t s = u % C::kC1, xc = C::kColX + 128 * (u % 2);
            ok = mbar_wait(bar(C::kBarC1Full + s), (u / C::kC1) & 1u, gave_up, p.status);
            if (ok) ok = mbar_wait(bar(C::kBarPReady + u % 2), (u / 2) & 1u, gave_up, p.status);
            if (!ok) break;
            tc_fence_after();
            accumulate(acc, xc, c_lo + s * kTileD, x > 0);                // dQ += dS K
            accumulate(acc, xc + 64, c_lo + s * kTileD + 512, 1u);
            tc_commit(bar(C::kBarC1Empty + s));
          }
          if (ok) tc_commit(bar(C::kBarAccFull + ab));
        }
      } else {
        // half hf of dP of step v, whose row operands are in buffer rb
        auto issue_dp = [&](uint32_t v, uint32_t rb, int hf) {
          product(C::kColX + 64 * hf, r_lo + (rb * 2 + 1) * kTileD, c2_lo + (v % C::kC2) * kTileD + 512 * hf,
                  idesc_h);
          tc_commit(bar(C::kBarDpFull + hf));
        };
        auto c2_wait = [&](uint32_t v) {
          ok = mbar_wait(bar(C::kBarC2Full + v % C::kC2), (v / C::kC2) & 1u, gave_up, p.status);
        };
        if ((int)blockIdx.x < total) {
          ok = mbar_wait(bar(C::kBarRFull), 0u, gave_up, p.status);
          if (ok) c2_wait(0);
          for (int hf = 0; hf < 2 && ok; ++hf) issue_dp(0, 0, hf);
        }
        for (int w_item = blockIdx.x; w_item < total && ok; w_item += gridDim.x, ++it, i = next_item(i)) {
          const uint32_t ab = it % C::kAccBufs, acc = C::kColAcc + ab * C::kAccCols;
          if (it >= (uint32_t)C::kAccBufs)
            ok = mbar_wait(bar(C::kBarAccFree + ab), (it / C::kAccBufs - 1) & 1u, gave_up, p.status);
          for (int x = 0; x < i.iters && ok; ++x, ++u) {
            const uint32_t s = u % C::kC1, c1 = c_lo + s * kTileD, c2 = c2_lo + (u % C::kC2) * kTileD;
            const bool last = x + 1 == i.iters;
            ok = mbar_wait(bar(C::kBarC1Full + s), (u / C::kC1) & 1u, gave_up, p.status);
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              if (ok) ok = mbar_wait(bar(C::kBarPReady + hf), u & 1u, gave_up, p.status);
              if (!ok) break;
              tc_fence_after();
              accumulate(acc + D, C::kColX + 64 * hf, c1 + 512 * hf, x > 0 || hf);       // dK += dS^T Q
              if (D == 128 && hf) tc_commit(bar(C::kBarC1Empty + s));
              accumulate(acc, C::kColX + 64 * hf + 8, c2 + 512 * hf, x > 0 || hf);       // dV += (g P)^T dY
              if (D == 64 && hf) tc_commit(bar(C::kBarC1Empty + s));
              if (!last) {
                if (hf == 0) c2_wait(u + 1);
                if (ok) issue_dp(u + 1, it % C::kRBufs, hf);
              }
            }
          }
          if (!ok) break;
          tc_commit(bar(C::kBarAccFull + ab));
          tc_commit(bar(C::kBarREmpty + it % C::kRBufs));     // S and dP of this item are over
          if (w_item + (int)gridDim.x < total) {
            const uint32_t nr = (it + 1) % C::kRBufs;
            ok = mbar_wait(bar(C::kBarRFull + nr), ((it + 1) / C::kRBufs) & 1u, gave_up, p.status);
            if (ok) c2_wait(u);
            for (int hf = 0; hf < 2 && ok; ++hf) issue_dp(u, nr, hf);
          }
        }
      }
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    // --------------------------------------------------------------------- row threads
    const int quad = warp & 3, cg = warp >> 2;          // TMEM lanes, 32-column group
    const int row = quad * 32 + lane, c0 = 32 * cg;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t stage = sbase + C::kOffStage + warp * (C::kStageRows * 64);
    const float inv_scale = 1.f / p.scale;
    uint32_t u = 0, it = 0;
    bool ok = true;
    auto arrive = [&](int i) {            // one arrival per warp, behind its tensor-memory accesses
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(i));
    };
    auto gate = [&](int hq) {
      return p.gate_logit ? 1.f / (1.f + __expf(-__ldcg(p.gate_logit + hq))) : 1.f;
    };
    // an item and what its rows need from memory, fetched one item ahead
    struct RowItem { Item i; int tok; float lse, delta, g; };
    auto fetch = [&](const Item& item) {
      RowItem r;
      r.i = item;
      const int slot = min(r.i.r0 + row, p.n - 1);
      r.tok = p.perm ? __ldcg(p.perm + (size_t)r.i.b * p.n + slot) : slot;
      r.g = gate(KEYS ? r.i.hk * p.G : r.i.hr);
      r.lse = r.delta = 0.f;
      if (!KEYS) {
        const size_t at = ((size_t)r.i.b * p.Hq + r.i.hr) * p.o.spitch + p.o.sleft + slot;
        r.lse = __ldcg(p.lse2 + at);
        r.delta = __ldcg(p.delta + at);
      }
      return r;
    };
    int done_tok = 0, done_b = 0, done_hr = 0, done_r0 = 0;     // the item before
    // Epilogue of the item before: it runs behind the first step of the next one, so that neither the
    // last accumulation's latency nor the row threads' stores leave the pipes idle.
    auto finish = [&]() {
      // Accumulator columns 32 at a time (rows = keys: dV, then dK), the pieces dealt to the column
      // groups.  A thread holds 64 bytes of a row; they are turned in the warp's staging rows, so
      // that 4 lanes store 64 consecutive bytes.  What the first branch left in the rows comes in
      // the same way, and is added before the one rounding.
      constexpr int kPieces = C::kAccCols / 32, kPass = 32 / C::kStageRows, kPer = C::kStageRows / 8;
      const int prow = lane >> 2, pc = lane & 3;
      auto turned = [&](int r) { return stage + r * 64 + ((pc ^ ((r >> 1) & 3)) << 4); };
      auto own = [&](int x8) {
        return stage + (lane & (C::kStageRows - 1)) * 64 + ((x8 ^ ((lane >> 1) & 3)) << 4);
      };
      const int64_t* st = KEYS ? p.ks : p.qs;
      const int64_t head = done_b * st[0] + done_hr * st[1] + 8 * pc;
      int64_t off[4];                       // this lane's rows prow, prow + 8, ...
      bool have[4];
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        off[y] = head + (int64_t)__shfl_sync(0xffffffffu, done_tok, 8 * y + prow) * st[2];
        have[y] = done_r0 + quad * 32 + 8 * y + prow < p.n;
      }
      auto out_of = [&](int piece) {
        return (__nv_bfloat16*)(!KEYS ? p.dq : piece < D / 32 ? p.dv : p.dk) + 32 * (piece % (D / 32));
      };
      uint4 old[4];
      auto load_old = [&](int piece) {
        const __nv_bfloat16* out = out_of(piece);
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          old[y] = make_uint4(0u, 0u, 0u, 0u);
          if (have[y]) old[y] = __ldcg(reinterpret_cast<const uint4*>(out + off[y]));
        }
      };
      if (p.late_wait) grid_dependency_wait();
      if (cg < kPieces && p.accumulate) load_old(cg);
      const uint32_t ab = (it - 1) % C::kAccBufs;
      ok = mbar_wait(bar(C::kBarAccFull + ab), ((it - 1) / C::kAccBufs) & 1u, gave_up, p.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) return;
      tc_fence_after();
#pragma unroll 1
      for (int piece = cg; piece < kPieces; piece += 4) {
        __nv_bfloat16* out = out_of(piece);
        uint32_t acc[32];
        tmem_ld32(trow + C::kColAcc + ab * C::kAccCols + 32 * piece, acc);
        tmem_wait_ld();
        if (piece + 4 >= kPieces) arrive(C::kBarAccFree + ab);
        if (p.accumulate) {
          if (piece != cg) load_old(piece);
#pragma unroll
          for (int hf = 0; hf < kPass; ++hf) {
            __syncwarp();
#pragma unroll
            for (int y = 0; y < kPer; ++y)
              sts128(turned(8 * y + prow), reinterpret_cast<const uint32_t(&)[4]>(old[kPer * hf + y]));
            __syncwarp();
            if (kPass == 1 || (lane >> 4) == hf) {
#pragma unroll
              for (int x8 = 0; x8 < 4; ++x8) {
                uint32_t v[4];
                lds128(v, own(x8));
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v[c]));
                  const float2 sum = __fadd2_rn(f, make_float2(__uint_as_float(acc[8 * x8 + 2 * c]),
                                                               __uint_as_float(acc[8 * x8 + 2 * c + 1])));
                  acc[8 * x8 + 2 * c] = __float_as_uint(sum.x);
                  acc[8 * x8 + 2 * c + 1] = __float_as_uint(sum.y);
                }
              }
            }
          }
        }
        uint32_t pk[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const __nv_bfloat162 h2 =
              __floats2bfloat162_rn(__uint_as_float(acc[2 * c]), __uint_as_float(acc[2 * c + 1]));
          pk[c] = *reinterpret_cast<const uint32_t*>(&h2);
        }
#pragma unroll
        for (int hf = 0; hf < kPass; ++hf) {
          __syncwarp();
          if (kPass == 1 || (lane >> 4) == hf) {
#pragma unroll
            for (int x8 = 0; x8 < 4; ++x8)
              sts128(own(x8), reinterpret_cast<const uint32_t(&)[4]>(pk[4 * x8]));
          }
          __syncwarp();
#pragma unroll
          for (int y = 0; y < kPer; ++y) {
            uint32_t v[4];
            lds128(v, turned(8 * y + prow));
            if (have[kPer * hf + y])
              *reinterpret_cast<uint4*>(out + off[kPer * hf + y]) = make_uint4(v[0], v[1], v[2], v[3]);
          }
        }
      }
      if (cg >= kPieces) arrive(C::kBarAccFree + ab);
    };
    RowItem nxt{};
    int w_item = blockIdx.x;
    if (w_item < total) nxt = fetch(first_item());
    Item i = nxt.i;
    int rtok = nxt.tok, hq = KEYS ? i.hk * p.G : i.hr, x = 0, j = 0;
    float lse_r = nxt.lse, delta_r = nxt.delta, g = nxt.g;
    while (true) {
      if (w_item < total) {
        const int rslot = i.r0 + row;
        if (x == 0 && p.accumulate && rslot < p.n) {
          // the epilogue will add to these rows: start bringing them into L2
          const int64_t* st = KEYS ? p.ks : p.qs;
          const int64_t at = i.b * st[0] + i.hr * st[1] + (int64_t)rtok * st[2];
#pragma unroll
          for (int piece = cg; piece < C::kAccCols / 32; piece += 4) {
            const __nv_bfloat16* out = (const __nv_bfloat16*)(!KEYS ? p.dq : piece < D / 32 ? p.dv : p.dk);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(out + at + 32 * (piece % (D / 32))));
          }
        }
        const uint32_t s = u % C::kC1;
        const float* vec = reinterpret_cast<const float*>(smem + C::kOffVec) + s * C::kVec + c0;
        const int cb = i.cstart + j * kTile;
        if (kVec) ok = mbar_wait(bar(C::kBarVFull + s), (u / C::kC1) & 1u, gave_up, p.status);
        if (ok) ok = mbar_wait(bar(C::kBarSFull), u & 1u, gave_up, p.status);
        ok = __all_sync(0xffffffffu, ok);   // the tensor-memory accesses below are warp-collective
        if (!ok) break;
        tc_fence_after();
        // P times scale: exp2(s scale2 - lse2), kept in registers
        uint32_t sv[32];
        tmem_ld32(trow + C::kColS + c0, sv);
        tmem_wait_ld();
        arrive(C::kBarSRead);
        const float2 sc2 = make_float2(p.scale2, p.scale2);
#pragma unroll
        for (int y = 0; y < 32; y += 4) {
          float4 l4 = make_float4(lse_r, lse_r, lse_r, lse_r);
          if (KEYS) l4 = *reinterpret_cast<const float4*>(vec + y);
          const float2 a = __ffma2_rn(make_float2(__uint_as_float(sv[y]), __uint_as_float(sv[y + 1])),
                                      sc2, make_float2(-l4.x, -l4.y));
          const float2 b = __ffma2_rn(make_float2(__uint_as_float(sv[y + 2]), __uint_as_float(sv[y + 3])),
                                      sc2, make_float2(-l4.z, -l4.w));
          sv[y] = __float_as_uint(exp2f(a.x));
          sv[y + 1] = __float_as_uint(exp2f(a.y));
          sv[y + 2] = __float_as_uint(exp2f(b.x));
          sv[y + 3] = __float_as_uint(exp2f(b.y));
        }
        if (TOK) {
          // rows = queries: hide later key tokens; rows = keys: earlier query tokens
          const int32_t* ct = reinterpret_cast<const int32_t*>(vec + C::kVecTok);
#pragma unroll
          for (int y = 0; y < 32; y += 4) {
            const int4 c4 = *reinterpret_cast<const int4*>(ct + y);
            if (KEYS ? c4.x < rtok : c4.x > rtok) sv[y] = 0u;
            if (KEYS ? c4.y < rtok : c4.y > rtok) sv[y + 1] = 0u;
            if (KEYS ? c4.z < rtok : c4.z > rtok) sv[y + 2] = 0u;
            if (KEYS ? c4.w < rtok : c4.w > rtok) sv[y + 3] = 0u;
          }
        }
        // Is every column of the tile in the window of every row of it?  (The window moves with the
        // row's slot, one column per row.)  If not: the columns [lo, hi] of this row.
        bool inside;
        if (p.full_range) inside = false;
        else if (p.one_sided)
          inside = KEYS ? cb >= i.r0 + kTile - 1 && cb + kTile <= min(i.r0 + p.w, p.n)
                        : cb >= max(i.r0 + kTile - p.w, 0) && cb + kTile - 1 <= i.r0;
        else
          inside = cb >= i.r0 + kTile - 1 - p.h && cb + kTile - 1 <= i.r0 + p.h &&
                   (!p.linear || (cb >= 0 && cb + kTile <= p.n));
        if (!inside) {
          int lo = -cb, hi = p.n - 1 - cb;                 // inside the sequence
          if (p.one_sided) {
            if (KEYS) {
              lo = rslot - cb;
              if (!p.full_range) hi = min(hi, rslot + p.w - 1 - cb);
            } else {
              if (!p.full_range) lo = max(lo, rslot - (p.w - 1) - cb);
              hi = min(hi, rslot - cb);
            }
          } else if (!p.full_range || p.linear) {
            const int a = rslot - p.h - cb, e = rslot + p.h - cb;
            lo = p.linear ? max(lo, a) : a;
            hi = p.linear ? min(hi, e) : e;
          }
          // as one bit per column: a bit test per element is cheaper than a comparison
          lo = max(lo - c0, 0);
          hi = min(hi - c0, 31);
          const uint32_t seen = hi < lo ? 0u : (0xffffffffu >> (31 - hi)) & (0xffffffffu << lo);
#pragma unroll
          for (int y = 0; y < 32; ++y)
            if (!(seen & (1u << y))) sv[y] = 0u;
        }
        // what the next item's rows need is on its way while this one's last step is worked on
        if (x + 1 == i.iters && w_item + (int)gridDim.x < total) nxt = fetch(next_item(i));
        // P times the gate for dV, then dP and dS; both go back as bf16 pairs over dP
        const uint32_t xa = trow + C::kColX + 128 * (u % C::kNX) + c0;
        uint32_t pk[KEYS ? 16 : 1];
        if constexpr (KEYS) {
          const float gp = g * inv_scale;
#pragma unroll
          for (int y = 0; y < 16; ++y) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(sv[2 * y]) * gp,
                                                            __uint_as_float(sv[2 * y + 1]) * gp);
            pk[y] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          ok = mbar_wait(bar(C::kBarDpFull + (cg >> 1)), u & 1u, gave_up, p.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
        }
        const float2 g2 = make_float2(g, g);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t dv[16], ds[8];
          tmem_ld16(xa + 16 * hf, dv);
          tmem_wait_ld();
#pragma unroll
          for (int y = 0; y < 16; y += 4) {
            const int e = 16 * hf + y;
            float4 d4 = make_float4(delta_r, delta_r, delta_r, delta_r);
            if (KEYS) d4 = *reinterpret_cast<const float4*>(vec + kTile + e);
            const float2 a = __ffma2_rn(g2, make_float2(__uint_as_float(dv[y]), __uint_as_float(dv[y + 1])),
                                        make_float2(-d4.x, -d4.y));
            const float2 b = __ffma2_rn(g2, make_float2(__uint_as_float(dv[y + 2]), __uint_as_float(dv[y + 3])),
                                        make_float2(-d4.z, -d4.w));
            const float2 sa = __fmul2_rn(make_float2(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])), a);
            const float2 sb = __fmul2_rn(make_float2(__uint_as_float(sv[e + 2]), __uint_as_float(sv[e + 3])), b);
            const __nv_bfloat162 ha = __floats2bfloat162_rn(sa.x, sa.y), hb = __floats2bfloat162_rn(sb.x, sb.y);
            ds[y / 2] = *reinterpret_cast<const uint32_t*>(&ha);
            ds[y / 2 + 1] = *reinterpret_cast<const uint32_t*>(&hb);
          }
          // over the 16 columns of dP just read: dS, then P
          tmem_st8(xa + 16 * hf, ds);
          if (KEYS) tmem_st8(xa + 16 * hf + 8, reinterpret_cast<const uint32_t(&)[8]>(pk[KEYS ? 8 * hf : 0]));
        }
        tmem_wait_st();
        // (with two dP buffers a quick warp may be here for step u + 1 before a slow one for step u)
        arrive(C::kBarPReady + (KEYS ? cg >> 1 : (int)(u & 1u)));
        ++u;
      }
      if (x == 0 && it > 0) finish();
      if (!ok || w_item >= total) break;
      ++x;
      if (++j == i.T) {
        j = 0;
        ++hq;
        if (KEYS && x < i.iters) g = gate(hq);
      }
      if (x == i.iters) {                   // on to the next item
        done_tok = rtok;
        done_b = i.b;
        done_hr = i.hr;
        done_r0 = i.r0;
        ++it;
        w_item += gridDim.x;
        i = nxt.i;
        rtok = nxt.tok;
        lse_r = nxt.lse;
        delta_r = nxt.delta;
        g = nxt.g;
        hq = KEYS ? i.hk * p.G : i.hr;
        x = j = 0;
      }
    }
  }

  // ----------------------------------------------------------------------- teardown
  if (p.late_wait) grid_dependency_wait();    // also where no item came to its epilogue
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------- preparation

struct PrepParams {
  const __nv_bfloat16 *q, *k, *v, *dy, *y[2];
  const int32_t *perm, *inv;          // of the branch the copies are for; null: token order
  const float *lse[2], *gate_logits;
  __nv_bfloat16 *cq, *cdy, *ck, *cv;  // copies; cq null: none
  int32_t* tok;                       // [B, spitch] of that branch, null: not needed
  float *lse2[2], *delta[2];          // per branch; null: this launch makes no statistics
  float* partials;                    // [2, B, Hq, chunks]
  const int* abort_flag;
  int B, Hq, Hkv, n, nbranch, chunks, copy_branch;
  float log2_scale;
  Order o[2];
  int64_t qs[3], ks[3];
};

constexpr int kPrepRows = 64;

// blockIdx.y: the Hq query heads (Delta, lse, copies of dY and Q), then the Hkv KV heads (copies of K and
// V; the first of them also writes the token list).  D / 8 lanes per row, 16 bytes each; rows are read
// in token order and stored at their slot.  HBM-bound: every tensor read once and written once.
template <int D>
__global__ void __launch_bounds__(256) prep_kernel(const __grid_constant__ PrepParams p) {
  __shared__ float wsum[2][8];
  constexpr int kCpr = D / 8, kRpp = 256 / kCpr;      // lanes per row, rows per pass
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = tid / kCpr, c = tid % kCpr;
  const int b = blockIdx.z, i0 = blockIdx.x * kPrepRows;
  const bool qside = (int)blockIdx.y < p.Hq, copies = p.cq != nullptr, stats = p.lse2[0] != nullptr;
  const int h = qside ? blockIdx.y : blockIdx.y - p.Hq;
  grid_dependency_wait();
  grid_dependents_launch();
  if (p.abort_flag && *p.abort_flag) return;          // an earlier check rejected perm/inv
  const Order& oc = p.o[p.copy_branch];
  // a row goes to its slot, and on to the other side where the circular window reaches over the end
  auto places = [&](int slot, int left, int (&at)[3], const Order& o) {
    at[0] = left + slot;
    const int reach = o.circular ? o.sleft : 0;
    at[1] = slot >= p.n - reach ? left + slot - p.n : -1;
    at[2] = slot < reach ? left + p.n + slot : -1;
  };
  auto store = [&](__nv_bfloat16* base, const int (&at)[3], const uint4& v) {
#pragma unroll
    for (int x = 0; x < 3; ++x)
      if (at[x] >= 0) *reinterpret_cast<uint4*>(base + (int64_t)at[x] * D + 8 * c) = v;
  };
  if (!qside) {
    if (!copies) return;
    const int64_t src = b * p.ks[0] + h * p.ks[1] + 8 * c;
    const int64_t dst = ((int64_t)b * p.Hkv + h) * oc.ext * D;
#pragma unroll
    for (int r = 0; r < kPrepRows / kRpp; ++r) {
      const int i = i0 + r * kRpp + sub;
      if (i >= p.n) break;
      const int slot = p.inv ? p.inv[(size_t)b * p.n + i] : i;
      const uint4 kk = __ldg(reinterpret_cast<const uint4*>(p.k + src + (int64_t)i * p.ks[2]));
      const uint4 vv = __ldg(reinterpret_cast<const uint4*>(p.v + src + (int64_t)i * p.ks[2]));
      int at[3];
      places(slot, oc.left, at, oc);
      store(p.ck + dst, at, kk);
      store(p.cv + dst, at, vv);
    }
    if (h == 0 && p.tok) {            // this block's share of the list, in slot order
      const int per = (oc.spitch + gridDim.x - 1) / gridDim.x;
      for (int e = blockIdx.x * per + tid; e < min((int)(blockIdx.x + 1) * per, oc.spitch); e += 256) {
        int slot = e - oc.sleft;
        if (oc.circular) { slot %= p.n; slot = slot < 0 ? slot + p.n : slot; }
        int t = 0;
        if (slot >= 0 && slot < p.n) t = p.perm ? p.perm[(size_t)b * p.n + slot] : slot;
        p.tok[(size_t)b * oc.spitch + e] = t;
      }
    }
    return;
  }
  const int64_t src = b * p.qs[0] + h * p.qs[1] + 8 * c;
  const int64_t dst = ((int64_t)b * p.Hq + h) * oc.ext * D;
  const size_t bh = (size_t)b * p.Hq + h;
  float g[2], part[2] = {0.f, 0.f};
  for (int x = 0; x < 2; ++x)
    g[x] = p.gate_logits ? 1.f / (1.f + __expf(-p.gate_logits[x * p.Hq + h])) : 1.f;
#pragma unroll
  for (int r = 0; r < kPrepRows / kRpp; ++r) {
    const int i = i0 + r * kRpp + sub;
    const bool have = i < p.n;
    const int64_t off = src + (int64_t)min(i, p.n - 1) * p.qs[2];
    int slot = i;
    if (have && p.inv) slot = p.inv[(size_t)b * p.n + i];
    const uint4 dy = __ldg(reinterpret_cast<const uint4*>(p.dy + off));
    if (stats) {
      const __nv_bfloat162* hd = reinterpret_cast<const __nv_bfloat162*>(&dy);
      for (int x = 0; x < p.nbranch; ++x) {
        const uint4 y = __ldg(reinterpret_cast<const uint4*>((x ? p.y[1] : p.y[0]) + off));
        const __nv_bfloat162* hy = reinterpret_cast<const __nv_bfloat162*>(&y);
        float dot = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 u = __bfloat1622float2(hd[e]), w = __bfloat1622float2(hy[e]);
          dot = fmaf(u.x, w.x, dot);
          dot = fmaf(u.y, w.y, dot);
        }
#pragma unroll
        for (int o = kCpr / 2; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        if (!have) dot = 0.f;
        if (c == 0) part[x] += dot;
        if (c == 0 && have) {
          const Order& o = p.o[x];
          int at[3];
          places(x == 0 ? slot : i, o.sleft, at, o);
          const float l2 = p.lse[x][bh * p.n + i] * kLog2e - p.log2_scale;
#pragma unroll
          for (int y3 = 0; y3 < 3; ++y3)
            if (at[y3] >= 0) {
              p.lse2[x][bh * o.spitch + at[y3]] = l2;
              p.delta[x][bh * o.spitch + at[y3]] = g[x] * dot;
            }
        }
      }
    }
    if (copies && have) {
      const uint4 qq = __ldg(reinterpret_cast<const uint4*>(p.q + off));
      int at[3];
      places(slot, oc.left, at, oc);
      store(p.cdy + dst, at, dy);
      store(p.cq + dst, at, qq);
    }
  }
  if (!stats) return;
  for (int x = 0; x < p.nbranch; ++x) {
    // what lies outside the sequence is read with the last tiles: it has to be finite
    const Order& o = p.o[x];
    const int end = o.sleft + p.n + (o.circular ? o.sleft : 0), lead = o.circular ? 0 : o.sleft;
    if (blockIdx.x == 0)
      for (int e = tid; e < lead + o.spitch - end; e += 256) {
        const size_t at = bh * o.spitch + (e < lead ? e : end + e - lead);
        p.lse2[x][at] = 0.f;
        p.delta[x][at] = 0.f;
      }
    const float s = warp_sum(part[x]);
    if (lane == 0) wsum[x][warp] = s;
  }
  __syncthreads();
  if (tid < p.nbranch) {
    float s = 0.f;
    for (int wv = 0; wv < 8; ++wv) s += wsum[tid][wv];
    p.partials[((size_t)tid * p.B * p.Hq + bh) * p.chunks + blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------------------- host

Order order_of(int n, int w, uint32_t flags, bool swa) {
  const MaskGeom g = make_geom(n, w, flags, swa);
  const bool full = g.one_sided ? false : 2ll * g.h + 1 >= n;
  Order o;
  o.circular = !g.one_sided && !g.linear && !full;
  o.left = o.circular ? g.h : 0;
  o.ext = n + 2 * o.left;
  o.sleft = g.one_sided || full ? 0 : g.h;
  o.spitch = (o.sleft + n + (o.circular ? g.h : 0) + 256 + 3) / 4 * 4;   // the last tiles read on
  return o;
}

struct BwdCarve {
  size_t partials, lse2[2], delta[2], tok, q, dy, k, v, total;
};

// Sized for circular windows, the largest case: the flags do not matter.
BwdCarve carve(int B, int Hq, int Hkv, int n, int d, int w) {
  const Order o[2] = {order_of(n, w, 0, false), order_of(n, w, 0, true)};
  BwdCarve c;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t r = at;
    at += (bytes + 255) / 256 * 256;
    return r;
  };
  c.partials = take((size_t)2 * B * Hq * ((n + kPrepRows - 1) / kPrepRows) * 4);
  int spitch = 0, ext = 0;
  for (int x = 0; x < 2; ++x) {
    c.lse2[x] = take((size_t)B * Hq * o[x].spitch * 4);
    c.delta[x] = take((size_t)B * Hq * o[x].spitch * 4);
    spitch = o[x].spitch > spitch ? o[x].spitch : spitch;
    ext = o[x].ext > ext ? o[x].ext : ext;
  }
  c.tok = take((size_t)B * spitch * 4);
  c.q = take((size_t)B * Hq * ext * d * 2);
  c.dy = take((size_t)B * Hq * ext * d * 2);
  c.k = take((size_t)B * Hkv * ext * d * 2);
  c.v = take((size_t)B * Hkv * ext * d * 2);
  c.total = at;
  return c;
}

template <int D, bool KEYS, bool TOK>
cudaError_t launch_side(const BwdTcParams& p, const CUtensorMap* tm, int sms, cudaStream_t st) {
  using C = BCfg<D, KEYS>;
  auto kernel = bwd_tc_kernel<D, KEYS, TOK>;
  const cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kBytes);
  if (e != cudaSuccess) return e;
  const int H = KEYS ? p.Hkv : p.Hq, total = p.B * H * p.n_tiles, grid = total < sms ? total : sms;
  BwdTcParams q = p;
  q.step_r0 = grid % p.n_tiles * kTile;
  q.step_h = grid / p.n_tiles % H;
  q.step_b = grid / p.n_tiles / H;
  q.magic_g = p.G > 1 ? (uint32_t)(((1ull << 32) + p.G - 1) / p.G) : 0u;
  return launch_dependent(kernel, dim3(grid), dim3(kThreads), C::kBytes, st, q, tm[0], tm[1], tm[2], tm[3]);
}

template <int D>
cudaError_t launch_branch(const BwdTcParams& p, bool tok, const CUtensorMap* tm, int sms,
                          cudaStream_t st) {
  cudaError_t e = tok ? launch_side<D, false, true>(p, tm, sms, st)
                      : launch_side<D, false, false>(p, tm, sms, st);
  BwdTcParams keys = p;
  keys.late_wait = 1;
  if (e == cudaSuccess)
    e = tok ? launch_side<D, true, true>(keys, tm, sms, st) : launch_side<D, true, false>(keys, tm, sms, st);
  if (e == cudaSuccess) bump_launches(2);
  return e;
}

bool bwd_tc_disabled() { return debug_option(SA_DEBUG_TENSOR_CORES) == 0; }

}  // namespace

bool tc_backward_supported(const BwdArgs& a, int dtype) {
  if (bwd_tc_disabled() || dtype != SA_BF16 || (a.d != 128 && a.d != 64)) return false;
  return a.n >= 1 && a.Hq + a.Hkv <= 65535 &&
         (int64_t)a.B * a.Hq * ((a.n + kTile - 1) / kTile) <= 0x3fffffff;
}

size_t tc_backward_ws_bytes(int B, int Hq, int Hkv, int n, int d, int w) {
  return d == 64 || d == 128 ? carve(B, Hq, Hkv, n, d, w).total : 0;
}

cudaError_t launch_bwd_tc(BwdArgs& a, cudaStream_t st) {
  const BwdCarve c = carve(a.B, a.Hq, a.Hkv, a.n, a.d, a.w);
  char* ws = (char*)a.ws;
  int* status = status_ptr();
  if (!status) return cudaErrorUnknown;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  a.partials = (float*)(ws + c.partials);
  a.chunks = (a.n + kPrepRows - 1) / kPrepRows;

  PrepParams pp{};
  pp.q = (const __nv_bfloat16*)a.q; pp.k = (const __nv_bfloat16*)a.k;
  pp.v = (const __nv_bfloat16*)a.v; pp.dy = (const __nv_bfloat16*)a.dy;
  pp.gate_logits = a.gate_logits;
  pp.partials = a.partials;
  pp.abort_flag = a.abort_flag;
  pp.B = a.B; pp.Hq = a.Hq; pp.Hkv = a.Hkv; pp.n = a.n; pp.nbranch = a.nbranch; pp.chunks = a.chunks;
  pp.log2_scale = log2f(a.scale);
  pp.cq = (__nv_bfloat16*)(ws + c.q); pp.cdy = (__nv_bfloat16*)(ws + c.dy);
  pp.ck = (__nv_bfloat16*)(ws + c.k); pp.cv = (__nv_bfloat16*)(ws + c.v);
  pp.tok = (int32_t*)(ws + c.tok);
  for (int i = 0; i < 3; ++i) { pp.qs[i] = a.qs[i]; pp.ks[i] = a.ks[i]; }
  for (int x = 0; x < a.nbranch; ++x) {
    pp.y[x] = (const __nv_bfloat16*)a.y_x[x];
    pp.lse[x] = a.lse_x[x];
    pp.o[x] = order_of(a.n, a.w, a.flags, x == 1);
  }
  auto prepare = [&](int branch, bool stats) {
    pp.copy_branch = branch;
    pp.perm = branch == 0 ? a.perm : nullptr;
    pp.inv = branch == 0 ? a.inv : nullptr;
    for (int x = 0; x < 2; ++x) {
      pp.lse2[x] = stats ? (float*)(ws + c.lse2[x]) : nullptr;
      pp.delta[x] = stats ? (float*)(ws + c.delta[x]) : nullptr;
    }
    const dim3 grid(a.chunks, a.Hq + a.Hkv, a.B);
    bump_launches();
    return launch_dependent(a.d == 128 ? prep_kernel<128> : prep_kernel<64>, grid, dim3(256), 0, st, pp);
  };

  for (int x = 0; x < a.nbranch; ++x) {
    const MaskGeom mg = make_geom(a.n, a.w, a.flags, x == 1);
    BwdTcParams p{};
    p.perm = x == 0 ? a.perm : nullptr;
    p.tok = pp.tok;
    p.lse2 = (const float*)(ws + c.lse2[x]);
    p.delta = (const float*)(ws + c.delta[x]);
    p.gate_logit = a.gate_logits ? a.gate_logits + (size_t)x * a.Hq : nullptr;
    p.dq = a.dq; p.dk = a.dk; p.dv = a.dv;
    p.accumulate = x > 0;
    p.status = status;
    p.abort_flag = a.abort_flag;
    p.B = a.B; p.Hq = a.Hq; p.Hkv = a.Hkv; p.G = a.Hq / a.Hkv; p.n = a.n; p.w = a.w;
    p.h = mg.h;
    p.linear = mg.linear; p.one_sided = mg.one_sided;
    p.full_range = mg.one_sided ? (a.w - 1 >= a.n) : (2ll * mg.h + 1 >= a.n);
    p.n_tiles = (a.n + kTile - 1) / kTile;
    p.o = pp.o[x];
    p.scale = a.scale;
    p.scale2 = a.scale * kLog2e;
    for (int i = 0; i < 3; ++i) { p.qs[i] = a.qs[i]; p.ks[i] = a.ks[i]; }
    // The one-sided SWA branch is read in place where the maps can express the strides;
    // sa_debug_set(SA_DEBUG_SWA_TILE_LOADS, 0) makes it use copies too.
    CUtensorMap tm[4];
    const bool in_place =
        x == 1 && mg.one_sided && debug_option(SA_DEBUG_SWA_TILE_LOADS) != 0 && aligned16(a.q) &&
        aligned16(a.k) && aligned16(a.v) && aligned16(a.dy) &&
        make_map_bhnd(&tm[0], a.q, a.B, a.Hq, a.n, a.d, a.qs) &&
        make_map_bhnd(&tm[1], a.k, a.B, a.Hkv, a.n, a.d, a.ks) &&
        make_map_bhnd(&tm[2], a.v, a.B, a.Hkv, a.n, a.d, a.ks) &&
        make_map_bhnd(&tm[3], a.dy, a.B, a.Hq, a.n, a.d, a.qs);
    p.late_wait = in_place;             // behind the first branch's kernels, not behind prep_kernel
    if (!in_place) {
      if ((e = prepare(x, x == 0)) != cudaSuccess) return e;
      const int64_t ext = p.o.ext;
      const int64_t cqs[3] = {a.Hq * ext * a.d, ext * a.d, a.d}, cks[3] = {a.Hkv * ext * a.d, ext * a.d, a.d};
      if (!make_map_bhnd(&tm[0], pp.cq, a.B, a.Hq, p.o.ext, a.d, cqs) ||
          !make_map_bhnd(&tm[1], pp.ck, a.B, a.Hkv, p.o.ext, a.d, cks) ||
          !make_map_bhnd(&tm[2], pp.cv, a.B, a.Hkv, p.o.ext, a.d, cks) ||
          !make_map_bhnd(&tm[3], pp.cdy, a.B, a.Hq, p.o.ext, a.d, cqs))
        return cudaErrorInvalidValue;
    }
    const bool tok = mg.causal && !mg.one_sided;        // the token order decides, not the slots
    e = a.d == 128 ? launch_branch<128>(p, tok, tm, sms, st) : launch_branch<64>(p, tok, tm, sms, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace sa

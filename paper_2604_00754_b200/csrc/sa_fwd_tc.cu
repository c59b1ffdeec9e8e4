// Fused permuted-window attention forward for sm_100a on the 5th-generation tensor cores.
//
// A persistent grid (one CTA per SM) walks a list of work items.  One item is two 128-row
// query tiles that share one stream of 128-key K/V tiles: two query heads of one GQA group
// over the same 128 slots (group size even), or two adjacent slot tiles of one head
// (otherwise).  S = Q K^T and O += P V run as tcgen05.mma with fp32 accumulators in tensor
// memory; the softmax (Eq. 1, with the mask of App. B applied per element) runs in registers,
// one thread per query row, and writes P back to tensor memory as the A operand of the second
// product.  The epilogue normalises, applies the gates of Eq. 5 when asked, and scatters each row
// to its original position.
//
// Where the tiles come from (template SRC):
//   kGather   rows of Q, K and V straight from HBM through perm, with 16-byte cp.async copies into
//             128-byte-swizzled tiles, so no permuted copy of any tensor exists.  A warp instruction
//             (512 bytes) is accepted every ~28 cycles per SM; TMA row gather needs ~70 cycles for
//             them.  (Copying K and V in slot order first and loading whole tiles by TMA was
//             built and timed: 875 against 859 us at 32/8 heads, n = 32768, w = 1024.)
//   kNatural  the one-sided SWA branch, whose rows are consecutive tokens: Q, K, V by TMA.
//   kOrdered  gathered as well, by the lists of sa_order.cu: the keys of a group of slots in token order,
//             query tiles by token, and one bit per row and key for the mask.
//
// Warp roles (384 threads): warps 0-3 softmax/epilogue of query tile 0, warps 4-7 of query tile
// 1, warp 8 MMA issuer and TMEM allocator (d = 64: warps 8 and 9, one per tile), then the
// producers.
// While one tile's softmax runs, the tensor core works on the other tile.  K and V tiles
// travel through one ring of shared-memory slots (K0 V0 K1 V1 ...), and every barrier is
// addressed by counters that run on across items, so the loads, products and epilogue of
// neighbouring items overlap.
//
// Every mbarrier wait is bounded; on expiry the CTA records SA_ERR_TIMEOUT in the device
// status word, stops issuing work, drains what it started and returns.
#include <type_traits>

#include "sa_fwd_tc.cuh"
#include "sa_gemm_common.cuh"
#include "sa_order.cuh"
#include "sa_tc_common.cuh"

namespace sa {
namespace {

constexpr int kTile = 128;           // query rows per tile and keys per K/V tile
constexpr uint32_t kTmemCols = 512;

enum Src { kGather = 0, kNatural = 1, kOrdered = 2 };
// Who does what.  At d = 64 each query tile has an issuing thread of its own: a tcgen05.commit holds
// its thread up for some 180 cycles, which the other tile's products fill (8 x 12 heads of 64,
// n = 4096, w = 128: SWA 114 -> 88 us, SA 144 -> 129; 256 heads of 64, n = 2048, w = 256: 165 -> 143
// and 239 -> 202).  At d = 128 the products take most of the time, and two issuers bring the two
// tiles into step, so that both softmaxes and then both products come at once (32/8 heads,
// n = 32768, w = 1024: SWA 600 -> 717 us): one issuer, which keeps them apart.
constexpr int kRowWarps = 8, kThreads = 32 * (kRowWarps + 4);
__host__ __device__ constexpr int issuers(int d) { return d == 64 ? 2 : 1; }

// Division of numbers below 2^30 by one known at the launch: a multiplication and a shift (Granlund and
// Montgomery, Division by invariant integers using multiplication, 1994), where the
// division proper costs every warp some twenty instructions, five times per item (2 x 16 heads of 128,
// n = 4096, w = 256 82 -> 75 us, its SWA branch 54 -> 50; 8 x 12 heads of 64, w = 128 132 -> 125 and 77 -> 71).
struct FastDiv {
  uint32_t mul = 0;
  int shift = 0;
  FastDiv() = default;
  explicit FastDiv(uint32_t d) {
    while ((1ull << shift) < d) ++shift;
    mul = (uint32_t)((((1ull << shift) - d) << 32) / d + 1);
  }
  __device__ __forceinline__ int of(int x) const { return (int)((__umulhi((uint32_t)x, mul) + (uint32_t)x) >> shift); }
};

struct TcParams {
  const void *q, *k, *v;
  const int32_t* perm;        // null for the SWA branch
  const float *rope_cos, *rope_sin;   // null, or [n, D/2] each: rotate Q and K rows on the way in
  void* y;
  void* y_branch;
  const void* y_other;
  float* lse;
  const float* gate_logits;
  int* status;
  const int* abort_flag;
  int B, Hq, Hkv, G, n, w, h;
  int causal, linear, one_sided, swa, full_range;
  int pair_heads;             // 1: tiles = two heads, same slots; 0: two slot tiles, one head
  int n_tiles;                // slot tiles of 128
  int items_per_kv;           // work items per (b, hk)
  int total_items;
  FastDiv by_items, by_kv, by_inner, by_full;   // items_per_kv, Hkv; make_geo / ordered_tiles
  float scale2;               // softmax scale * log2(e)
  OrderView order;            // kOrdered: what sa_order.cu made
  OrderGeom og;
  int64_t qs[3];              // element strides of q / y / y_branch / y_other: batch, head, token
  int64_t ks[3];              // element strides of k / v
};

// ------------------------------------------------------------------------- geometry

// Work item -> item of a KV head, KV head, sequence.
struct Place { int item, hk, b; };

__device__ __forceinline__ Place place_of(const TcParams& p, int w_item) {
  const int bh = p.by_items.of(w_item), b = p.by_kv.of(bh);
  return {w_item - bh * p.items_per_kv, bh - b * p.Hkv, b};
}

struct Geo {
  int q0[2];        // first slot of each query tile
  int hq[2];        // query head of each tile
  int valid[2];     // tile exists
  int kstart;       // virtual slot of the first key of K/V tile 0
  int T;            // K/V tiles in the stream
  int Tt[2];        // kOrdered: those that each query tile meets, the first of the stream
};

// Score blocks whose first key kv lies in [*lo, *hi] are wholly inside the window of every query
// of the tile at q0: only the token order can hide keys there.  Empty (lo > hi) where every block
// is to be tested element by element.
__device__ __forceinline__ void inner_range(const TcParams& p, int q0, int kw, int* lo, int* hi) {
  const int q1 = q0 + kTile - 1;
  *lo = 1;
  *hi = 0;
  if (p.full_range) return;
  if (p.one_sided) {
    *lo = max(0, q1 - (p.w - 1));
    *hi = q0 - kw + 1;
  } else if (q1 < p.n) {
    *lo = q1 - p.h;
    *hi = q0 + p.h - kw + 1;
    if (p.linear) {
      *lo = max(*lo, 0);
      *hi = min(*hi, p.n - kw);
    }
  }
}

// The score blocks h (keys kstart + (h << shift) and the 2^shift - 1 after it) that hold a key of the window of the
// query tile at q0: a contiguous range [first, last], empty (first > last) for a tile
// that does not exist.
__device__ __forceinline__ void active_halves(const TcParams& p, int q0, int valid, int kstart,
                                              int H, int shift, int* first, int* last) {
  const int q1 = q0 + kTile - 1;
  int lo, hi;   // keys of interest: some key of the half >= lo, its first key <= hi
  if (p.full_range) { lo = 0; hi = p.n - 1; }
  else if (p.one_sided) { lo = q0 - (p.w - 1); hi = q1; }
  else { lo = q0 - p.h; hi = q1 + p.h; }
  const int f = max(0, (lo - kstart) >> shift), l = min(H - 1, (hi - kstart) >> shift);
  *first = valid ? f : (1 << 30);
  *last = valid ? l : -1;
}

__device__ __forceinline__ Geo make_geo(const TcParams& p, int item, int hk) {
  Geo g;
  if (p.pair_heads) {
    const int pairs = p.G / 2;
    const int tile = p.by_inner.of(item), pr = item - tile * pairs;
    g.q0[0] = g.q0[1] = tile * kTile;
    g.hq[0] = hk * p.G + 2 * pr;
    g.hq[1] = g.hq[0] + 1;
    g.valid[0] = g.valid[1] = 1;
  } else {
    const int tpairs = (p.n_tiles + 1) / 2;
    const int hh = p.by_inner.of(item), tp = item - hh * tpairs;
    g.q0[0] = 2 * tp * kTile;
    g.q0[1] = g.q0[0] + kTile;
    g.hq[0] = g.hq[1] = hk * p.G + hh;
    g.valid[0] = 1;
    g.valid[1] = g.q0[1] < p.n;
  }
  const int qfirst = g.q0[0];
  const int qlast = min((g.valid[1] ? g.q0[1] : g.q0[0]) + kTile - 1, p.n - 1);
  int kend;
  if (p.full_range) {
    g.kstart = 0;
    kend = p.n - 1;
  } else if (p.one_sided) {
    g.kstart = max(qfirst - (p.w - 1), 0);
    kend = qlast;
  } else if (p.linear) {
    g.kstart = max(qfirst - p.h, 0);
    kend = min(qlast + p.h, p.n - 1);
  } else {
    g.kstart = qfirst - p.h;
    kend = qlast + p.h;
  }
  g.T = (kend - g.kstart + kTile) / kTile;
  return g;
}

// kOrdered: the query tiles of an item.  Within a KV head those that meet the most blocks come first, class
// by class, so that the classes fall evenly on the CTAs; the last rounds of the last KV head are of the
// shortest.
__device__ __forceinline__ void ordered_tiles(const TcParams& p, int item, int hk, int (&tile)[2],
                                              int (&hq)[2]) {
  const int per_unit = p.pair_heads ? 1 : 2, units = p.og.slots / (kTile * per_unit);
  const int full = p.n_tiles / (units * per_unit);                   // groups with all their tiles
  const int heads = p.pair_heads ? p.G / 2 : p.G;
  const int x = p.by_inner.of(item), hh = item - x * heads;
  int unit = x;
  if (x < full * units) {
    const int cls = p.by_full.of(x);
    unit = (x - cls * full) * units + units - 1 - cls;
  }
  tile[0] = unit * per_unit;
  tile[1] = tile[0] + per_unit - 1;
  hq[0] = hk * p.G + (p.pair_heads ? 2 * hh : hh);
  hq[1] = hq[0] + (p.pair_heads ? 1 : 0);
}

// kOrdered: q0 are places in the tokens of the query tiles, keys count from the start of the group's list.
__device__ __forceinline__ Geo ordered_geo(const TcParams& p, int item, int hk, int b) {
  Geo g;
  int tile[2];
  ordered_tiles(p, item, hk, tile, g.hq);
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    g.q0[t] = tile[t] * kTile;
    g.valid[t] = tile[t] < p.n_tiles;
    g.Tt[t] = g.valid[t] ? __ldcg(p.order.tiles + (size_t)b * p.n_tiles + tile[t]) : 0;
  }
  g.kstart = 0;
  g.T = max(g.Tt[0], g.Tt[1]);
  return g;
}

__device__ __forceinline__ int actual_slot(const TcParams& p, int v) {
  if (p.full_range || p.linear || p.one_sided) return min(max(v, 0), p.n - 1);
  v %= p.n;
  return v < 0 ? v + p.n : v;
}

// ------------------------------------------------------------------- shared memory

// K and V tiles have a ring of kRing slots each.  The products of step j read V_j and K_{j+1} last,
// so one commit per step frees both (a tcgen05.commit holds the tensor pipe up for some 180
// cycles): free events are numbered through, one for K_0 of an item and one per step.  A token list
// is written with K, one tile more than the ring deep: K of tile u + kTok is loaded behind the
// event of K of tile u + 1, i.e. behind P V of tile u and so behind its softmax, the last reader.
// Four slots at d = 128 leave 32 KB in which the epilogue turns rows held by one thread each into
// coalesced stores.
template <int D>
struct Cfg {
  static constexpr int kTileBytes = kTile * D * 2;
  static constexpr int kChunkBytes = kTile * 128;
  static constexpr int kSlots = D == 128 ? 4 : 8;
  static constexpr int kRing = kSlots / 2, kEvents = 2 * kRing, kTok = kRing + 1;
  // Q buffers (two query tiles each).  With two (d = 64 leaves the room) the next item's Q is
  // loaded, and its first scores are issued, while the row threads still finish this item:
  // short items (narrow windows) otherwise idle a quarter of their time at every item start.
  static constexpr int kQBufs = D == 128 ? 1 : 2;
  static constexpr int kOffQ = 0;
  static constexpr int kOffRing = kQBufs * 2 * kTileBytes;
  static constexpr int kOffStage = kOffRing + kSlots * kTileBytes;  // 8 warps x 32 rows x 128 bytes
  static constexpr int kOffTok = kOffStage + 8 * 4096;
  static constexpr int kOffBar = kOffTok + kTok * kTile * 4;
  // mbarriers, 8 bytes each
  static constexpr int kBarQFull = 0, kBarQEmpty = kQBufs, kBarSlotFull = 2 * kQBufs,
                       kBarFree = kBarSlotFull + kSlots, kBarTokFull = kBarFree + kEvents,
                       kBarSFull = kBarTokFull + kTok, kBarPReady = kBarSFull + 4,
                       kBarPvDone = kBarPReady + 4, kBarODone = kBarPvDone + 2,
                       kNumBars = kBarODone + 2;
  static constexpr int kOffMisc = kOffBar + kNumBars * 8;   // TMEM base address, gave_up flag
  static constexpr int kBytes = kOffMisc + 16;
  static constexpr uint32_t kColO = 256;                     // O_t at 256 + t*D; S_t at t*128
  static_assert(kBytes <= 232448, "shared memory");
};

// Which free event tells that the slot of tile gt may be loaded: the tile R before it was tile c of
// item i in running numbers; its K is freed by event c + i and its V by the next one.
template <int R>
struct Ring {
  uint32_t items[R + 1];          // items of the last tiles, newest first
  __device__ __forceinline__ Ring() {
#pragma unroll
    for (int x = 0; x <= R; ++x) items[x] = 0;
  }
  __device__ __forceinline__ void advance(uint32_t it) {
#pragma unroll
    for (int x = R; x > 0; --x) items[x] = items[x - 1];
    items[0] = it;
  }
  __device__ __forceinline__ uint32_t k_event(uint32_t gt) const { return gt - R + items[R]; }
};

// ------------------------------------------------------------------------- kernel

// D: head dimension.  KB: keys per score block, 64 or 128.  With 64 a tile's S columns hold
// two blocks and the scores run two blocks ahead of the softmax; with 128 a block is the
// whole K/V tile and the next scores of a tile follow its P V.
// SRC: where the tiles come from, see the top of the file.
// ROPE (kGather only): the gather producers rotate the rows of Q and K by their tokens' angles
// (rotary position embedding with ORIGINAL positions, Sec. 4.2 / App. B) after the copies have
// landed.
// COMBINE: the epilogue reads the other branch's finished rows and applies the gates of Eq. 5
// (the instantiation of the launch that closes a gated forward); without it the kernel
// carries no gate code at all.
template <int D, int KB, int SRC, bool ROPE = false, bool COMBINE = false>
__global__ void __launch_bounds__(kThreads, 1)
fwd_tc_kernel(const __grid_constant__ TcParams p, const __grid_constant__ CUtensorMap tm_q,
              const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v) {
  extern __shared__ __align__(1024) uint8_t smem[];
  using C = Cfg<D>;
  constexpr int kHalf = KB;             // keys per score block
  constexpr int NB = kTile / KB;        // score blocks per K/V tile = S buffers per query tile
  constexpr int kShift = KB == 64 ? 6 : 7;
  constexpr int kIssuers = issuers(D);
  constexpr int kMmaWarp = kRowWarps, kLoadWarp = kRowWarps + kIssuers;
  constexpr int kGWarps = 4 - kIssuers;      // the loading warps, when rows are gathered
  constexpr bool kRows = SRC != kNatural;    // tiles are gathered row by row
  static_assert(SRC != kOrdered || (KB == 128 && !ROPE && !COMBINE), "ordered lists");
  auto geo_of = [&](int item, int hk, int b) {
    if constexpr (SRC == kOrdered) return ordered_geo(p, item, hk, b);
    else return make_geo(p, item, hk);
  };
  auto active_of = [&](const Geo& g, int t, int H, int shift, int* first, int* last) {
    if constexpr (SRC == kOrdered) { *first = 0; *last = (t ? g.Tt[1] : g.Tt[0]) - 1; }
    else active_halves(p, t ? g.q0[1] : g.q0[0], t ? g.valid[1] : g.valid[0], g.kstart, H, shift, first, last);
  };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {                        // the swizzled tiles need 1024-byte alignment
    if (threadIdx.x == 0) atomicCAS(p.status, SA_OK, SA_ERR_CUDA);
    return;
  }
  const uint32_t bar0 = sbase + C::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  volatile int* gave_up = reinterpret_cast<volatile int*>(smem + C::kOffMisc + 4);

  // The second branch of a gated pass: the launch before is the first branch, which waited for all
  // before it and lets this one start when its last CTAs run.  Q, K and V (read through L2 by TMA) are
  // complete by then, so only the epilogue, which reads the first branch's rows, waits for it: this
  // branch's CTAs fill the SMs that the first one's last round leaves idle.
  // Gated, 32/8 heads of 128: n = 700, w = 256 38.5 -> 36.0 us; n = 8192, w = 1024 457 -> 449.
  constexpr bool kLateWait = COMBINE && SRC == kNatural;
  if (threadIdx.x == 0) {
    *gave_up = 0;
    for (int i = 0; i < C::kNumBars; ++i) {
      int count = 1;
      if (i >= C::kBarPReady && i < C::kBarPvDone) count = kTile;
      if ((i < C::kBarQEmpty || (i >= C::kBarSlotFull && i < C::kBarFree)) && kRows)
        count = 32 * kGWarps;
      if ((i >= C::kBarQEmpty && i < C::kBarSlotFull) || (i >= C::kBarFree && i < C::kBarTokFull))
        count = kIssuers;
      mbar_init(bar(i), count);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!kLateWait) grid_dependency_wait();   // what earlier launches wrote may be read from here on
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
  if (kLateWait && *reinterpret_cast<volatile int*>(smem + C::kOffMisc + 8)) grid_dependency_wait();
  SA_LEAVE_IF_SKIPPED(reinterpret_cast<volatile int*>(smem + C::kOffMisc + 8), kMmaWarp, tmem, kTmemCols)

  // Registers move from the issuer and producer warps to the row threads, which hold a whole score
  // row each.  Per lane over the 12 warps: 4 x 56 + 8 x 224 = 4 x 72 + 8 x 216 = 2016, all that the
  // launch holds (12 x 168).  The four warps of a warpgroup must ask for the same count, so the issuing
  // warps and the producer warps go down together.  72 where rows are gathered: at 56 the gathering
  // warps spilled their tokens, and what they reload queues behind their own copies (SA, 8 x 12 heads of 64,
  // n = 4096, w = 128 128 -> 105 us; 2 x 16 heads of 128, w = 256 76 -> 71); the row threads keep their
  // 128 scores at 216 as at 224 (at 208 they spilled).  (The sum may never exceed what the
  // launch holds: a warpgroup asking for more waits for ever.)
  constexpr int kLow = kRows ? 72 : 56, kHigh = kRows ? 216 : 224;
  static_assert(4 * kLow + kRowWarps * kHigh == (kRowWarps + 4) * 168, "register split");
  if (warp >= kRowWarps) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kLow));
  if (SRC == kNatural && warp == kLoadWarp) {
    // ------------------------------------------------------ tile loads by TMA (one thread)
    // A tile is D / 64 boxes of 128 rows x 64 columns that the TMA unit lays out in the same
    // swizzled form a gather produces; no producer instructions compete with the softmax warps.
    // The token index is a dimension of the map, so rows past the sequence are filled with zeros
    // (never with whatever follows in memory, which could be NaN and would poison P V through
    // 0 * NaN); the window mask does not let them count and their outputs are not stored.  No
    // token lists: the one-sided rule tests slots only.
    if (lane == 0) {
      uint32_t gt = 0, it = 0, q_armed = 0xffffffffu, k_on = 0, v_on = 0;   // tiles started
      Ring<C::kRing> ring;
      bool live = true;
      auto load_tile = [&](const CUtensorMap* tm, uint32_t dst, int tok, int head, int b,
                           uint32_t mb) {
#pragma unroll
        for (int c = 0; c < D / 64; ++c)
          tma_load_4d(dst + c * C::kChunkBytes, tm, 64 * c, tok, head, b, mb);
      };
      auto wait_free = [&](uint32_t e) {
        return mbar_wait(bar(C::kBarFree + e % C::kEvents), (e / C::kEvents) & 1u, gave_up, p.status);
      };
      for (int w_item = blockIdx.x; w_item < p.total_items && live; w_item += gridDim.x, ++it) {
        const Place at = place_of(p, w_item);
        const int item = at.item, hk = at.hk, b = at.b;
        const Geo g = make_geo(p, item, hk);
        for (int j = 0; j < g.T; ++j, ++gt) {
          const uint32_t pr = gt % C::kRing;
          ring.advance(it);
          if (gt >= (uint32_t)C::kRing) live = wait_free(ring.k_event(gt));
          if (!live) break;
          const int row = g.kstart + j * kTile;
          const uint32_t dst = sbase + C::kOffRing + 2 * pr * C::kTileBytes;
          uint32_t mb = bar(C::kBarSlotFull + 2 * pr);
          mbar_expect_tx(mb, C::kTileBytes);
          load_tile(&tm_k, dst, row, hk, b, mb);
          k_on = gt + 1;
          if (j == 0) {
            const uint32_t qb = it % C::kQBufs;
            if (it >= (uint32_t)C::kQBufs)
              live = mbar_wait(bar(C::kBarQEmpty + qb), (it / C::kQBufs - 1) & 1u, gave_up, p.status);
            if (!live) break;
            mbar_expect_tx(bar(C::kBarQFull + qb), 2 * C::kTileBytes);
            q_armed = it;
#pragma unroll
            for (int t = 0; t < 2; ++t)
              load_tile(&tm_q, sbase + C::kOffQ + (2 * qb + t) * C::kTileBytes, g.q0[t], g.hq[t], b,
                        bar(C::kBarQFull + qb));
          }
          if (gt >= (uint32_t)C::kRing) live = wait_free(ring.k_event(gt) + 1);
          if (!live) break;
          mb = bar(C::kBarSlotFull + 2 * pr + 1);
          mbar_expect_tx(mb, C::kTileBytes);
          load_tile(&tm_v, dst + C::kTileBytes, row, hk, b, mb);
          v_on = gt + 1;
        }
      }
      // loads that were started but never consumed (only after a failed wait) must land
      // before the shared memory goes away: wait for them, again with a limit
      if (!live || *gave_up) {
        auto landed = [&](int index, uint32_t parity) {
          for (int tries = 0; tries < 100000; ++tries) {
            if (mbar_try(bar(index), parity)) break;
            __nanosleep(100);
          }
        };
        for (uint32_t u = k_on > (uint32_t)C::kRing ? k_on - C::kRing : 0u; u < k_on; ++u)
          landed(C::kBarSlotFull + 2 * (u % C::kRing), (u / C::kRing) & 1u);
        for (uint32_t u = v_on > (uint32_t)C::kRing ? v_on - C::kRing : 0u; u < v_on; ++u)
          landed(C::kBarSlotFull + 2 * (u % C::kRing) + 1, (u / C::kRing) & 1u);
        if (q_armed != 0xffffffffu)
          landed(C::kBarQFull + q_armed % C::kQBufs, (q_armed / C::kQBufs) & 1u);
      }
    }
  } else if (kRows && warp >= kLoadWarp) {
    // ------------------------------------------------------------------ gather producers
    // Each 16-byte piece of a row goes from global memory to its swizzled place in shared
    // memory with cp.async; one warp instruction moves kRpi whole rows.
    constexpr int kCpr = D / 8;            // 16-byte pieces per row
    constexpr int kRpi = 32 / kCpr;        // rows per warp instruction
    constexpr int kPt = 32 * kGWarps;      // producer threads
    const int ptid = threadIdx.x - 32 * kLoadWarp, pw = warp - kLoadWarp;
    const int sub = lane / kCpr, chunk = lane % kCpr;
    const uint32_t dst_lane = (uint32_t)(chunk >> 3) * C::kChunkBytes;
    const __nv_bfloat16* qg = (const __nv_bfloat16*)p.q;
    const __nv_bfloat16* kg = (const __nv_bfloat16*)p.k;
    const __nv_bfloat16* vg = (const __nv_bfloat16*)p.v;
    int32_t* const ktok_base = reinterpret_cast<int32_t*>(smem + C::kOffTok);
    uint32_t gt = 0, it = 0;
    Ring<C::kRing> ring;
    // A tile's barrier counts one arrival per producer thread, triggered by the hardware
    // when that thread's copies have landed (cp.async.mbarrier.arrive.noinc), so issuing
    // never waits for data.  The consumer publishes the data to the tensor core's proxy
    // (fence.proxy.async) after its wait.
    auto signal = [&](uint32_t mb) {
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(mb) : "memory");
    };
    auto wait_free = [&](uint32_t e) {     // a failure sets *gave_up
      mbar_wait(bar(C::kBarFree + e % C::kEvents), (e / C::kEvents) & 1u, gave_up, p.status);
    };
    // The rows of a tile are dealt to the gathering warps in groups of kRpi.  A warp takes four
    // of its groups per pass: the swizzle term of each of the four is the same in every pass (it
    // only depends on the group modulo 8 / kRpi), so it is prepared once per thread and the
    // destination of a copy is one addition away from the pass's base.
    constexpr int kGroups = kTile / kRpi;
    uint32_t sw[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r7 = ((pw + kGWarps * k) * kRpi + sub) & 7;
      sw[k] = (uint32_t)(((chunk & 7) ^ r7) << 4) + (uint32_t)(kGWarps * k * kRpi * 128);
    }
    auto gather = [&](const __nv_bfloat16* base, int64_t tok_stride, auto tok_of, uint32_t dst_tile) {
      // token and token stride are both below 2^31: one 32 x 32 -> 64 bit multiply per row
      const uint32_t ts = (uint32_t)tok_stride * 2u;      // bytes
      const char* src0 = reinterpret_cast<const char*>(base + chunk * 8);
      const uint32_t dst0 = dst_tile + dst_lane + sub * 128;
      int grp = pw, nth = 0;                       // group, the nth of this warp
#pragma unroll 1
      for (; grp + 3 * kGWarps < kGroups; grp += 4 * kGWarps, nth += 4) {
        const uint32_t d = dst0 + grp * (kRpi * 128);
        uint32_t tok[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) tok[k] = (uint32_t)tok_of((grp + kGWarps * k) * kRpi + sub, nth + k);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const char* src = src0 + (uint64_t)tok[k] * ts;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + sw[k]), "l"(src)
                       : "memory");
        }
      }
#pragma unroll 1
      for (; grp < kGroups; grp += kGWarps, ++nth) {
        const int r = grp * kRpi + sub;
        const char* src = src0 + (uint64_t)(uint32_t)tok_of(r, nth) * ts;
        const uint32_t dst = dst_tile + dst_lane + r * 128 + (((chunk & 7) ^ (r & 7)) << 4);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
      }
    };
    // Barrier over the gathering warps that also agrees on whether anyone in the CTA
    // has given up: every producer thread leaves the loops at the same point.
    auto group_sync_stop = [&]() {
      uint32_t any;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.u32 q, %1, 0;\n\t"
          "bar.red.or.pred p, 1, %2, q;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(any)
          : "r"((uint32_t)*gave_up), "n"(kPt)
          : "memory");
      return any != 0;
    };

    // ROPE: rows of a landed tile that this warp copied are turned in place.  A lane owns the
    // 16-byte piece `chunk` of its rows; the piece half a row further on holds the partner
    // dimensions (c <-> c + D/2).  Every lane reads both pieces, the warp meets, every lane
    // writes its own piece back: out = own * cos -/+ partner * sin (first / second half), in
    // fp32, rounded once to bf16 -- the arithmetic of the stand-alone rotation pass.
    auto rotate = [&](auto tok_of, uint32_t tile) {
      constexpr int kHalfC = kCpr / 2;
      const int pc = chunk < kHalfC ? chunk + kHalfC : chunk - kHalfC;
      const int fc = chunk < kHalfC ? chunk : chunk - kHalfC;
      const float sgn = chunk < kHalfC ? -1.f : 1.f;
      for (int grp = pw; grp < kGroups; grp += kGWarps) {
        const int r = grp * kRpi + sub;
        const uint32_t rb = tile + r * 128;
        const uint32_t a_own = rb + (uint32_t)(chunk >> 3) * C::kChunkBytes +
                               (uint32_t)(((chunk & 7) ^ (r & 7)) << 4);
        const uint32_t a_oth = rb + (uint32_t)(pc >> 3) * C::kChunkBytes +
                               (uint32_t)(((pc & 7) ^ (r & 7)) << 4);
        uint32_t own[4], oth[4];
        lds128(own, a_own);
        lds128(oth, a_oth);
        const size_t at = (size_t)tok_of(r) * (D / 2) + 8 * fc;
        __syncwarp();
        uint32_t res[4];
#pragma unroll
        for (int hx = 0; hx < 2; ++hx) {           // four dimensions at a time: few live registers
          const float4 c4 = *reinterpret_cast<const float4*>(p.rope_cos + at + 4 * hx);
          const float4 s4 = *reinterpret_cast<const float4*>(p.rope_sin + at + 4 * hx);
          const float co[4] = {c4.x, c4.y, c4.z, c4.w}, si[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const int w = 2 * hx + x;
            const float2 o = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&own[w]));
            const float2 t = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&oth[w]));
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(
                fmaf(o.x, co[2 * x], sgn * (t.x * si[2 * x])),
                fmaf(o.y, co[2 * x + 1], sgn * (t.y * si[2 * x + 1])));
            res[w] = *reinterpret_cast<const uint32_t*>(&h2);
          }
        }
        sts128(a_own, res);
      }
    };
    auto commit_group = [&]() { asm volatile("cp.async.commit_group;" ::: "memory"); };

    bool live = true;
    for (int w_item = blockIdx.x; w_item < p.total_items && live; w_item += gridDim.x, ++it) {
      const Place at = place_of(p, w_item);
      const int item = at.item, hk = at.hk, b = at.b;
      const Geo g = geo_of(item, hk, b);
      const int32_t* perm = p.perm ? p.perm + (size_t)b * p.n : nullptr;
      const int32_t* list = nullptr;           // kOrdered: the group's keys
      if constexpr (SRC == kOrdered) {
        perm = p.order.q + (size_t)b * p.n_tiles * kTile;
        list = p.order.k + ((size_t)b * p.og.groups + g.q0[0] / p.og.slots) * p.og.pitch;
      }
      const uint32_t q_bar = bar(C::kBarQFull + it % C::kQBufs);
      const uint32_t q_dst = sbase + C::kOffQ + 2 * (it % C::kQBufs) * C::kTileBytes;
      auto q_tok = [&](int t, int r) {
        const int slot = min((t ? g.q0[1] : g.q0[0]) + r, (SRC == kOrdered ? p.n_tiles * kTile : p.n) - 1);
        return perm ? perm[slot] : slot;
      };
      const __nv_bfloat16* kb = kg + b * p.ks[0] + hk * p.ks[1];
      const __nv_bfloat16* vb = vg + b * p.ks[0] + hk * p.ks[1];
      auto key_tok = [&](int j, int r) {
        if constexpr (SRC == kOrdered) return list[j * kTile + r];
        const int slot = actual_slot(p, g.kstart + j * kTile + r);
        return perm ? perm[slot] : slot;
      };
      // The tokens of a query tile come all at once, at most two per lane: those of the rows that this
      // warp moves, in its order.  Fetched group by group, each four groups waited for a load of their
      // own, six times some 700 cycles per tile with the tensor core idle (SA, 32/8 heads of 128: n = 32768,
      // w = 1024 833 -> 780 us, over lists 790 -> 629; n = 10007, w = 512 184 -> 166).  Not where rows of
      // d = 128 are turned on the way: with two tokens more to hold, those warps spill 108 bytes for 60
      // (sa_forward_rope, 8/2 heads, n = 4096, w = 1024 110.7 us for 108.3; d = 64, 64 bytes for 56: 12 heads,
      // w = 128 76.5 for 78.1).
      constexpr bool kRowTokens = !(ROPE && D == 128);
      static_assert((kGroups + kGWarps - 1) / kGWarps * kRpi <= 64, "two tokens per lane");
      int qt[2];
      auto fetch_q = [&](int t) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int e = 32 * x + lane;
          qt[x] = q_tok(t, min((pw + kGWarps * (e / kRpi)) * kRpi + e % kRpi, kTile - 1));
        }
      };
      if constexpr (kRowTokens) fetch_q(0);
      // tokens are fetched one tile ahead of their use
      int tk0 = key_tok(0, ptid), tk1 = ptid + kPt < kTile ? key_tok(0, ptid + kPt) : 0;
      for (int j = 0; j < g.T; ++j, ++gt) {
        // ---- K_j and the tokens of its keys
        const uint32_t pr = gt % C::kRing;
        ring.advance(it);
        if (gt >= (uint32_t)C::kRing) wait_free(ring.k_event(gt));
        int32_t* ktok = ktok_base + (gt % C::kTok) * kTile;
        ktok[ptid] = tk0;
        if (ptid + kPt < kTile) ktok[ptid + kPt] = tk1;
        if (group_sync_stop()) { live = false; break; }
        if (SRC == kGather && ptid == 0) mbar_arrive(bar(C::kBarTokFull + gt % C::kTok));
        const uint32_t k_dst = sbase + C::kOffRing + 2 * pr * C::kTileBytes;
        const uint32_t k_bar = bar(C::kBarSlotFull + 2 * pr);
        auto tok_of = [&](int r, int = 0) { return ktok[r]; };
        gather(kb, p.ks[2], tok_of, k_dst);
        if (ROPE) commit_group(); else signal(k_bar);
        if (j + 1 < g.T) {
          tk0 = key_tok(j + 1, ptid);
          if (ptid + kPt < kTile) tk1 = key_tok(j + 1, ptid + kPt);
        }
        if (j == 0) {
          // ---- Q of this item, once the products of the previous item no longer read it
          if (it >= (uint32_t)C::kQBufs)
            mbar_wait(bar(C::kBarQEmpty + it % C::kQBufs), (it / C::kQBufs - 1) & 1u, gave_up, p.status);
          if (group_sync_stop()) { live = false; break; }
#pragma unroll 1
          for (int t = 0; t < 2; ++t) {
            if (kRowTokens && t && !p.pair_heads) fetch_q(1);
            gather(qg + b * p.qs[0] + (t ? g.hq[1] : g.hq[0]) * p.qs[1], p.qs[2],
                   [&](int r, int nth) {
                     if constexpr (!kRowTokens) return q_tok(t, r);
                     return __shfl_sync(0xffffffffu, nth < 32 / kRpi ? qt[0] : qt[1], (nth * kRpi + sub) & 31);
                   },
                   q_dst + t * C::kTileBytes);
          }
          if (ROPE) commit_group(); else signal(q_bar);
        }
        // ---- V_j
        if (gt >= (uint32_t)C::kRing) {
          wait_free(ring.k_event(gt) + 1);
          if (group_sync_stop()) { live = false; break; }
        }
        gather(vb, p.ks[2], tok_of, k_dst + C::kTileBytes);
        signal(bar(C::kBarSlotFull + 2 * pr + 1));
        if (ROPE) {
          // K_j (and Q at the start of an item) have landed once at most the V_j copies are
          // still under way; turn the rows, publish them to the tensor core's proxy, arrive
          commit_group();
          asm volatile("cp.async.wait_group 1;" ::: "memory");
          __syncwarp();
          rotate(tok_of, k_dst);
          if (j == 0) {
            rotate([&](int r) { return q_tok(0, r); }, q_dst);
            rotate([&](int r) { return q_tok(1, r); }, q_dst + C::kTileBytes);
          }
          fence_proxy_async();
          mbar_arrive(k_bar);
          if (j == 0) mbar_arrive(q_bar);
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // nothing in flight when the CTA leaves
  } else if (warp < kMmaWarp + kIssuers) {
    // ----------------------------------------------------------------------- MMA issuers
    // One thread (or one per query tile) feeds the tensor core, so every instruction between two
    // tcgen05.mma counts: the descriptors are built from words prepared outside the loops and the
    // K steps are fully unrolled with immediate offsets.
    //
    // With 64-key blocks scores are produced into the two halves of a tile's S columns, two
    // half-steps ahead of the softmax: while the softmax works on one half, the other half
    // already holds the next scores.
    if (lane == 0) {
      constexpr uint32_t idesc_qk = instr_desc(kTile, kHalf, false);
      constexpr uint32_t idesc_pv = instr_desc(kTile, D, true);
      // shared-memory descriptor words (128-byte swizzle, 1024 bytes between 8-row groups)
      constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
      constexpr uint32_t kLoK = (16u >> 4) << 16;                          // K-major operands
      constexpr uint32_t kLoV = ((uint32_t)C::kChunkBytes >> 4) << 16;     // V: next 64 columns
      constexpr int kN = 2 / kIssuers;          // query tiles of this thread: tb .. tb + kN - 1
      const int tb = kIssuers == 2 ? warp - kMmaWarp : 0;
      const uint64_t q_first = desc64(((sbase + C::kOffQ) >> 4) | kLoK, kDescHi);
      uint32_t q_item = 0;                      // this item's Q buffer, in descriptor units
      const uint32_t ring_lo = (sbase + C::kOffRing) >> 4;
      bool ok = true;
      uint32_t gt = 0, it = 0;
      uint32_t pcnt[kN][2] = {};                // p_ready waits so far; indices are compile-time
      // slot of K (v = 0) or V (v = 1) of tile pair u
      auto slot_lo = [&](uint32_t u, int v) {
        return ring_lo + (2 * (u % C::kRing) + v) * (C::kTileBytes >> 4);
      };
      auto slot_wait = [&](uint32_t u, int v) {
        return mbar_wait(bar(C::kBarSlotFull + 2 * (u % C::kRing) + v), (u / C::kRing) & 1u, gave_up,
                         p.status);
      };
      // S(t, half b) = Q_t K^T over keys [64 b, 64 b + 64) of the K tile at k_lo
      auto issue_qk = [&](int t, int b, uint32_t k_lo) {
        const uint64_t qd = q_first + q_item + t * (C::kTileBytes >> 4);
        const uint64_t kd = desc64((k_lo + b * (kHalf * 128 >> 4)) | kLoK, kDescHi);
        const uint32_t d = tmem + t * 128 + b * kHalf;
        mma_ss_x4(d, qd, kd, idesc_qk, 0u);
        if (D == 128)   // columns 64..127 live one 16 KB block further on
          mma_ss_x4(d, qd + (C::kChunkBytes >> 4), kd + (C::kChunkBytes >> 4), idesc_qk, 1u);
        tc_commit(bar(C::kBarSFull + 2 * t + b));
      };
      // O_t += P(t, half b) V over the same 64 keys of the V tile at v_lo
      auto issue_pv = [&](int t, int b, uint32_t v_lo, uint32_t acc0) {
        const uint64_t vd = desc64((v_lo + b * (kHalf * 128 >> 4)) | kLoV, kDescHi);
        mma_ts_x4(tmem + C::kColO + t * D, tmem + t * 128 + b * kHalf, vd, idesc_pv, acc0);
        if (KB == 128)
          mma_ts_x4(tmem + C::kColO + t * D, tmem + t * 128 + 32, vd + 512, idesc_pv, 1u);
        // With 128-key blocks the next scores of this tile follow this product in the pipe, and
        // their "S full" says that it is over as well.
        if (NB == 2) tc_commit(bar(C::kBarPvDone + t));
      };
      for (int w_item = blockIdx.x; w_item < p.total_items && ok; w_item += gridDim.x, ++it) {
        const Place at = place_of(p, w_item);
        const Geo g = geo_of(at.item, at.hk, at.b);
        const int H = NB * g.T;         // score blocks of this item
        // half-steps [first, last] that each query tile takes part in (a contiguous range)
        int first[kN], last[kN];
        uint32_t started[kN] = {};
#pragma unroll
        for (int x = 0; x < kN; ++x) {
          active_of(g, tb + x, H, kShift, &first[x], &last[x]);
        }
        const uint32_t qb = it % C::kQBufs;
        q_item = qb * (2 * C::kTileBytes >> 4);
        ok = mbar_wait(bar(C::kBarQFull + qb), (it / C::kQBufs) & 1u, gave_up, p.status);
        if (ok) ok = slot_wait(gt, 0);
        if (!ok) break;
        fence_proxy_async();
        tc_fence_after();
        const uint32_t k0 = slot_lo(gt, 0);
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int x = 0; x < kN; ++x)
            if (first[x] <= b && last[x] >= b) issue_qk(tb + x, b, k0);
        uint32_t event = gt + it;       // frees K_0; event + 1 + j: K_{j+1} and V_j
        tc_commit(bar(C::kBarFree + event % C::kEvents));
        if (g.T == 1) tc_commit(bar(C::kBarQEmpty + qb));
        for (int j = 0; j < g.T && ok; ++j, ++gt) {
          const bool more = j + 1 < g.T;
          // first touch of V_j and of K_{j+1}: both are needed within this step
          ok = slot_wait(gt, 1);
          if (ok && more) ok = slot_wait(gt + 1, 0);
          if (!ok) break;
          fence_proxy_async();
          const uint32_t v_lo = slot_lo(gt, 1), k_lo = slot_lo(gt + 1, 0);
          // (half, tile) by (half, tile): P V of half-step h, then Q K^T of half-step h + NB
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int x = 0; x < kN; ++x) {
              const int h = NB * j + b, t = tb + x;
              if (ok && h >= first[x] && h <= last[x]) {
                ok = mbar_wait(bar(C::kBarPReady + 2 * t + b), pcnt[x][b] & 1u, gave_up, p.status);
                if (ok) {
                  ++pcnt[x][b];
                  tc_fence_after();
                  issue_pv(t, b, v_lo, started[x]);
                  started[x] = 1;
                  if (h == last[x]) tc_commit(bar(C::kBarODone + t));
                }
              }
              if (ok && more && h + NB >= first[x] && h + NB <= last[x]) issue_qk(t, b, k_lo);
            }
          if (!ok) break;
          ++event;
          tc_commit(bar(C::kBarFree + event % C::kEvents));
          if (j + 2 == g.T) tc_commit(bar(C::kBarQEmpty + qb));
        }
      }
    }
    __syncwarp();
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kHigh));
    // ------------------------------------------------- softmax and epilogue
    const int t = warp / 4, quad = warp & 3;
    const int row = quad * 32 + lane;                  // 0..127 == TMEM lane
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t s_addr = tmem + lane_addr + t * 128;
    const uint32_t o_addr = tmem + lane_addr + C::kColO + t * D;
    uint32_t s_cnt0 = 0, s_cnt1 = 0, o_cnt = 0, pv_cnt = 0, gt = 0;
    bool ok = true;

    for (int w_item = blockIdx.x; w_item < p.total_items && ok; w_item += gridDim.x) {
      const Place at = place_of(p, w_item);
      const int b = at.b;
      int q0, hq, kstart, first, last, in_lo, in_hi;
      const uint32_t gt0 = gt;
      {
        const Geo g = geo_of(at.item, at.hk, b);
        q0 = t ? g.q0[1] : g.q0[0];
        hq = t ? g.hq[1] : g.hq[0];
        kstart = g.kstart;
        gt += g.T;
        active_of(g, t, NB * g.T, kShift, &first, &last);
      }
      if (first > last) continue;           // no such tile
      if (SRC != kOrdered) inner_range(p, q0, kHalf, &in_lo, &in_hi);
      const int qv = q0 + row;
      const bool row_valid = qv < p.n;
      int q_tok = 0;
      if (SRC != kOrdered && row_valid) q_tok = p.perm ? p.perm[(size_t)b * p.n + qv] : qv;
      const uint4* bits = nullptr;            // kOrdered: what this row sees, block by block
      uint4 seen_next = make_uint4(0u, 0u, 0u, 0u);
      if constexpr (SRC == kOrdered) {
        const size_t place = (size_t)b * p.n_tiles * kTile + qv;
        q_tok = __ldcg(p.order.q + place);
        bits = p.order.bits + (place - row) * p.og.blocks + row;
        seen_next = __ldcg(bits);
      }
      const int qcmp = (p.causal && !p.one_sided) ? q_tok : 0x7fffffff;
      if (COMBINE && row_valid) {
        // the epilogue will read the other branch's row: start bringing it into L2 now
        const __nv_bfloat16* orow = (const __nv_bfloat16*)p.y_other + b * p.qs[0] + hq * p.qs[1] +
                                    (int64_t)q_tok * p.qs[2];
#pragma unroll
        for (int x = 0; x < D / 64; ++x)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(orow + 64 * x));
      }
      float m = -INFINITY, l = 0.f;
      bool started = false;

      for (int h = first; h <= last; ++h) {
        const int kv = kstart + h * kHalf;
        const int hb = h & (NB - 1);
        const uint32_t tg = gt0 + (h >> (NB - 1));
        // the token list belongs to the whole 128-key tile: wait for it at its first half only
        if (SRC == kGather && (hb == 0 || h == first))
          ok = mbar_wait(bar(C::kBarTokFull + tg % C::kTok), (tg / C::kTok) & 1u, gave_up, p.status);
        if (ok)
          ok = mbar_wait(bar(C::kBarSFull + 2 * t + hb), (hb ? s_cnt1 : s_cnt0) & 1u, gave_up,
                         p.status);
        ok = __all_sync(0xffffffffu, ok);   // the tensor-memory loads below are warp-collective
        if (!ok) break;
        s_cnt0 += 1 - hb;
        s_cnt1 += hb;
        tc_fence_after();

        const uint32_t sh_addr = s_addr + hb * kHalf;
        uint32_t sr[kHalf];
        // Gathered branch: 32 columns are masked while the next 32 are on their way (SA, 32/8 heads of
        // 128, n = 10007, w = 1024: 277 -> 273 us).  The other, with next to no masks, takes all at once.
        constexpr int kFirst = kRows ? 32 : kHalf;
#pragma unroll
        for (int c = 0; c < kFirst / 32; ++c)
          tmem_ld32(sh_addr + 32 * c, reinterpret_cast<uint32_t(&)[32]>(sr[32 * c]));
        tmem_wait_ld();
        auto next32 = [&](int c) {
          if (kRows) {
            if (c > 0) tmem_wait_ld();
            if (c + 32 < kHalf)
              tmem_ld32(sh_addr + c + 32, reinterpret_cast<uint32_t(&)[32]>(sr[(c + 32) % kHalf]));
          }
        };
        // the token order: an integer compare and a select per score
        const uint8_t* tokens = smem + C::kOffTok + ((tg % C::kTok) * kTile + hb * kHalf) * 4;
        auto token_mask = [&](int c) {
          if constexpr (SRC == kGather) {
            const int4 kt = *reinterpret_cast<const int4*>(tokens + 4 * c);
            if (kt.x > qcmp) sr[c] = 0xff800000u;
            if (kt.y > qcmp) sr[c + 1] = 0xff800000u;
            if (kt.z > qcmp) sr[c + 2] = 0xff800000u;
            if (kt.w > qcmp) sr[c + 3] = 0xff800000u;
          }
        };
        // plain SWA: keys wholly before the queries need no causal test (no wrap inside)
        const bool tokens_matter =
            p.causal && !p.one_sided && !(p.swa && kv >= 0 && kv + kHalf - 1 <= q0);
        if constexpr (SRC == kOrdered) {
          const uint4 seen4 = seen_next;
          const uint32_t seen[4] = {seen4.x, seen4.y, seen4.z, seen4.w};
#pragma unroll
          for (int c0 = 0; c0 < kHalf; c0 += 32) {
            next32(c0);
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (!(seen[c0 / 32] & (1u << c))) sr[c0 + c] = 0xff800000u;
          }
        } else if (kv >= in_lo && kv <= in_hi) {
          if (tokens_matter) {
#pragma unroll
            for (int c0 = 0; c0 < kHalf; c0 += 32) {
              next32(c0);
#pragma unroll
              for (int c = c0; c < c0 + 32; c += 4) token_mask(c);
            }
          } else {
#pragma unroll
            for (int c0 = 0; c0 < kHalf; c0 += 32) next32(c0);
          }
        } else {
          // visible columns form one interval [lo, hi] of this row, cut by the token order
          int lo, hi;
          if (p.one_sided) { lo = p.full_range ? -kv : qv - (p.w - 1) - kv; hi = qv - kv; }
          else if (p.full_range && !p.linear) { lo = -kv; hi = p.n - 1 - kv; }
          else { lo = qv - p.h - kv; hi = qv + p.h - kv; }
          if (p.linear || p.full_range || p.one_sided) {
            lo = max(lo, -kv);
            hi = min(hi, p.n - 1 - kv);
          }
          // as one bit per column: a bit test and a select per score, where comparing the column
          // with both ends took a subtraction more (one-sided branch, 8 x 12 heads of 64, n = 4096,
          // w = 128: 86 -> 77 us; 2 x 16 heads of 128, w = 256: 56 -> 51, its SA branch 83 -> 79)
#pragma unroll
          for (int c0 = 0; c0 < kHalf; c0 += 32) {
            next32(c0);
            const int a = max(lo - c0, 0), e = min(hi - c0, 31);
            const uint32_t seen = e < a ? 0u : (0xffffffffu >> (31 - e)) & (0xffffffffu << a);
#pragma unroll
            for (int c = c0; c < c0 + 32; c += 4) {
              token_mask(c);
#pragma unroll
              for (int x = c; x < c + 4; ++x)
                if (!(seen & (1u << (x - c0)))) sr[x] = 0xff800000u;
            }
          }
        }
        float mx0 = __uint_as_float(sr[0]), mx1 = __uint_as_float(sr[1]);
#pragma unroll
        for (int c = 2; c < kHalf; c += 4) {
          mx0 = max3(mx0, __uint_as_float(sr[c]), __uint_as_float(sr[c + 1]));
          if (c + 2 < kHalf)
            mx1 = max3(mx1, __uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3]));
        }
        const float m_new = fmaxf(m, fmaxf(mx0, mx1));
        // Lazy rescaling: keep the old reference maximum while the new one is within 2^8.
        const bool grow = (m_new - m) * p.scale2 > 8.f || (m == -INFINITY && m_new > -INFINITY);
        if (!started) {
          m = m_new;
        } else if (__any_sync(0xffffffffu, grow)) {
          // O is still being accumulated by the previous P V: wait for it before touching O
          // (128-key blocks: these scores were issued behind that product, so it is over)
          if (NB == 2) {
            ok = mbar_wait(bar(C::kBarPvDone + t), (pv_cnt - 1) & 1u, gave_up, p.status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
          }
          const float f = grow ? exp2f((m - m_new) * p.scale2) : 1.f;
          if (grow) { l *= f; m = m_new; }
#pragma unroll
          for (int c = 0; c < D / 8; ++c) {            // 8 columns at a time: the scores are live
            uint32_t raw[8];
            tmem_ld8(o_addr + 8 * c, raw);
            tmem_wait_ld();
#pragma unroll
            for (int x = 0; x < 8; ++x) raw[x] = __float_as_uint(__uint_as_float(raw[x]) * f);
            tmem_st8(o_addr + 8 * c, raw);
          }
        }
        started = true;
        const float neg = (m == -INFINITY) ? 0.f : -m * p.scale2;
        const float2 sc2 = make_float2(p.scale2, p.scale2), ng2 = make_float2(neg, neg);
        float2 lsum = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kHalf / 32; ++c) {
          uint32_t pk[16];          // 32 probabilities, two bf16 per word
#pragma unroll
          for (int x = 0; x < 16; ++x) {
            const float2 a = __ffma2_rn(make_float2(__uint_as_float(sr[32 * c + 2 * x]),
                                                    __uint_as_float(sr[32 * c + 2 * x + 1])),
                                        sc2, ng2);
            const float2 e = make_float2(exp2f(a.x), exp2f(a.y));
            lsum = __fadd2_rn(lsum, e);
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(e.x, e.y);
            pk[x] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          tmem_st16(sh_addr + 16 * c, pk);
        }
        l += lsum.x + lsum.y;
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar(C::kBarPReady + 2 * t + hb));
        // (here, where the warp waits anyway)
        if constexpr (SRC == kOrdered)
          if (h < last) seen_next = __ldcg(bits + (size_t)(h + 1) * kTile);
        ++pv_cnt;                           // the issuer answers every arrive with one P V
      }
      if (!ok) break;

      // ------------------------------------------------------------------- epilogue
      // A thread holds a row, so storing from the registers would touch 32 lines per instruction
      // (4000 cycles per item).  Each warp turns 32 rows x 64 columns at a time in 4 KB of shared
      // memory (16-byte pieces, swizzled by the row number): 8 lanes then store 128 consecutive
      // bytes of a row, 4 rows per instruction.  The other branch's rows come in the same way.
      // Measured with the ring of the loads (8 x 12 heads of 64, n = 4096, w = 128, gated):
      // 346 -> 307 us; 32/8 heads of 128, n = 32768, w = 1024: 1711 -> 1605.
      constexpr int kPieces = 8;                       // 16-byte pieces of 64 columns = row groups
      const int prow = lane >> 3, pc = lane & 7;       // piece pc of rows prow, prow + 4, ...
      const uint32_t stage = sbase + C::kOffStage + warp * 4096;
      const uint32_t own_row = stage + lane * 128;
      auto turned = [&](int i) {                       // this lane's piece of row 4 i + prow
        const int r = 4 * i + prow;
        return stage + r * 128 + ((pc ^ (r & 7)) << 4);
      };
      const int64_t base = b * p.qs[0] + hq * p.qs[1] + pc * 8;
      int64_t at_row[kPieces];
      bool have[kPieces];
#pragma unroll
      for (int i = 0; i < kPieces; ++i) {
        at_row[i] = base + (int64_t)__shfl_sync(0xffffffffu, q_tok, 4 * i + prow) * p.qs[2];
        have[i] = q0 + quad * 32 + 4 * i + prow < p.n;
      }
      if (kLateWait) grid_dependency_wait();
      uint4 oth[COMBINE ? kPieces : 1];
      auto load_other = [&](int hf) {
        if constexpr (COMBINE) {
#pragma unroll
          for (int i = 0; i < kPieces; ++i) {
            oth[i] = make_uint4(0u, 0u, 0u, 0u);
            if (have[i])
              oth[i] = __ldcg(reinterpret_cast<const uint4*>((const __nv_bfloat16*)p.y_other +
                                                             at_row[i] + 64 * hf));
          }
        }
      };
      load_other(0);
      float g_this = 1.f, g_other = 0.f;
      if (COMBINE) {
        const float s_sa = 1.f / (1.f + __expf(-p.gate_logits[hq]));
        const float s_swa = 1.f / (1.f + __expf(-p.gate_logits[p.Hq + hq]));
        g_this = p.swa ? s_swa : s_sa;
        g_other = p.swa ? s_sa : s_swa;
      }

      ok = mbar_wait(bar(C::kBarODone + t), o_cnt & 1u, gave_up, p.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      ++o_cnt;
      tc_fence_after();
      const float inv_l = 1.f / l;
#pragma unroll
      for (int hf = 0; hf < D / 64; ++hf) {
        uint32_t raw[64];
        tmem_ld32(o_addr + 64 * hf, reinterpret_cast<uint32_t(&)[32]>(raw[0]));
        tmem_ld32(o_addr + 64 * hf + 32, reinterpret_cast<uint32_t(&)[32]>(raw[32]));
        if (COMBINE && !p.y_branch) {
          // the gates act on unrounded local rows: the other row goes to the row's thread
#pragma unroll
          for (int i = 0; i < kPieces; ++i) sts128(turned(i), reinterpret_cast<uint32_t(&)[4]>(oth[i]));
          __syncwarp();
        }
        tmem_wait_ld();
        // piece x of this thread's row: 8 output columns, normalised
#pragma unroll
        for (int x = 0; x < kPieces; ++x) {
          float o[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) o[c] = __uint_as_float(raw[8 * x + c]) * inv_l;
          const uint32_t at = own_row + ((x ^ (lane & 7)) << 4);
          uint32_t st[4];
          if (COMBINE && !p.y_branch) {
            lds128(st, at);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float2 w = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&st[c]));
              o[2 * c] = fmaf(g_other, w.x, o[2 * c] * g_this);
              o[2 * c + 1] = fmaf(g_other, w.y, o[2 * c + 1] * g_this);
            }
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(o[2 * c], o[2 * c + 1]);
            st[c] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          sts128(at, st);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
          uint32_t v[4];
          lds128(v, turned(i));
          const int64_t e = at_row[i] + 64 * hf;
          if (COMBINE && p.y_branch) {
            // both branches as they are stored, and as the backward pass will read them
            if (have[i])
              *reinterpret_cast<uint4*>((__nv_bfloat16*)p.y_branch + e) = make_uint4(v[0], v[1], v[2], v[3]);
            const __nv_bfloat162* ho = reinterpret_cast<const __nv_bfloat162*>(&oth[i]);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float2 w = __bfloat1622float2(ho[c]);
              const float2 u = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v[c]));
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(fmaf(g_other, w.x, u.x * g_this),
                                                              fmaf(g_other, w.y, u.y * g_this));
              v[c] = *reinterpret_cast<const uint32_t*>(&h2);
            }
          }
          if (have[i])
            *reinterpret_cast<uint4*>((__nv_bfloat16*)p.y + e) = make_uint4(v[0], v[1], v[2], v[3]);
        }
        // y may be the buffer the other branch's rows sit in: these columns are read before the
        // same columns are written, and nobody else touches them
        if (hf + 1 < D / 64) load_other(hf + 1);
        __syncwarp();
      }
      if (p.lse && row_valid)
        p.lse[((size_t)b * p.Hq + hq) * p.n + q_tok] = (m * p.scale2 + log2f(l)) * kLn2;
      // the next item's first P V overwrites O: order these reads before the arrive that
      // lets it start
      tc_fence_before();
    }
  }

  // ----------------------------------------------------------------------- teardown
  if (kLateWait) grid_dependency_wait();      // also where no item came to its epilogue
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------- host

// Score-block width: 128 keys from w = 129 on, and at every width where d = 128 tiles come by TMA.
// 64-key blocks skip more of a window's ends and let a tile's products and row work interleave; 128-key
// blocks take half as many products, commits and softmax rounds per key.  The first block of a row
// also sets the maximum that P is rounded under: of 128 keys it is more often the row's own, and its
// probability then exactly 1.  Error of y against float64, 64 / 128 keys: 2.152e-3 / 2.111e-3 (2 x 16
// heads of 128, n = 2048, w = 256), 2.172e-3 / 2.143e-3 (16/4 heads of 64, w = 320), TMA tiles 2.171e-3 /
// 2.154e-3 (16 heads of 64, w = 256).  Times, us with 64 / 128:
//   gathered: 8/2 heads of 128, n = 4096: w = 129 16.5 / 15.2, w = 256 20.0 / 18.4; 2 x 16 heads of 128,
//     n = 4096: w = 64 58.5 / 62.2, w = 160 72.0 / 75.8, w = 320 88.0 / 89.9; 32/8 heads of 128, n = 8192:
//     w = 384 133 / 127, w = 1024 244 / 216;
//   tiles by TMA, d = 128 (one issuing thread, 32/8 heads, n = 8192): w = 33 57.4 / 56.6, w = 128 65 / 57,
//     w = 1024 204 / 150;
//   tiles by TMA, d = 64 (two issuing threads hide the commits): 8 x 12 heads, n = 4096: w = 33 65 / 79,
//     w = 384 116 / 124.
// So between w = 129 and 320, and at d = 64 by TMA, the line is drawn by the error, not by the time.
// It depends on nothing that a part of a batch or of the heads changes: a sequence has the same bits
// alone, in a batch and in a piece of the host pipeline.
// The test hook sa_debug_set(SA_DEBUG_SCORE_BLOCK, 64 | 128) overrides the choice.
bool key_block_128(int w, int d, bool tma_tiles) {
  const int forced = debug_option(SA_DEBUG_SCORE_BLOCK);
  if (forced) return forced == 128;
  return w > 128 || (tma_tiles && d == 128);
}

// sa_debug_set(SA_DEBUG_SWA_TILE_LOADS, 0) keeps the cp.async gather for the one-sided SWA
// branch too.
bool swa_tma_disabled() { return debug_option(SA_DEBUG_SWA_TILE_LOADS) == 0; }

bool tc_disabled() { return debug_option(SA_DEBUG_TENSOR_CORES) == 0; }

}  // namespace

bool tc_forward_supported(const FwdArgs& a, int dtype) {
  if (tc_disabled() || dtype != SA_BF16 || (a.d != 128 && a.d != 64)) return false;
  if (a.n < 1 || (int64_t)a.B * a.Hq * ((a.n + kTile - 1) / kTile) > 0x3fffffff) return false;
  if (a.qs[2] >= (1ll << 30) || a.ks[2] >= (1ll << 30)) return false;   // 32-bit row strides
  return true;
}

bool tc_forward_ordered(const FwdArgs& a, int dtype, OrderGeom* g) {
  return !a.swa && !a.rope_cos && tc_forward_supported(a, dtype) &&
         debug_option(SA_DEBUG_SCORE_BLOCK) != 64 && order_geom(a.n, a.d, a.w, a.flags, g);
}

cudaError_t launch_fwd_tc(const FwdArgs& a, cudaStream_t st) {
  TcParams p{};
  p.q = a.q; p.k = a.k; p.v = a.v;
  p.perm = a.swa ? nullptr : a.perm;
  p.rope_cos = a.rope_cos; p.rope_sin = a.rope_sin;
  p.y = a.y; p.y_branch = a.y_branch; p.y_other = a.y_other; p.lse = a.lse;
  p.gate_logits = a.gate_logits;
  p.status = status_ptr();
  if (!p.status) return cudaErrorUnknown;
  p.abort_flag = a.abort_flag;
  p.B = a.B; p.Hq = a.Hq; p.Hkv = a.Hkv; p.G = a.Hq / a.Hkv; p.n = a.n; p.w = a.w;
  const MaskGeom mg = make_geom(a.n, a.w, a.flags, a.swa);
  p.h = mg.h;
  p.causal = mg.causal; p.linear = mg.linear; p.one_sided = mg.one_sided; p.swa = a.swa;
  p.full_range = mg.one_sided ? (a.w - 1 >= a.n) : (2ll * mg.h + 1 >= a.n);
  p.pair_heads = (p.G % 2 == 0);
  p.n_tiles = (a.n + kTile - 1) / kTile;
  p.items_per_kv = p.pair_heads ? p.n_tiles * (p.G / 2) : ((p.n_tiles + 1) / 2) * p.G;
  p.scale2 = a.scale * kLog2e;
  for (int i = 0; i < 3; ++i) { p.qs[i] = a.qs[i]; p.ks[i] = a.ks[i]; }
  const bool ordered = a.lists && tc_forward_ordered(a, SA_BF16, &p.og);
  if (ordered) {
    const int per_group = p.og.slots / kTile, full = p.n_tiles / per_group;
    if (!p.pair_heads)
      p.items_per_kv = (full * (per_group / 2) + (p.n_tiles - full * per_group + 1) / 2) * p.G;
    p.order = order_view(a.lists, a.B, p.og);
  }
  p.total_items = a.B * a.Hkv * p.items_per_kv;
  p.by_items = FastDiv(p.items_per_kv);
  p.by_kv = FastDiv(a.Hkv);
  p.by_inner = FastDiv(p.pair_heads ? p.G / 2 : ordered ? p.G : (p.n_tiles + 1) / 2);
  p.by_full = FastDiv(ordered ? max(p.n_tiles / (p.og.slots / kTile), 1) : 1);

  static int sm_count[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) return e != cudaSuccess ? e : cudaErrorInvalidDevice;
  if (!sm_count[dev]) {
    e = cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  const unsigned grid = (unsigned)min(p.total_items, sm_count[dev]);
  const bool combine = a.gate_logits && a.y_other;
  // gates only with the other branch's rows; branch rows of their own only where gates are applied
  if ((a.gate_logits && !a.y_other) || (a.y_branch && !combine) || !a.y) return cudaErrorInvalidValue;
  // whole-tile TMA loads for the one-sided SWA branch (any strides the maps can express;
  // otherwise the gather serves this branch too)
  CUtensorMap tm_q{}, tm_k{}, tm_v{};
  const bool natural =
      a.swa && mg.one_sided && !swa_tma_disabled() && !a.rope_cos &&   // TMA tiles cannot be turned
      aligned16(a.q) && aligned16(a.k) && aligned16(a.v) &&
      make_map_bhnd(&tm_q, a.q, a.B, a.Hq, a.n, a.d, a.qs) &&
      make_map_bhnd(&tm_k, a.k, a.B, a.Hkv, a.n, a.d, a.ks) &&
      make_map_bhnd(&tm_v, a.v, a.B, a.Hkv, a.n, a.d, a.ks);
  auto go = [&](auto kernel, int smem) {
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err != cudaSuccess) return err;
    return launch_dependent(kernel, dim3(grid), dim3(kThreads), smem, st, p, tm_q, tm_k, tm_v);
  };
  const bool wide = key_block_128(a.w, a.d, natural);
  if (ordered) {
    e = a.d == 128 ? go(fwd_tc_kernel<128, 128, kOrdered>, Cfg<128>::kBytes)
                   : go(fwd_tc_kernel<64, 128, kOrdered>, Cfg<64>::kBytes);
    if (e != cudaSuccess) return e;
    bump_launches();
    return cudaGetLastError();
  }
  // instantiation by (head dimension, score-block width, source of the tiles, rotation, combine)
  auto pick = [&](auto d_c, auto kb_c) {
    constexpr int DD = decltype(d_c)::value, KK = decltype(kb_c)::value;
    constexpr int kB = Cfg<DD>::kBytes;
    if (a.rope_cos)
      return combine ? go(fwd_tc_kernel<DD, KK, kGather, true, true>, kB)
                     : go(fwd_tc_kernel<DD, KK, kGather, true, false>, kB);
    if (natural)
      return combine ? go(fwd_tc_kernel<DD, KK, kNatural, false, true>, kB)
                     : go(fwd_tc_kernel<DD, KK, kNatural, false, false>, kB);
    return combine ? go(fwd_tc_kernel<DD, KK, kGather, false, true>, kB)
                   : go(fwd_tc_kernel<DD, KK, kGather, false, false>, kB);
  };
  using I64 = std::integral_constant<int, 64>;
  using I128 = std::integral_constant<int, 128>;
  if (a.d == 128) e = wide ? pick(I128{}, I128{}) : pick(I128{}, I64{});
  else e = wide ? pick(I64{}, I128{}) : pick(I64{}, I64{});
  if (e != cudaSuccess) return e;
  bump_launches();
  return cudaGetLastError();
}

}  // namespace sa

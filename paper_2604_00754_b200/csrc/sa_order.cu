// Key lists of the causal SA branch: per group of consecutive slots, the union of its queries' windows
// in token order.
//
// Causality is in token order and the window in slot order, so a tile of 128 consecutive slots meets
// every key of its window although half of the pairs are hidden.  Here a group of 256 or 512 slots is
// dealt to its query tiles by token: tile i holds the i-th 128 of the group's tokens.  The keys of the
// group's window, in token order, are one list for all its tiles, and a tile stops at the last token
// it holds: with w = 1024 two tiles meet 5.3 and 10 blocks of 128 keys where they met 9 each, with
// w = 2048 four tiles 3.6 to 20 (12.8 on the average) where they met 17.  What a row sees of a block is
// one bit per key, worked out here once for all heads.
// SA branch of 32/8 heads of 128, n = 32768, w = 1024: 818 us without lists, 674 with them and this launch (calls
// back to back, in turn); of 32/4 heads, n = 131072, w = 2048: 5363 and 4034.  The launch itself takes 17.5 us at
// n = 32768, w = 1024, 29 at w = 2048, 75 at n = 131072, w = 2048.  Clocks inside it, n = 32768, median of the
// CTAs from the start, w = 1024 / 2048: tokens counted 1.0 / 1.7 us, sorted 4.1 / 6.9, queries found 6.1 / 9.2,
// bits written 11.8 / 19.7, those of the longest list 16.4 / 28: the bits bound it (some 360 instructions per 32 keys
// and 128 rows, two CTAs on most SMs), then the chain of latencies before them.
#include "sa_order.cuh"

namespace sa {
namespace {

constexpr int kThreads = 512, kBuckets = 1024, kDeep = 16;

struct OrderParams {
  const int32_t* perm;
  int32_t *q, *k, *tiles;
  uint4* bits;
  int n, h, linear;
  OrderGeom g;
  uint32_t bucket_mul;          // bucket of a token: umulhi(token, bucket_mul) < kBuckets
};

size_t shared_bytes(int span) {
  const size_t l = ((size_t)span + 7) / 8 * 8;
  return l * 12 + kBuckets * 4;
}

// One CTA per query tile; the tiles of a group each sort the group's keys (a few microseconds that
// run side by side), and each works out its own bits.  Sort: counts per bucket of tokens, a place per
// key, and the rank inside the bucket by counting; any contents give the unique order.  A random
// permutation puts up to 8 keys on the average into a bucket.  One that keeps neighbours together (the
// identity, shuffled blocks) may put the whole window into a few: where some bucket holds more than kDeep
// keys, each is divided once more, after which sqrt(n / 1024) keys at most share one.  This launch, w = 2048,
// random / identity / blocks of 256: n = 131072 75 / 70 / 77 us where the second division was missing 74 /
// 194 / 201; w = 1024, n = 2^20 291 / 287 / 296 and 289 / 2861 / 1184.  16 is where the second division is worth
// it: with 32 keys to a bucket (identity, n = 32768, w = 1024) 17.5 us with it, 21.9 without.
// Whatever perm holds, a rejected one of SA_VALIDATE_PERM too, everything that the attention launch reads
// is written and in range: that launch looks at the status word for itself, later, and the word may have
// been read and cleared in between.
// 32 registers, four CTAs per SM (with the loops of the second division unrolled, 60 and two: n = 2^20, w = 1024
// 289 -> 375 us).
__global__ void __launch_bounds__(kThreads, 4) order_kernel(const __grid_constant__ OrderParams p) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t part[kThreads / 32];
  __shared__ int q_pos[kOrderTile], q_off[kOrderTile];
  constexpr uint32_t kGuard = 0x8000u;            // set in the sorted offsets (all below 2^15)
  const OrderGeom& g = p.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.y, tile = blockIdx.x, per_group = g.slots / kOrderTile;
  const int group = tile / per_group, part_of = tile % per_group;
  const int s0 = group * g.slots, slots = min(g.slots, p.n - s0), span = slots + 2 * p.h;
  const int cap = (g.span + 7) / 8 * 8;
  int32_t* tok = reinterpret_cast<int32_t*>(smem);
  int32_t* tok2 = tok + cap;
  uint16_t* off = reinterpret_cast<uint16_t*>(tok2 + cap);
  uint16_t* off2 = off + cap;
  uint32_t* start = reinterpret_cast<uint32_t*>(off2 + cap);

  for (int i = tid; i < kBuckets; i += kThreads) start[i] = 0u;
  grid_dependency_wait();
  grid_dependents_launch();
  __syncthreads();
  const int32_t* perm = p.perm + (size_t)b * p.n;
  auto bucket_of = [&](int32_t t) { return min(__umulhi((uint32_t)t, p.bucket_mul), kBuckets - 1u); };
  // a token of -1: outside the sequence (linear windows); of n and more, or negative: taken for n - 1
  for (int o = tid; o < span; o += kThreads) {
    int s = s0 - p.h + o;
    int32_t t = -1;
    if (!p.linear) { s = s < 0 ? s + p.n : s >= p.n ? s - p.n : s; }
    if (s >= 0 && s < p.n) t = (int32_t)min((uint32_t)perm[s], (uint32_t)p.n - 1u);
    tok[o] = t;
    if (t >= 0) off[o] = (uint16_t)atomicAdd(&start[bucket_of(t)], 1u);
  }
  __syncthreads();
  // exclusive scan over the block: `mine` per thread; returns the sum of those before it
  auto scan = [&](uint32_t mine, uint32_t* total) {
    uint32_t x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) part[warp] = x;
    __syncthreads();
    uint32_t before = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
      if (w < warp) before += part[w];
      sum += part[w];
    }
    __syncthreads();
    *total = sum;
    return before + x - mine;
  };
  uint32_t keys, most = 0;
  {
    constexpr int kPer = kBuckets / kThreads;
    uint32_t c[kPer], mine = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      c[i] = start[kPer * tid + i];
      mine += c[i];
      most = max(most, c[i]);
    }
    uint32_t at = scan(mine, &keys);
#pragma unroll
    for (int i = 0; i < kPer; ++i) { start[kPer * tid + i] = at; at += c[i]; }
  }
  if (!__syncthreads_or(most > kDeep)) {
    for (int o = tid; o < span; o += kThreads) {
      const int32_t t = tok[o];
      if (t < 0) continue;
      const uint32_t at = start[bucket_of(t)] + off[o];
      tok2[at] = t;
      off2[at] = (uint16_t)o;
    }
    __syncthreads();
    for (int x = tid; x < (int)keys; x += kThreads) {
      const int32_t t = tok2[x];
      const uint16_t o = off2[x];
      const uint32_t bk = bucket_of(t), lo = start[bk], hi = bk + 1 < kBuckets ? start[bk + 1] : keys;
      uint32_t rank = lo;
      for (uint32_t y = lo; y < hi; ++y) {
        const int32_t u = tok2[y];
        rank += u < t || (u == t && off2[y] < o);
      }
      tok[rank] = t;
      off[rank] = (uint16_t)(o | kGuard);
    }
  } else {
    // A bucket of c keys is cut into c of its own, by where a token lies in it; these are counted and scanned
    // like the first, in the room of tok2, and hold the keys' offsets alone.
    uint32_t* sub = reinterpret_cast<uint32_t*>(tok2);
    auto sub_of = [&](int32_t t) {
      const uint64_t at = (uint64_t)(uint32_t)t * p.bucket_mul;
      const uint32_t bk = (uint32_t)(at >> 32), lo = start[bk], hi = bk + 1 < kBuckets ? start[bk + 1] : keys;
      return lo + __umulhi((uint32_t)at, hi - lo);
    };
#pragma unroll 1
    for (int x = tid; x < (int)keys; x += kThreads) sub[x] = 0u;
    __syncthreads();
#pragma unroll 1
    for (int o = tid; o < span; o += kThreads) {
      const int32_t t = tok[o];
      if (t >= 0) off[o] = (uint16_t)atomicAdd(&sub[sub_of(t)], 1u);
    }
    __syncthreads();
    {
      const int per = ((int)keys + kThreads - 1) / kThreads, x0 = tid * per, x1 = min(x0 + per, (int)keys);
      uint32_t mine = 0, all;
#pragma unroll 1
      for (int x = x0; x < x1; ++x) mine += sub[x];
      uint32_t at = scan(mine, &all);
#pragma unroll 1
      for (int x = x0; x < x1; ++x) {
        const uint32_t c = sub[x];
        sub[x] = at;
        at += c;
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int o = tid; o < span; o += kThreads) {
      const int32_t t = tok[o];
      if (t >= 0) off2[sub[sub_of(t)] + off[o]] = (uint16_t)o;
    }
    __syncthreads();
#pragma unroll 1
    for (int x = tid; x < (int)keys; x += kThreads) {
      const uint16_t o = off2[x];
      const int32_t t = tok[o];
      const uint32_t sb = sub_of(t), lo = sub[sb], hi = sb + 1 < keys ? sub[sb + 1] : keys;
      uint32_t rank = lo;
#pragma unroll 1
      for (uint32_t y = lo; y < hi; ++y) {
        const uint16_t r = off2[y];
        const int32_t u = tok[r];
        rank += u < t || (u == t && r < o);
      }
      off[rank] = (uint16_t)(o | kGuard);
    }
    __syncthreads();
#pragma unroll 1
    for (int x = tid; x < (int)keys; x += kThreads) tok2[x] = tok[off[x] ^ kGuard];
    __syncthreads();
#pragma unroll 1
    for (int x = tid; x < (int)keys; x += kThreads) tok[x] = tok2[x];
  }
  if (tid < kOrderTile) q_pos[tid] = -1;
  __syncthreads();
  // this tile's queries: the 128 that follow 128 * part_of of the group's in token order
  const int rows = min(kOrderTile, slots - part_of * kOrderTile);
  int32_t* q_out = p.q + ((size_t)b * g.tiles + tile) * kOrderTile;
  {
    const int per = ((int)keys + kThreads - 1) / kThreads, x0 = tid * per, x1 = min(x0 + per, (int)keys);
    auto query = [&](int x) { return (int)(off[x] ^ kGuard) - p.h; };     // in [0, slots): a query of the group
    uint32_t mine = 0, all;
    for (int x = x0; x < x1; ++x) mine += (uint32_t)query(x) < (uint32_t)slots;
    int r = (int)scan(mine, &all) - part_of * kOrderTile;
    for (int x = x0; x < x1; ++x)
      if ((uint32_t)query(x) < (uint32_t)slots) {
        if (r >= 0 && r < kOrderTile) {
          q_pos[r] = x;
          q_off[r] = query(x);
          q_out[r] = tok[x];
        }
        ++r;
      }
  }
  __syncthreads();
  const int end = max(q_pos[rows - 1], 0), blocks = end / kOrderTile + 1;
  if (tid >= rows && tid < kOrderTile) q_out[tid] = tok[end];      // rows that do not exist
  if (tid == 0) p.tiles[(size_t)b * g.tiles + tile] = blocks;
  if (part_of * kOrderTile + rows == slots) {                    // the last tile meets the whole list
    int32_t* k_out = p.k + ((size_t)b * g.groups + group) * g.pitch;
    for (int x = tid; x < blocks * kOrderTile; x += kThreads) k_out[x] = tok[min(x, (int)keys - 1)];
  }
  // A key's bit: it is in the row's window (its offset in [q, q + 2 h]) and not after the row's token
  // (its place in the list is not after the row's own).  Two offsets at a time: with the guard bits
  // set a subtraction of both halves borrows nothing across, and leaves the bit where the offset is
  // not below the bound.
  uint4* bits = p.bits + ((size_t)b * g.tiles + tile) * g.blocks * kOrderTile;
  for (int task = warp; task < 4 * blocks; task += kThreads / 32) {
    const int j = task >> 2, r = (task & 3) * 32 + lane;
    const int pos = q_pos[r], qo = pos < 0 ? 0 : q_off[r];
    const int last = __reduce_max_sync(0xffffffffu, pos);
    const uint32_t from = qo * 0x10001u, past = (uint32_t)(qo + 2 * p.h + 1) * 0x10001u;
    uint32_t word[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int x0 = kOrderTile * j + 32 * y;
      word[y] = 0u;
      if (x0 > last) continue;
      uint32_t v = 0;
#pragma unroll
      for (int c = 0; c < 32; c += 8) {
        const uint4 o8 = *reinterpret_cast<const uint4*>(off + x0 + c);
        const uint32_t o[4] = {o8.x, o8.y, o8.z, o8.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) v = (v >> 1) | ((o[e] - from) & ~(o[e] - past) & 0x80008000u);
      }
      // the even keys are in the lower half, the odd in the upper: merge them
      uint32_t even = v & 0xffffu, odd = v >> 16;
#pragma unroll
      for (int e = 8; e > 0; e >>= 1) {
        const uint32_t keep = e == 8 ? 0x00ff00ffu : e == 4 ? 0x0f0f0f0fu : e == 2 ? 0x33333333u : 0x55555555u;
        even = (even | (even << e)) & keep;
        odd = (odd | (odd << e)) & keep;
      }
      const int upto = pos - x0;
      word[y] = upto < 0 ? 0u : (even | (odd << 1)) & (upto >= 31 ? ~0u : (2u << upto) - 1u);
    }
    bits[(size_t)j * kOrderTile + r] = make_uint4(word[0], word[1], word[2], word[3]);
  }
}

size_t up(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

bool order_geom(int n, int d, int w, uint32_t flags, OrderGeom* g) {
  const MaskGeom m = make_geom(n, w, flags, false);
  // Times of the SA branch without lists / with lists and their launch, us (heads of d; n):
  //                          w = 512      768          1024         2048
  //   4/2 of 64;    8192      23 / 40      29 / 48      34 / 58      57 / 100
  //                16384      41 / 56      52 / 69      63 / 84     108 / 144
  //                32768      76 / 78      98 / 96     121 / 116    210 / 199
  //   4/1 of 128;  32768      74 / 81      92 / 97     112 / 116    188 / 174
  //                49152     106 / 112    134 / 135    163 / 160    275 / 239
  //   8/2 of 128;   8192      41 / 56      51 / 68      60 / 81      99 / 136
  //                16384      74 / 80      92 / 95     111 / 113    187 / 187
  //                32768     126 / 130    161 / 156    203 / 193    331 / 298
  //   32/8 of 128;  8192     128 / 126    162 / 151    195 / 177    334 / 293
  //                10007     163 / 167    205 / 206    252 / 244    421 / 398
  //                16384     243 / 228    310 / 278    377 / 328    659 / 530
  //                32768     490 / 455    637 / 553    818 / 674   1355 / 1030
  //   2/1 of 64;   32768      41 / 52      52 / 63      64 / 75     108 / 125
  //                49152      59 / 68      75 / 84      92 / 101    160 / 154
  //                65536      76 / 80      99 / 98     121 / 117    210 / 182
  //   2/1 of 128;  32768      41 / 52      50 / 62      60 / 74      99 / 120
  //                65536      74 / 84      93 / 100    114 / 119    191 / 178
  // The line is drawn where four query heads break even.  Thirty-two would gain from n = 8192 on, and two lose
  // up to 22 us, a quarter at most, below n = 65536 (2/1 of 128, w = 1024: 3 % at 131072 still): the launch takes
  // the same time for any number of heads.  The line is one for all of them because a sequence has the same
  // bits alone and in a batch, and a KV head the same in any part of the heads (tensor-parallel shards).
  // 256 slots or 512: blocks per tile 7.7 / 7.8 at w = 1024, 10.7 / 10.3 at 1536, 13.7 / 12.8 at 2048.
  if (!m.causal || w < 1024 || n < 32768 || (d != 64 && d != 128)) return false;
  g->slots = w <= 1280 ? 256 : 512;
  // 16 bits per offset with one to spare, 102 KB of shared memory; and no slot twice, as 8192 < n
  if ((int64_t)g->slots + 2ll * m.h > 8192) return false;
  g->span = g->slots + 2 * m.h;
  g->groups = (n + g->slots - 1) / g->slots;
  g->tiles = (n + kOrderTile - 1) / kOrderTile;
  g->blocks = (g->span + kOrderTile - 1) / kOrderTile;
  g->pitch = g->blocks * kOrderTile;
  return true;
}

size_t order_bytes(int B, const OrderGeom& g) {
  return up((size_t)B * g.tiles * kOrderTile * 4) + up((size_t)B * g.groups * g.pitch * 4) +
         up((size_t)B * g.tiles * 4) + up((size_t)B * g.tiles * g.blocks * kOrderTile * 16);
}

OrderView order_view(void* ws, int B, const OrderGeom& g) {
  OrderView v;
  char* at = (char*)ws;
  v.q = (int32_t*)at;
  at += up((size_t)B * g.tiles * kOrderTile * 4);
  v.k = (int32_t*)at;
  at += up((size_t)B * g.groups * g.pitch * 4);
  v.tiles = (int32_t*)at;
  at += up((size_t)B * g.tiles * 4);
  v.bits = (uint4*)at;
  return v;
}

cudaError_t launch_order(const int32_t* perm, int B, int n, int w, uint32_t flags, const OrderGeom& g,
                         const OrderView& v, cudaStream_t st) {
  const MaskGeom m = make_geom(n, w, flags, false);
  OrderParams p{};
  p.perm = perm;
  p.q = v.q; p.k = v.k; p.tiles = v.tiles; p.bits = v.bits;
  p.n = n; p.h = m.h; p.linear = m.linear;
  p.g = g;
  p.bucket_mul = (uint32_t)(((uint64_t)kBuckets << 32) / (uint64_t)n);     // n > kBuckets: fits
  const size_t smem = shared_bytes(g.span);
  const cudaError_t e =
      cudaFuncSetAttribute(order_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return reported(e);
  bump_launches();
  return launch_dependent(order_kernel, dim3(g.tiles, B), dim3(kThreads), smem, st, p);
}

}  // namespace sa

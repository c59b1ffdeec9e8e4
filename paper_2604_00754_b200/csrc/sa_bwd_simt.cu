// Backward pass outside the tensor-core kernels:
//   1. delta:   D_x[i] = g_x * sum_c dY[i,c] Y_x[i,c] per branch x, plus per-block partial
//               sums of dY.Y_x from which the gate-logit gradients are reduced in a fixed
//               order (no floating-point atomics anywhere: results are run-to-run identical);
//   2. fp32:    tiles of 32 rows x 32 columns on the CUDA cores, rows = queries for dq and
//               rows = keys for dk / dv;
//   3. bf16 with other head dimensions than 64 / 128: one warp per query token (dq) or key token
//               (dk / dv), which adds both branches in fp32 before the one rounding.
// Formulas: derivative of Eq. 1 / Eq. 5 with the permutation held constant,
//   P_ij = exp(scale q_i.k_j - lse_i), dS_ij = P_ij (dY_x[i].V_j - D_x[i]).
#include <type_traits>

#include "sa_bwd_tc.cuh"
#include "sa_common.cuh"
#include "sa_simt_common.cuh"

namespace sa {
namespace {

constexpr int kWarps = 8;
constexpr int kMaxColsPerLane = 8;
constexpr int kDeltaRowsPerBlock = 64;

template <typename T>
__device__ __forceinline__ float dot_f32_row(const float* __restrict__ s, const T* __restrict__ row,
                                             int d) {
  float acc = 0.f;
  for (int c = 0; c < d; c += 4) {
    const float4 sv = *reinterpret_cast<const float4*>(s + c);
    acc = fmaf(sv.x, to_f32(row[c]), acc);
    acc = fmaf(sv.y, to_f32(row[c + 1]), acc);
    acc = fmaf(sv.z, to_f32(row[c + 2]), acc);
    acc = fmaf(sv.w, to_f32(row[c + 3]), acc);
  }
  return acc;
}

__device__ __forceinline__ float sigmoidf(float x) { return 1.f / (1.f + __expf(-x)); }

__device__ __forceinline__ float dot16(const float* a, const float* b, float acc) {
  const float4 x = ld4(a), y = ld4(b);
  acc = fmaf(x.x, y.x, acc);
  acc = fmaf(x.y, y.y, acc);
  acc = fmaf(x.z, y.z, acc);
  return fmaf(x.w, y.w, acc);
}
__device__ __forceinline__ float dot16(const __nv_bfloat16* a, const __nv_bfloat16* b, float acc) {
  const uint4 x = *reinterpret_cast<const uint4*>(a), y = *reinterpret_cast<const uint4*>(b);
  const __nv_bfloat162* hx = reinterpret_cast<const __nv_bfloat162*>(&x);
  const __nv_bfloat162* hy = reinterpret_cast<const __nv_bfloat162*>(&y);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 u = __bfloat1622float2(hx[i]), v = __bfloat1622float2(hy[i]);
    acc = fmaf(u.x, v.x, acc);
    acc = fmaf(u.y, v.y, acc);
  }
  return acc;
}

// Eight lanes per row and 16 bytes per lane and load: HBM-bound (dY and every Y_x once; one block
// serves both branches, so dY is read once for the two).
template <typename T>
__global__ void __launch_bounds__(kWarps * 32) bwd_delta_kernel(const BwdArgs a) {
  __shared__ float wsum[2][kWarps];
  constexpr int kE = 16 / (int)sizeof(T);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane >> 3, l8 = lane & 7;
  const int hq = blockIdx.y, b = blockIdx.z;
  const int64_t base = b * a.qs[0] + hq * a.qs[1];
  const int r0 = blockIdx.x * kDeltaRowsPerBlock + warp * 4 + sub;
  grid_dependency_wait();
  grid_dependents_launch();
  float part[2] = {0.f, 0.f};
  float dot[2][kDeltaRowsPerBlock / 32];
#pragma unroll
  for (int u = 0; u < kDeltaRowsPerBlock / 32; ++u) {
    dot[0][u] = dot[1][u] = 0.f;
    const int i = r0 + 32 * u;
    if (i < a.n) {
      const int64_t off = base + (int64_t)i * a.qs[2];
      for (int c = kE * l8; c < a.d; c += 8 * kE) {
        dot[0][u] = dot16((const T*)a.dy + off + c, (const T*)a.y_x[0] + off + c, dot[0][u]);
        if (a.nbranch == 2)
          dot[1][u] = dot16((const T*)a.dy + off + c, (const T*)a.y_x[1] + off + c, dot[1][u]);
      }
    }
  }
  for (int x = 0; x < a.nbranch; ++x) {
    const float g = a.gate_logits ? sigmoidf(a.gate_logits[x * a.Hq + hq]) : 1.f;
    float* delta = a.delta + (((size_t)x * a.B + b) * a.Hq + hq) * a.n;
#pragma unroll
    for (int u = 0; u < kDeltaRowsPerBlock / 32; ++u) {
      float v = x ? dot[1][u] : dot[0][u];
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      if (l8 == 0 && r0 + 32 * u < a.n) delta[r0 + 32 * u] = g * v;
      part[x] += v;
    }
    float v = part[x];
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    if (lane == 0) wsum[x][warp] = v;
  }
  __syncthreads();
  if ((int)threadIdx.x < a.nbranch) {
    float s = 0.f;
    for (int wv = 0; wv < kWarps; ++wv) s += wsum[threadIdx.x][wv];
    a.partials[(((size_t)threadIdx.x * a.B + b) * a.Hq + hq) * a.chunks + blockIdx.x] = s;
  }
}

// One block per (branch, head): its B * chunks partial sums, in a fixed order.
__global__ void __launch_bounds__(128) dgate_kernel(const BwdArgs a) {
  __shared__ float wsum[4];
  const int hq = blockIdx.x, x = blockIdx.y;
  grid_dependency_wait();
  grid_dependents_launch();
  float s = 0.f;
  for (int i = threadIdx.x; i < a.B * a.chunks; i += 128)
    s += a.partials[(((size_t)x * a.B + i / a.chunks) * a.Hq + hq) * a.chunks + i % a.chunks];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    const float g = sigmoidf(a.gate_logits[x * a.Hq + hq]);
    a.dgate[x * a.Hq + hq] = g * (1.f - g) * ((wsum[0] + wsum[1]) + (wsum[2] + wsum[3]));
  }
}

// ------------------------------------------------------------------- fp32 tiles
//
// 32 rows per CTA of 128 threads, columns 32 at a time through two shared-memory buffers, as in
// the forward (sa_fwd_simt.cu).  Rows = queries: R = (Q, dY), columns (K, V), output dQ.  Rows =
// keys: R = (K, V), columns (Q, dY) of every query head the CTA covers, outputs dK and dV.
//
// Small problems have too few row tiles for the SMs, so there each branch, and with grouped heads each
// of `parts` shares of a group's query heads, gets CTAs of its own, for all outputs in one launch, and
// writes a partial gradient that reduce_kernel adds up in a fixed order ("split").  Large ones run one
// launch per branch, the second adding to what the first stored, with the heads of a group inside the
// CTA.
//
// Bound: FMA issue and shared-memory wavefronts, about equal, behind the latency of 32-column
// steps, so warps per SM count: dS and P take turns in one buffer and the registers are held to 128
// (d <= 64), for four CTAs per SM.  With that and packed multiply-adds in the products: 2 x 4/2 heads
// of 64, n = 1500, w = 128, gated 157 -> 139 us; 8/4 heads of 128, n = 2000, w = 256 636 -> 572.

// Split (number of parts of a group's query heads; 0: not split) while the row tiles of the keys are
// fewer than eight per SM, in so many parts that they are not.  us, split / not: 2 x 4/2 heads of 64,
// n = 1500 (1.3 per SM) 139 / 186; 32/8 heads of 128, n = 512 (0.9) 538 / 864, n = 2000 (3.4) 2151 / 2309;
// 2 x 8 heads of 128, n = 1800 (6.2) 995 / 1048, n = 2000 (6.8) 685 / 717; 16 heads of 64, n = 2000 (6.8)
// 332 / 337.
// The partial gradients are two tensors of Q's size, and four of K's per part.  One part per query head
// would make them six of Q's and be slower: 64/1 heads of 128, n = 8000 (eight parts for 64) 9834 / 10302
// us, n = 16000 (four) 19547 / 20627; 64/8 heads, n = 4096 (two for eight) 5126 / 5304.
// A constant for the SMs: the size of the workspace may not depend on the device that happens to be
// current.
constexpr int kPlanSms = 148;
int split_parts(int B, int Hq, int Hkv, int n) {
  const int64_t tiles = (int64_t)B * Hkv * ((n + kRows - 1) / kRows), enough = 8 * kPlanSms;
  if (tiles >= enough) return 0;
  const int G = Hq / Hkv;
  for (int p = 1; p < G; ++p)
    if (G % p == 0 && tiles * p >= enough) return p;
  return G;
}

// Without SEEN nothing is stored and false returned where a sum of this CTA ended in a NaN: see
// tile_accumulate_seen.
template <bool KEYS, int NCG, bool SEEN>
__device__ __forceinline__ bool bwd_tile(const BwdArgs& a, unsigned char* smem_raw, int b, int x,
                                         int hfirst, int heads, float* out1, float* out2,
                                         bool split) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tx = lane & 15, half = lane >> 4, row0 = warp * 8 + half * 4;
  const int d = a.d, s0 = blockIdx.x * kRows, hk = hfirst / (a.Hq / a.Hkv);
  const bool swa = x == 1;
  const int32_t* perm = swa ? nullptr : a.perm + (size_t)b * a.n;
  const TileSmem<float> sm(d);
  float* r1 = reinterpret_cast<float*>(smem_raw);
  float* r2 = r1 + kRows * sm.row_elems();
  float* cols = r2 + kRows * sm.row_elems();           // (C1 C2) x 2
  float* pw = cols + 4 * sm.col_elems() + warp * (kCols * 8);   // dS, then P: [32][8]
  typedef int IntCols[kCols];
  typedef float FloatCols[kCols];
  char* stat = reinterpret_cast<char*>(cols + 4 * sm.col_elems() + kTileThreads / 32 * kCols * 8);
  IntCols *s_slot = reinterpret_cast<IntCols*>(stat), *s_tok = s_slot + 2;
  FloatCols *s_lse = reinterpret_cast<FloatCols*>(s_tok + 2), *s_delta = s_lse + 2;

  const int64_t q_off = b * a.qs[0], k_off = b * a.ks[0] + hk * a.ks[1];
  const float scale2 = a.scale * kLog2e;
  const float* kbase = (const float*)a.k + k_off;
  const float* vbase = (const float*)a.v + k_off;
  if (KEYS) {
    load_rows<float>(r1, d, kbase, a.ks[2], perm, s0, a.n, scale2);
    load_rows<float>(r2, d, vbase, a.ks[2], perm, s0, a.n, 1.f);
  } else {
    const int64_t o = q_off + hfirst * a.qs[1];
    load_rows<float>(r1, d, (const float*)a.q + o, a.qs[2], perm, s0, a.n, scale2);
    load_rows<float>(r2, d, (const float*)a.dy + o, a.qs[2], perm, s0, a.n, 1.f);
  }
  const TileMask g(a.n, a.w, a.flags, swa, s0, KEYS);
  const float* lse = a.lse_x[x] + (size_t)b * a.Hq * a.n;
  const float* delta = a.delta + ((size_t)x * a.B + b) * a.Hq * a.n;
  int rslot[4], rtok[4];
  float rlse[4], rdelta[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    rslot[r] = s0 + row0 + r;
    const int sl = min(rslot[r], a.n - 1);
    rtok[r] = perm ? perm[sl] : sl;
    if (!KEYS) {
      rlse[r] = lse[(size_t)hfirst * a.n + rtok[r]] * kLog2e;
      rdelta[r] = delta[(size_t)hfirst * a.n + rtok[r]];
    }
  }
  ColLoader<float> ld(d);
  const int total = KEYS ? g.tiles * heads : g.tiles;
  float c_lse = 0.f, c_delta = 0.f;
  auto fetch = [&](int u) {
    ld.fetch(g, perm, KEYS ? u % g.tiles : u);
    if (KEYS && tid < kCols) {
      const size_t at = (size_t)(hfirst + u / g.tiles) * a.n + max(ld.tok, 0);
      c_lse = lse[at] * kLog2e;
      c_delta = delta[at];
    }
  };
  auto issue = [&](int u) {
    const int buf = u & 1;
    float* d1 = cols + 2 * buf * sm.col_elems();
    if (KEYS) {
      if (tid < kCols) { s_lse[buf][tid] = c_lse; s_delta[buf][tid] = c_delta; }
      const int64_t o = q_off + (hfirst + u / g.tiles) * a.qs[1];
      ld.issue(d1, (const float*)a.q + o, d1 + sm.col_elems(), (const float*)a.dy + o, a.qs[2],
               s_slot[buf], s_tok[buf]);
    } else {
      ld.issue(d1, kbase, d1 + sm.col_elems(), vbase, a.ks[2], s_slot[buf], s_tok[buf]);
    }
  };

  float o1[4][4 * NCG], o2[4][KEYS ? 4 * NCG : 1];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4 * NCG; ++c) {
      o1[r][c] = 0.f;
      if (KEYS) o2[r][c] = 0.f;
    }
  float gx = a.gate_logits ? sigmoidf(a.gate_logits[x * a.Hq + hfirst]) : 1.f;

  fetch(0);
  issue(0);
  if (total > 1) fetch(1);
  for (int u = 0; u < total; ++u) {
    const int buf = u & 1;
    if (u + 1 < total) {
      issue(u + 1);
      if (u + 2 < total) fetch(u + 2);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    if (KEYS && heads > 1 && a.gate_logits && u % g.tiles == 0)
      gx = sigmoidf(a.gate_logits[x * a.Hq + hfirst + u / g.tiles]);
    __syncthreads();
    const float* c1 = cols + 2 * buf * sm.col_elems();
    const float* c2 = c1 + sm.col_elems();
    float s[4][2], dp[4][2];
    tile_dot<float>(s, r1 + row0 * sm.row_elems(), sm.row_elems(), c1 + tx * sm.stride(),
                    16 * sm.stride(), d);
    tile_dot<float>(dp, r2 + row0 * sm.row_elems(), sm.row_elems(), c2 + tx * sm.stride(),
                    16 * sm.stride(), d);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int col = tx + 16 * c;
      const int cs = s_slot[buf][col], ct = s_tok[buf][col];
      const float cl = KEYS ? s_lse[buf][col] : 0.f, cd = KEYS ? s_delta[buf][col] : 0.f;
      float ds[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const bool see = rslot[r] < a.n && g.sees(rslot[r], rtok[r], cs, ct);
        const float p = see ? exp2f(s[r][c] - (KEYS ? cl : rlse[r])) : 0.f;
        ds[r] = p * fmaf(gx, dp[r][c], -(KEYS ? cd : rdelta[r]));
        s[r][c] = p * gx;
      }
      st4(pw + 8 * col + 4 * half, make_float4(ds[0], ds[1], ds[2], ds[3]));
    }
    __syncwarp();
    auto seen = [&](int r, int k) {
      return rslot[r] < a.n && g.sees(rslot[r], rtok[r], s_slot[buf][k], s_tok[buf][k]);
    };
    if constexpr (SEEN) tile_accumulate_seen<float, NCG>(o1, pw + 4 * half, c1, sm.stride(), tx, d, seen);
    else tile_accumulate<float, NCG>(o1, pw + 4 * half, c1, sm.stride(), tx, d);
    if constexpr (KEYS) {
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c)
        st4(pw + 8 * (tx + 16 * c) + 4 * half, make_float4(s[0][c], s[1][c], s[2][c], s[3][c]));
      __syncwarp();
      if constexpr (SEEN) tile_accumulate_seen<float, NCG>(o2, pw + 4 * half, c2, sm.stride(), tx, d, seen);
      else tile_accumulate<float, NCG>(o2, pw + 4 * half, c2, sm.stride(), tx, d);
    }
    __syncthreads();
  }
  if constexpr (!SEEN) {
    bool nan = any_nan(o1);
    if constexpr (KEYS) nan |= any_nan(o2);
    if (__syncthreads_or(nan)) return false;
  }

#pragma unroll
  for (int r = 0; r < 4; ++r) {
    if (rslot[r] >= a.n) continue;
    const int64_t off = split ? (int64_t)rtok[r] * d
                              : (int64_t)rtok[r] * (KEYS ? a.ks[2] : a.qs[2]);
#pragma unroll
    for (int cg = 0; cg < NCG; ++cg) {
      const int c = 64 * cg + 4 * tx;
      if (c >= d) continue;
      float4 v = make_float4(o1[r][4 * cg] * a.scale, o1[r][4 * cg + 1] * a.scale,
                             o1[r][4 * cg + 2] * a.scale, o1[r][4 * cg + 3] * a.scale);
      if (swa && !split) {
        const float4 w = ld4(out1 + off + c);
        v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
      }
      st4(out1 + off + c, v);
      if constexpr (KEYS) {
        v = make_float4(o2[r][4 * cg], o2[r][4 * cg + 1], o2[r][4 * cg + 2], o2[r][4 * cg + 3]);
        if (swa && !split) {
          const float4 w = ld4(out2 + off + c);
          v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
        }
        st4(out2 + off + c, v);
      }
    }
  }
  return true;
}

// The tile of this CTA.  y0 + blockIdx.y: first the nb * Hq (branch, head) pairs of dQ, then those of dK /
// dV, whose CTAs cover `heads` query heads of a group each.  Branches x0 .. x0 + nb - 1.  heads and the
// place of dV's partials come as parameters: worked out here, they would take registers from the walk
// (one head of 64, n = 700: 33.7 -> 35.9 us).
template <int NCG, bool SEEN>
__device__ __forceinline__ bool bwd_block(const BwdArgs& a, unsigned char* smem_raw, int y0, int x0,
                                          int nb, int heads, bool split, size_t dv_at) {
  const int b = blockIdx.z, G = a.Hq / a.Hkv;
  const size_t rows_q = (size_t)a.B * a.Hq * a.n * a.d;
  int y = y0 + blockIdx.y;
  if (y < nb * a.Hq) {
    const int hq = y % a.Hq, x = x0 + y / a.Hq;
    float* out = split ? a.parts + x * rows_q + ((size_t)b * a.Hq + hq) * a.n * a.d
                       : (float*)a.dq + b * a.qs[0] + hq * a.qs[1];
    return bwd_tile<false, NCG, SEEN>(a, smem_raw, b, x, hq, 1, out, nullptr, split);
  }
  y -= nb * a.Hq;
  const int groups = a.Hq / heads, h0 = (y % groups) * heads, x = x0 + y / groups, hk = h0 / G;
  const int64_t off = b * a.ks[0] + hk * a.ks[1];
  // partial (x, part of the group): [B,Hkv,n,d] each; dK's first, dV's dv_at further on
  float* part = a.parts + 2 * rows_q + (size_t)((x * G + h0 % G) / heads) * (rows_q / G) +
                ((size_t)b * a.Hkv + hk) * a.n * a.d;
  return bwd_tile<true, NCG, SEEN>(a, smem_raw, b, x, h0, heads, split ? part : (float*)a.dk + off,
                                   split ? part + dv_at : (float*)a.dv + off, split);
}

template <int NCG>
__global__ void __launch_bounds__(kTileThreads, NCG == 1 ? 4 : NCG == 2 ? 2 : 1)
bwd_tile_kernel(const __grid_constant__ BwdArgs a, int y0, int x0, int nb, int heads, bool split,
                size_t dv_at) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw;
  grid_dependency_wait();
  grid_dependents_launch();
  if (a.abort_flag && *a.abort_flag) return;
  if (bwd_block<NCG, false>(a, smem, y0, x0, nb, heads, split, dv_at)) return;
  // Nothing of the first walk is to be kept in registers for this one.  Measured on 1 x 1 head of 64,
  // n = 700 / 2 x 4/2 heads of 64, n = 1500 / 8/2 heads of 128, n = 1000, us: without it 33.6 / 138.4 /
  // 128.6, like this 33.9 / 137.1 / 130.6, with the second walk as a function 36.3 / 140.4 / 133.6, as
  // another turn of the first 36.1 / 139.0 / 131.4.
  asm volatile("" : "+r"(x0), "+r"(nb), "+r"(heads), "+l"(smem));
  bwd_block<NCG, true>(a, smem, y0, x0, nb, heads, split, dv_at);
}

// dq, dk, dv from the partial gradients of the split form, 16 bytes per thread.
__global__ void __launch_bounds__(256) reduce_kernel(const BwdArgs a, int parts) {
  const int G = a.Hq / a.Hkv, q4 = a.d / 4;
  const size_t nq = (size_t)a.B * a.Hq * a.n * q4, nk = nq / G;
  size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  grid_dependency_wait();
  grid_dependents_launch();
  if (i >= nq + 2 * nk) return;
  const int which = i < nq ? 0 : (i < nq + nk ? 1 : 2);
  i -= which == 0 ? 0 : (which == 1 ? nq : nq + nk);
  const float4* p = reinterpret_cast<const float4*>(a.parts) +
                    (which == 0 ? i : 2 * nq + (which - 1) * 2 * parts * nk + i);
  const size_t step = which ? nk : nq;
  const int terms = which ? a.nbranch * parts : a.nbranch;
  float4 s = p[0];
  for (int t = 1; t < terms; ++t) {
    const float4 v = p[t * step];
    s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w);
  }
  const int c = 4 * (int)(i % q4), H = which ? a.Hkv : a.Hq;
  const size_t row = i / q4;
  const int t = (int)(row % a.n), h = (int)((row / a.n) % H), b = (int)(row / ((size_t)a.n * H));
  const int64_t* st = which ? a.ks : a.qs;
  float* out = (float*)(which == 0 ? a.dq : which == 1 ? a.dk : a.dv);
  st4(out + b * st[0] + h * st[1] + (int64_t)t * st[2] + c, s);
}

template <int NCG>
cudaError_t launch_tiles(const BwdArgs& a, cudaStream_t st) {
  const TileSmem<float> sm(a.d);
  const int smem = 2 * sm.rows_bytes() + 4 * sm.col_bytes() + (kTileThreads / 32 * kCols * 8 + 8 * kCols) * 4;
  cudaError_t e = allow_smem((const void*)bwd_tile_kernel<NCG>, smem);
  if (e != cudaSuccess) return e;
  const unsigned tiles = (a.n + kRows - 1) / kRows;
  const int G = a.Hq / a.Hkv, parts = split_parts(a.B, a.Hq, a.Hkv, a.n);
  // `blocks` of the grid's second dimension, in launches of as many as it can have
  auto walk = [&](int x0, int nb, int heads, bool split, size_t dv_at) {
    const int blocks = nb * (a.Hq + a.Hq / heads), most = 65535;
    for (int y0 = 0; y0 < blocks && e == cudaSuccess; y0 += most) {
      e = launch_dependent(bwd_tile_kernel<NCG>, dim3(tiles, min(blocks - y0, most), a.B),
                           dim3(kTileThreads), smem, st, a, y0, x0, nb, heads, split, dv_at);
      bump_launches();
    }
  };
  if (parts) {
    walk(0, a.nbranch, G / parts, true, (size_t)2 * parts * a.B * a.Hkv * a.n * a.d);
    if (e != cudaSuccess) return e;
    const size_t items = ((size_t)a.Hq + 2 * a.Hkv) * a.B * a.n * (a.d / 4);
    bump_launches();
    return launch_dependent(reduce_kernel, dim3((unsigned)((items + 255) / 256)), dim3(256), 0, st, a, parts);
  }
  for (int x = 0; x < a.nbranch && e == cudaSuccess; ++x) walk(x, 1, G, false, 0);
  return e;
}

template <typename T>
__global__ void __launch_bounds__(kWarps * 32) bwd_dq_kernel(const BwdArgs a) {
  extern __shared__ float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* qs = smem + warp * 2 * a.d;
  float* dys = qs + a.d;
  const int tok = blockIdx.x * kWarps + warp;
  const int hq = blockIdx.y, b = blockIdx.z;
  if (tok >= a.n) return;
  if (a.abort_flag && *a.abort_flag) return;
  const int hk = hq / (a.Hq / a.Hkv);
  const int64_t qoff = b * a.qs[0] + hq * a.qs[1] + tok * a.qs[2];
  const T* kbase = (const T*)a.k + b * a.ks[0] + hk * a.ks[1];
  const T* vbase = (const T*)a.v + b * a.ks[0] + hk * a.ks[1];
  const float scale2 = a.scale * kLog2e;
  for (int c = lane; c < a.d; c += 32) {
    qs[c] = to_f32(((const T*)a.q)[qoff + c]) * scale2;
    dys[c] = to_f32(((const T*)a.dy)[qoff + c]);
  }
  __syncwarp();

  float acc[kMaxColsPerLane];
#pragma unroll
  for (int x = 0; x < kMaxColsPerLane; ++x) acc[x] = 0.f;

  for (int x = 0; x < a.nbranch; ++x) {
    const bool swa = x == 1;
    const int32_t* perm = swa ? nullptr : a.perm + (size_t)b * a.n;
    const int slot = swa ? tok : a.inv[(size_t)b * a.n + tok];
    const MaskGeom g = make_geom(a.n, a.w, a.flags, swa);
    const SlotRange r = key_range(g, slot);
    const size_t row = (((size_t)x * a.B + b) * a.Hq + hq) * a.n + tok;
    const float lse2 = a.lse_x[x][((size_t)b * a.Hq + hq) * a.n + tok] * kLog2e;
    const float delta = a.delta[row];
    const float gx = a.gate_logits ? sigmoidf(a.gate_logits[x * a.Hq + hq]) : 1.f;
    for (int t0 = 0; t0 < r.count; t0 += 32) {
      const int t = t0 + lane;
      int ks = r.start + t, kt = -1;
      bool ok = t < r.count;
      if (ok) {
        if (r.wrap) ks = wrap_slot(ks, a.n);
        else ok = ks >= 0 && ks < a.n;
      }
      if (ok) {
        kt = perm ? perm[ks] : ks;
        ok = visible(g, slot, tok, ks, kt);
      }
      float ds = 0.f;
      if (ok) {
        const float p = exp2f(dot_f32_row<T>(qs, kbase + kt * a.ks[2], a.d) - lse2);
        const float dp = gx * dot_f32_row<T>(dys, vbase + kt * a.ks[2], a.d);
        ds = p * (dp - delta);
      }
      for (uint32_t rest = __ballot_sync(0xffffffffu, ok); rest; rest &= rest - 1) {
        const int src = __ffs(rest) - 1;
        const float dsj = __shfl_sync(0xffffffffu, ds, src);
        const int jt = __shfl_sync(0xffffffffu, kt, src);
        const T* kr = kbase + jt * a.ks[2];
#pragma unroll
        for (int y = 0; y < kMaxColsPerLane; ++y) {
          const int c = lane + 32 * y;
          if (c < a.d) acc[y] = fmaf(dsj, to_f32(kr[c]), acc[y]);
        }
      }
    }
  }
#pragma unroll
  for (int y = 0; y < kMaxColsPerLane; ++y) {
    const int c = lane + 32 * y;
    if (c < a.d) ((T*)a.dq)[qoff + c] = from_f32<T>(acc[y] * a.scale);
  }
}

template <typename T>
__global__ void __launch_bounds__(kWarps * 32) bwd_dkv_kernel(const BwdArgs a) {
  extern __shared__ float smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* ksm = smem + warp * 2 * a.d;
  float* vsm = ksm + a.d;
  const int tok = blockIdx.x * kWarps + warp;  // key token
  const int hk = blockIdx.y, b = blockIdx.z;
  if (tok >= a.n) return;
  if (a.abort_flag && *a.abort_flag) return;
  const int G = a.Hq / a.Hkv;
  const int64_t koff = b * a.ks[0] + hk * a.ks[1] + tok * a.ks[2];
  const float scale2 = a.scale * kLog2e;
  for (int c = lane; c < a.d; c += 32) {
    ksm[c] = to_f32(((const T*)a.k)[koff + c]) * scale2;
    vsm[c] = to_f32(((const T*)a.v)[koff + c]);
  }
  __syncwarp();

  float dk[kMaxColsPerLane], dv[kMaxColsPerLane];
#pragma unroll
  for (int y = 0; y < kMaxColsPerLane; ++y) dk[y] = dv[y] = 0.f;

  for (int x = 0; x < a.nbranch; ++x) {
    const bool swa = x == 1;
    const int32_t* perm = swa ? nullptr : a.perm + (size_t)b * a.n;
    const int kslot = swa ? tok : a.inv[(size_t)b * a.n + tok];
    const MaskGeom g = make_geom(a.n, a.w, a.flags, swa);
    const SlotRange r = query_range(g, kslot);
    for (int hq = hk * G; hq < (hk + 1) * G; ++hq) {
      const float gx = a.gate_logits ? sigmoidf(a.gate_logits[x * a.Hq + hq]) : 1.f;
      const T* qbase = (const T*)a.q + b * a.qs[0] + hq * a.qs[1];
      const T* dybase = (const T*)a.dy + b * a.qs[0] + hq * a.qs[1];
      const float* lse = a.lse_x[x] + ((size_t)b * a.Hq + hq) * a.n;
      const float* delta = a.delta + (((size_t)x * a.B + b) * a.Hq + hq) * a.n;
      for (int t0 = 0; t0 < r.count; t0 += 32) {
        const int t = t0 + lane;
        int qsl = r.start + t, qt = -1;
        bool ok = t < r.count;
        if (ok) {
          if (r.wrap) qsl = wrap_slot(qsl, a.n);
          else ok = qsl >= 0 && qsl < a.n;
        }
        if (ok) {
          qt = perm ? perm[qsl] : qsl;
          ok = visible(g, qsl, qt, kslot, tok);
        }
        float p = 0.f, ds = 0.f;
        if (ok) {
          p = exp2f(dot_f32_row<T>(ksm, qbase + qt * a.qs[2], a.d) - lse[qt] * kLog2e);
          const float dp = gx * dot_f32_row<T>(vsm, dybase + qt * a.qs[2], a.d);
          ds = p * (dp - delta[qt]);
          p *= gx;  // dV_j += P_ij * (g_x dY_i)
        }
        for (uint32_t rest = __ballot_sync(0xffffffffu, ok); rest; rest &= rest - 1) {
          const int src = __ffs(rest) - 1;
          const float pi = __shfl_sync(0xffffffffu, p, src);
          const float dsi = __shfl_sync(0xffffffffu, ds, src);
          const int it = __shfl_sync(0xffffffffu, qt, src);
          const T* qr = qbase + it * a.qs[2];
          const T* dyr = dybase + it * a.qs[2];
#pragma unroll
          for (int y = 0; y < kMaxColsPerLane; ++y) {
            const int c = lane + 32 * y;
            if (c < a.d) {
              dv[y] = fmaf(pi, to_f32(dyr[c]), dv[y]);
              dk[y] = fmaf(dsi, to_f32(qr[c]), dk[y]);
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int y = 0; y < kMaxColsPerLane; ++y) {
    const int c = lane + 32 * y;
    if (c < a.d) {
      ((T*)a.dk)[koff + c] = from_f32<T>(dk[y] * a.scale);
      ((T*)a.dv)[koff + c] = from_f32<T>(dv[y]);
    }
  }
}

inline size_t align_up(size_t x, size_t al) { return (x + al - 1) / al * al; }

cudaError_t launch_dgate(const BwdArgs& a, cudaStream_t st) {
  if (!a.gate_logits || !a.dgate) return cudaSuccess;
  bump_launches();
  return launch_dependent(dgate_kernel, dim3(a.Hq, 2), dim3(128), 0, st, a);
}

template <typename T>
cudaError_t launch_all(BwdArgs a, cudaStream_t st) {
  cudaError_t e;
  if (tc_backward_supported(a, std::is_same<T, float>::value ? SA_F32 : SA_BF16)) {
    e = launch_bwd_tc(a, st);
    return e != cudaSuccess ? e : launch_dgate(a, st);
  }
  if ((e = launch_dependent(bwd_delta_kernel<T>, dim3(a.chunks, a.Hq, a.B), dim3(kWarps * 32), 0, st,
                            a)) != cudaSuccess)
    return e;
  bump_launches();
  if ((e = launch_dgate(a, st)) != cudaSuccess) return e;
  if constexpr (std::is_same<T, float>::value) {
    if (a.d <= 64) return launch_tiles<1>(a, st);
    return a.d <= 128 ? launch_tiles<2>(a, st) : launch_tiles<4>(a, st);
  } else {
    const size_t smem = (size_t)kWarps * 2 * a.d * sizeof(float);
    bwd_dq_kernel<T><<<dim3((a.n + kWarps - 1) / kWarps, a.Hq, a.B), kWarps * 32, smem, st>>>(a);
    bwd_dkv_kernel<T><<<dim3((a.n + kWarps - 1) / kWarps, a.Hkv, a.B), kWarps * 32, smem, st>>>(a);
    bump_launches(2);
    return cudaGetLastError();
  }
}

}  // namespace

size_t bwd_ws_bytes(int B, int Hq, int Hkv, int n, int d, int w, int dtype, int* chunks_out,
                    size_t* parts_at) {
  const int chunks = (n + kDeltaRowsPerBlock - 1) / kDeltaRowsPerBlock;
  if (chunks_out) *chunks_out = chunks;
  size_t bytes = align_up((size_t)2 * B * Hq * n * sizeof(float), 256) +
                 align_up((size_t)2 * B * Hq * chunks * sizeof(float), 256);
  if (parts_at) *parts_at = bytes;
  if (dtype == SA_F32)
    if (const int parts = split_parts(B, Hq, Hkv, n))
      bytes += ((size_t)2 * Hq + (size_t)4 * Hkv * parts) * B * n * d * sizeof(float);
  if (dtype == SA_BF16) {      // room for either way: the tensor cores' kernels carve their own
    const size_t tc = tc_backward_ws_bytes(B, Hq, Hkv, n, d, w);
    bytes = tc > bytes ? tc : bytes;
  }
  return bytes;
}

cudaError_t launch_bwd_simt(const BwdArgs& a, int dtype, cudaStream_t st) {
  return dtype == SA_F32 ? launch_all<float>(a, st) : launch_all<__nv_bfloat16>(a, st);
}

}  // namespace sa

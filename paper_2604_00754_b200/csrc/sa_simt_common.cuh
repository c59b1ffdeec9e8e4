// Pieces shared by the tiled CUDA-core kernels (forward and backward): the geometry and mask of
// a tile of 32 rows, the asynchronous gather of 32 column rows, and the two register-tiled
// products.  Rows are queries and columns keys, or (backward, rows = keys) the other way round.
#pragma once

#include "sa_common.cuh"

namespace sa {
namespace {

constexpr int kRows = 32, kCols = 32, kTileThreads = 128;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a),
                                            *reinterpret_cast<const uint32_t*>(&b));
}
template <typename T> __device__ __forceinline__ float4 round4(float4 v);
template <> __device__ __forceinline__ float4 round4<float>(float4 v) { return v; }
template <> __device__ __forceinline__ float4 round4<__nv_bfloat16>(float4 v) {
  auto r = [](float x) { return __bfloat162float(__float2bfloat16_rn(x)); };
  return make_float4(r(v.x), r(v.y), r(v.z), r(v.w));
}

// Shared-memory sizes.  Row strides are d plus 16 bytes: an odd multiple of 16 bytes (fp32), so
// that 8 rows read at one column fall into different banks.
template <typename T>
struct TileSmem {
  int d;
  __host__ __device__ explicit TileSmem(int d_) : d(d_) {}
  __host__ __device__ int row_elems() const { return d + 4; }                 // fp32 row operand
  __host__ __device__ int rows_bytes() const { return kRows * row_elems() * 4; }
  __host__ __device__ int stride() const { return d + 16 / (int)sizeof(T); }  // column operand
  __host__ __device__ int col_elems() const { return kCols * stride(); }
  __host__ __device__ int col_bytes() const { return col_elems() * (int)sizeof(T); }
};

// Columns that any of the rows [s0, s0 + 32) meets: `count` slots from `start`, unwrapped (start
// may be negative or the end past n - 1 where the window is circular), in `tiles` tiles; never a
// slot twice.  sees() is the mask of App. B for one (row, column) pair.
struct TileMask {
  MaskGeom g;
  bool keys, full;
  int start, count, tiles;
  __device__ TileMask(int n, int w, uint32_t flags, bool swa, int s0, bool rows_are_keys)
      : g(make_geom(n, w, flags, swa)), keys(rows_are_keys), full(false) {
    const int last = min(s0 + kRows, n) - 1, reach = min(g.w - 1, n);
    int end;
    if (g.one_sided) {
      start = keys ? s0 : max(s0 - reach, 0);
      end = keys ? min(last + reach, n - 1) : last;
    } else if (2ll * g.h + 1 >= n || (!g.linear && (int64_t)(last - s0 + 1) + 2ll * g.h > n)) {
      full = true;              // the band of these rows together wraps onto itself
      start = 0;
      end = n - 1;
    } else {
      start = g.linear ? max(s0 - g.h, 0) : s0 - g.h;
      end = g.linear ? min(last + g.h, n - 1) : last + g.h;
    }
    count = end - start + 1;
    tiles = (count + kCols - 1) / kCols;
  }
  // row: slot and token; column: unwrapped slot and token (-1: no such column)
  __device__ __forceinline__ bool sees(int rs, int rt, int cs, int ct) const {
    if (ct < 0) return false;
    const int back = keys ? ct - rt : rt - ct;        // query token minus key token
    if (g.one_sided) return back >= 0 && back <= g.w - 1;
    int dist = rs > cs ? rs - cs : cs - rs;
    if (full && !g.linear) dist = min(dist, g.n - dist);
    return dist <= g.h && (!g.causal || back >= 0);
  }
};

// Rows [s0, s0 + 32) of a tensor into shared memory as fp32 times `scale`; zero past n - 1.
template <typename T>
__device__ __forceinline__ void load_rows(float* dst, int d, const T* base, int64_t tok_stride,
                                          const int32_t* perm, int s0, int n, float scale) {
  const int q4 = d / 4;
  for (int i = threadIdx.x; i < kRows * q4; i += kTileThreads) {
    const int r = i / q4, c = 4 * (i - r * q4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (s0 + r < n) {
      const int tok = perm ? perm[s0 + r] : s0 + r;
      v = ld4(base + (int64_t)tok * tok_stride + c);
      v.x *= scale; v.y *= scale; v.z *= scale; v.w *= scale;
    }
    st4(dst + r * (d + 4) + c, v);
  }
}

// Gathers the column rows of one tile.  Lane r of every warp holds the token of column r, one
// tile ahead of its use; the 16-byte pieces of the 32 rows are dealt to the 128 threads.
template <typename T>
struct ColLoader {
  int pieces, stride, vslot = 0, tok = -1;
  uint32_t magic;
  __device__ explicit ColLoader(int d)
      : pieces(d * (int)sizeof(T) / 16), stride(TileSmem<T>(d).stride()) {
    magic = ((1u << 20) + pieces - 1) / pieces;       // exact i / pieces for i < 2048
  }
  __device__ __forceinline__ void fetch(const TileMask& g, const int32_t* perm, int tile) {
    const int t = tile * kCols + (threadIdx.x & 31);
    vslot = g.start + t;
    tok = -1;
    if (t < g.count) {
      const int s = wrap_slot(vslot, g.g.n);
      tok = perm ? perm[s] : s;
    }
  }
  // c1, c2: the two column tensors (one tile each); slots and tokens for the mask
  __device__ __forceinline__ void issue(T* d1, const T* c1, T* d2, const T* c2, int64_t tok_stride,
                                        int* slots, int* toks) {
    if (threadIdx.x < kCols) {
      slots[threadIdx.x] = vslot;
      toks[threadIdx.x] = tok;
    }
    const uint32_t a1 = (uint32_t)__cvta_generic_to_shared(d1);
    const uint32_t a2 = (uint32_t)__cvta_generic_to_shared(d2);
    for (int i = threadIdx.x; i < kCols * pieces; i += kTileThreads) {   // whole warps
      const int r = (int)((uint32_t)i * magic >> 20), p = i - r * pieces;
      const int t = __shfl_sync(0xffffffffu, tok, r);
      const uint32_t bytes = t < 0 ? 0u : 16u;         // 0: zero-filled
      const int64_t off = (int64_t)max(t, 0) * tok_stride + p * (16 / (int)sizeof(T));
      const uint32_t at = (uint32_t)(r * stride * (int)sizeof(T) + 16 * p);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                   ::"r"(a1 + at), "l"(c1 + off), "r"(bytes) : "memory");
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                   ::"r"(a2 + at), "l"(c2 + off), "r"(bytes) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
};

// s[r][c] = rows[r] . cols[c] for 4 rows and 2 columns (cols kstep elements apart); packed
// two-element fused multiply-adds along d.
template <typename T>
__device__ __forceinline__ void tile_dot(float (&s)[4][2], const float* rows, int row_stride,
                                         const T* cols, int kstep, int d) {
  float2 acc[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int x = 0; x < d; x += 4) {
    const float4 k0 = ld4(cols + x), k1 = ld4(cols + kstep + x);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 q = ld4(rows + r * row_stride + x);
      acc[r][0] = __ffma2_rn(make_float2(q.x, q.y), make_float2(k0.x, k0.y), acc[r][0]);
      acc[r][1] = __ffma2_rn(make_float2(q.x, q.y), make_float2(k1.x, k1.y), acc[r][1]);
      acc[r][0] = __ffma2_rn(make_float2(q.z, q.w), make_float2(k0.z, k0.w), acc[r][0]);
      acc[r][1] = __ffma2_rn(make_float2(q.z, q.w), make_float2(k1.z, k1.w), acc[r][1]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    s[r][0] = acc[r][0].x + acc[r][0].y;
    s[r][1] = acc[r][1].x + acc[r][1].y;
  }
}

// o[r][4 cg + x] += sum_k p[k][r] cols[k][64 cg + 4 tx + x]; p: [32][8] fp32, this thread's 4 rows;
// packed over two columns
template <typename T, int NCG>
__device__ __forceinline__ void tile_accumulate(float (&o)[4][4 * NCG], const float* p,
                                                const T* cols, int stride, int tx, int d) {
#pragma unroll 4
  for (int k = 0; k < kCols; ++k) {
    const float4 w = ld4(p + 8 * k);
    const float wr[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int cg = 0; cg < NCG; ++cg) {
      const float4 v = ld4(cols + k * stride + min(64 * cg + 4 * tx, d - 4));
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float2 w2 = make_float2(wr[r], wr[r]);
        const float2 a = __ffma2_rn(w2, make_float2(v.x, v.y), make_float2(o[r][4 * cg], o[r][4 * cg + 1]));
        const float2 b = __ffma2_rn(w2, make_float2(v.z, v.w), make_float2(o[r][4 * cg + 2], o[r][4 * cg + 3]));
        o[r][4 * cg] = a.x;
        o[r][4 * cg + 1] = a.y;
        o[r][4 * cg + 2] = b.x;
        o[r][4 * cg + 3] = b.y;
      }
    }
  }
}

// The same, leaving out the pairs that sees(r, k) hides: their weight is 0, and 0 times an infinity or
// a NaN would reach rows that do not see that column.  One select per pair more than the tile needs
// otherwise, so a tile's walk is repeated with it only where the plain sums ended in a NaN.
template <typename T, int NCG, typename F>
__device__ __forceinline__ void tile_accumulate_seen(float (&o)[4][4 * NCG], const float* p,
                                                     const T* cols, int stride, int tx, int d, F&& sees) {
#pragma unroll 1
  for (int k = 0; k < kCols; ++k) {
    const float4 w = ld4(p + 8 * k);
    const float wr[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int cg = 0; cg < NCG; ++cg) {
      const float4 v = ld4(cols + k * stride + min(64 * cg + 4 * tx, d - 4));
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (!sees(r, k)) continue;
        o[r][4 * cg] = fmaf(wr[r], v.x, o[r][4 * cg]);
        o[r][4 * cg + 1] = fmaf(wr[r], v.y, o[r][4 * cg + 1]);
        o[r][4 * cg + 2] = fmaf(wr[r], v.z, o[r][4 * cg + 2]);
        o[r][4 * cg + 3] = fmaf(wr[r], v.w, o[r][4 * cg + 3]);
      }
    }
  }
}

template <int N>
__device__ __forceinline__ bool any_nan(const float (&o)[4][N]) {
  bool nan = false;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < N; ++c) nan |= isnan(o[r][c]);
  return nan;
}

// Dynamic shared memory above 48 KB has to be asked for.
inline cudaError_t allow_smem(const void* kernel, int bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace
}  // namespace sa

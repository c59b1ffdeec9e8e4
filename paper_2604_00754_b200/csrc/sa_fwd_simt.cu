// General forward kernel on the CUDA cores: any d (multiple of 8, <= 256), fp32 or bf16
// storage, fp32 arithmetic.  It serves the fp32 configuration (a single-pass TF32 product
// cannot hold 1e-4 max-abs error), odd shapes and strides, and is the on-device cross-check
// of the tensor-core path.
//
// A CTA of 128 threads owns 32 query rows (consecutive slots of one head) and walks the keys
// any of them can see, 32 at a time: rows of K and V are gathered through perm with cp.async
// into one of two shared-memory buffers while the other one is worked on.  Scores and the
// weighted sum are register-tiled products (4 rows x 2 keys, 4 rows x 4 columns per 64 per
// thread): a K or V row is read from memory once per 32 queries, and a shared-memory word is
// used by 4 fused multiply-adds.  Bound: the FMA pipe and shared-memory reads in about equal
// parts (8 wavefronts per 32 packed FMAs).  32 rows and not 64, because narrow windows pay
// (32 + w - 1) / w of their keys, and small calls need the CTAs.
#include "sa_common.cuh"
#include "sa_simt_common.cuh"

namespace sa {
namespace {

typedef int IntCols[kCols];

// NCG: groups of 64 output columns (d <= 64 * NCG).  Without SEEN nothing is stored and false returned
// where a sum of this CTA ended in a NaN: see tile_accumulate_seen.
template <typename T, int NCG, bool SEEN>
__device__ __forceinline__ bool fwd_tile(const FwdArgs& a, unsigned char* smem_raw, IntCols* s_slot,
                                         IntCols* s_tok) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tx = lane & 15, half = lane >> 4;         // key / column index, row group of the warp
  const int row0 = warp * 8 + half * 4;               // this thread's four rows
  const int hq = blockIdx.y, b = blockIdx.z, s0 = blockIdx.x * kRows;
  const int hk = hq / (a.Hq / a.Hkv), d = a.d;
  const int32_t* perm = a.swa ? nullptr : a.perm + (size_t)b * a.n;
  const TileSmem<T> sm(d);
  float* qs = reinterpret_cast<float*>(smem_raw);
  T* kv = reinterpret_cast<T*>(smem_raw + sm.rows_bytes());       // K0 V0 K1 V1
  float* ps = reinterpret_cast<float*>(smem_raw + sm.rows_bytes() + 4 * sm.col_bytes());
  float* pw = ps + warp * (kCols * 8);                // this warp's probabilities [key][8 rows]

  const T* kbase = (const T*)a.k + b * a.ks[0] + hk * a.ks[1];
  const T* vbase = (const T*)a.v + b * a.ks[0] + hk * a.ks[1];
  const float scale2 = a.scale * kLog2e;
  load_rows<T>(qs, d, (const T*)a.q + b * a.qs[0] + hq * a.qs[1], a.qs[2], perm, s0, a.n, scale2);

  const TileMask g(a.n, a.w, a.flags, a.swa, s0, false);
  int qslot[4], qtok[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    qslot[r] = s0 + row0 + r;
    const int sl = min(qslot[r], a.n - 1);
    qtok[r] = perm ? perm[sl] : sl;
  }
  ColLoader<T> ld(d);
  auto fetch = [&](int t) { ld.fetch(g, perm, t); };
  auto issue = [&](int buf) {
    ld.issue(kv + (2 * buf) * sm.col_elems(), kbase, kv + (2 * buf + 1) * sm.col_elems(), vbase,
             a.ks[2], s_slot[buf], s_tok[buf]);
  };

  float o[4][4 * NCG];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4 * NCG; ++c) o[r][c] = 0.f;
  float m[4], l[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) { m[r] = -INFINITY; l[r] = 0.f; }

  fetch(0);
  issue(0);
  if (g.tiles > 1) fetch(1);
  for (int j = 0; j < g.tiles; ++j) {
    const int buf = j & 1;
    if (j + 1 < g.tiles) {
      issue(buf ^ 1);
      if (j + 2 < g.tiles) fetch(j + 2);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const T* ks_ = kv + (2 * buf) * sm.col_elems();
    const T* vs_ = kv + (2 * buf + 1) * sm.col_elems();
    float s[4][2];
    tile_dot<T>(s, qs + row0 * sm.row_elems(), sm.row_elems(), ks_ + tx * sm.stride(),
                16 * sm.stride(), d);
    float mt[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) mt[r] = m[r];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int sk = s_slot[buf][tx + 16 * c], jk = s_tok[buf][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (!g.sees(qslot[r], qtok[r], sk, jk)) s[r][c] = -INFINITY;
        mt[r] = fmaxf(mt[r], s[r][c]);
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) mt[r] = fmaxf(mt[r], __shfl_xor_sync(0xffffffffu, mt[r], x));
      const float ref = mt[r] == -INFINITY ? 0.f : mt[r];
      const float corr = exp2f(m[r] - ref);            // m = -inf gives 0
      m[r] = mt[r];
      s[r][0] = exp2f(s[r][0] - ref);
      s[r][1] = exp2f(s[r][1] - ref);
      l[r] = fmaf(l[r], corr, s[r][0] + s[r][1]);
#pragma unroll
      for (int c = 0; c < 4 * NCG; ++c) o[r][c] *= corr;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
      *reinterpret_cast<float4*>(pw + (tx + 16 * c) * 8 + 4 * half) =
          make_float4(s[0][c], s[1][c], s[2][c], s[3][c]);
    __syncwarp();
    if constexpr (SEEN)
      tile_accumulate_seen<T, NCG>(o, pw + 4 * half, vs_, sm.stride(), tx, d, [&](int r, int k) {
        return g.sees(qslot[r], qtok[r], s_slot[buf][k], s_tok[buf][k]);
      });
    else
      tile_accumulate<T, NCG>(o, pw + 4 * half, vs_, sm.stride(), tx, d);
    __syncthreads();                                  // the buffer may be refilled now
  }
  if (!SEEN && __syncthreads_or(any_nan(o))) return false;

  float g_this = 1.f, g_other = 0.f;
  if (a.gate_logits) {
    const float l_sa = a.gate_logits[hq], l_swa = a.gate_logits[a.Hq + hq];
    const float s_sa = 1.f / (1.f + __expf(-l_sa)), s_swa = 1.f / (1.f + __expf(-l_swa));
    g_this = a.swa ? s_swa : s_sa;
    g_other = a.swa ? s_sa : s_swa;
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int x = 8; x > 0; x >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], x);
    if (qslot[r] >= a.n) continue;
    const float inv_l = 1.f / l[r];
    const int64_t off = b * a.qs[0] + hq * a.qs[1] + (int64_t)qtok[r] * a.qs[2];
#pragma unroll
    for (int cg = 0; cg < NCG; ++cg) {
      const int c = 64 * cg + 4 * tx;
      if (c >= d) continue;
      float4 v = make_float4(o[r][4 * cg] * inv_l, o[r][4 * cg + 1] * inv_l,
                             o[r][4 * cg + 2] * inv_l, o[r][4 * cg + 3] * inv_l);
      if (a.y_branch) {   // combine what was stored, as the backward pass will read it
        st4((T*)a.y_branch + off + c, v);
        v = round4<T>(v);
      }
      if (a.gate_logits) {
        v.x *= g_this; v.y *= g_this; v.z *= g_this; v.w *= g_this;
        if (a.y_other) {
          const float4 w4 = ld4((const T*)a.y_other + off + c);
          v.x = fmaf(g_other, w4.x, v.x); v.y = fmaf(g_other, w4.y, v.y);
          v.z = fmaf(g_other, w4.z, v.z); v.w = fmaf(g_other, w4.w, v.w);
        }
      }
      if (a.y) st4((T*)a.y + off + c, v);
    }
    if (a.lse && tx == 0)
      a.lse[((size_t)b * a.Hq + hq) * a.n + qtok[r]] = (m[r] + log2f(l[r])) * kLn2;
  }
  return true;
}

template <typename T, int NCG>
__device__ __noinline__ void fwd_tile_seen(const FwdArgs& a, unsigned char* smem_raw, IntCols* s_slot,
                                           IntCols* s_tok) {
  fwd_tile<T, NCG, true>(a, smem_raw, s_slot, s_tok);
}

template <typename T, int NCG>
__global__ void __launch_bounds__(kTileThreads) fwd_tile_kernel(const __grid_constant__ FwdArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_slot[2][kCols], s_tok[2][kCols];
  grid_dependency_wait();
  grid_dependents_launch();
  if (a.abort_flag && *a.abort_flag) return;          // an earlier check rejected perm/inv
  if (!fwd_tile<T, NCG, false>(a, smem_raw, s_slot, s_tok))
    fwd_tile_seen<T, NCG>(a, smem_raw, s_slot, s_tok);
}

template <typename T, int NCG>
cudaError_t go(const FwdArgs& a, cudaStream_t st) {
  const TileSmem<T> sm(a.d);
  const int smem = sm.rows_bytes() + 4 * sm.col_bytes() + kTileThreads / 32 * kCols * 8 * 4;
  cudaError_t e = allow_smem((const void*)fwd_tile_kernel<T, NCG>, smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(fwd_tile_kernel<T, NCG>, dim3((a.n + kRows - 1) / kRows, a.Hq, a.B),
                          dim3(kTileThreads), smem, st, a);
}

template <typename T>
cudaError_t by_width(const FwdArgs& a, cudaStream_t st) {
  if (a.d <= 64) return go<T, 1>(a, st);
  return a.d <= 128 ? go<T, 2>(a, st) : go<T, 4>(a, st);
}

}  // namespace

cudaError_t launch_fwd_simt(const FwdArgs& a, int dtype, cudaStream_t st) {
  const cudaError_t e = dtype == SA_F32 ? by_width<float>(a, st) : by_width<__nv_bfloat16>(a, st);
  if (e != cudaSuccess) return e;
  bump_launches();
  return cudaGetLastError();
}

}  // namespace sa

// Rotary position embedding with ORIGINAL token positions (the paper applies RoPE to Q and K
// before the shuffle: Sec. 4.2, attention paragraph of App. B).  This file holds the table of
// angles and the stand-alone pass over one tensor, or over Q and K in one launch; the forward
// kernels can apply the same rotation inside their row gather (sa_forward_rope).
//
// Layout of the rotation: dimension c of the first half of a head is paired with dimension
// c + d/2; token t turns the pair by t * base^(-2c/d).
#include "sa_common.cuh"

namespace sa {
namespace {

__global__ void rope_table_kernel(int n, int half, double log2_base_over_half, float* cs,
                                  float* sn) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n * half) return;
  const int t = (int)(i / half), c = (int)(i % half);
  // base^(-2c/d) = 2^(-c * log2(base) / half), in double: the angle reaches n radians
  const double ang = (double)t * exp2(-(double)c * log2_base_over_half);
  double s, co;
  sincos(ang, &s, &co);
  cs[i] = (float)co;
  sn[i] = (float)s;
}

// One thread per 8 consecutive dimensions of the first half of a row and their partners.
// General form (any even d, any dtype): element by element.
template <typename T>
__global__ void rope_apply_kernel(const T* __restrict__ x, T* __restrict__ out, int B, int H,
                                  int n, int d, int64_t s0, int64_t s1, int64_t s2,
                                  const float* __restrict__ cs, const float* __restrict__ sn,
                                  float sign) {
  const int half = d / 2, groups = (half + 7) / 8;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * H * n * groups) return;
  const int g = (int)(i % groups);
  const int64_t row = i / groups;
  const int t = (int)(row % n), h = (int)((row / n) % H), b = (int)(row / ((int64_t)n * H));
  const int64_t off = b * s0 + h * s1 + (int64_t)t * s2;
  for (int c = 8 * g; c < min(8 * g + 8, half); ++c) {
    const float co = cs[(int64_t)t * half + c], si = sign * sn[(int64_t)t * half + c];
    const float x1 = to_f32(x[off + c]), x2 = to_f32(x[off + c + half]);
    out[off + c] = from_f32<T>(fmaf(x1, co, -x2 * si));
    out[off + c + half] = from_f32<T>(fmaf(x2, co, x1 * si));
  }
}

// One tensor of a rotation pass: [B,H,n,d] with element strides (d contiguous).
struct RopeTensor {
  const __nv_bfloat16* x;
  __nv_bfloat16* out;
  int H;
  int64_t s0, s1, s2;
};

// bf16 with d a multiple of 16: the same arithmetic with 16-byte accesses (8 dimensions of
// each half per thread; consecutive threads take consecutive pieces of a row).  HBM-bound: one
// read and one write of the tensors.  blockIdx.y counts the heads of the first tensor, then
// those of the second, so that Q and K share a launch.
__global__ void __launch_bounds__(256)
rope_apply_bf16_kernel(const RopeTensor ta, const RopeTensor tb, int n, int d,
                       const float* __restrict__ cs, const float* __restrict__ sn, float sign) {
  const int half = d / 2, groups = half / 8;
  const int i = blockIdx.x * 256 + threadIdx.x;
  grid_dependency_wait();
  if (i >= n * groups) return;
  const int t = i / groups, g = i - t * groups, b = blockIdx.z;
  const bool first = (int)blockIdx.y < ta.H;
  const RopeTensor& r = first ? ta : tb;
  const int h = first ? blockIdx.y : blockIdx.y - ta.H;
  const __nv_bfloat16* x = r.x;
  __nv_bfloat16* out = r.out;
  const int64_t off = b * r.s0 + h * r.s1 + (int64_t)t * r.s2 + 8 * g;
  const uint4 a1 = *reinterpret_cast<const uint4*>(x + off);
  const uint4 a2 = *reinterpret_cast<const uint4*>(x + off + half);
  const float4 c0 = *reinterpret_cast<const float4*>(cs + (int64_t)t * half + 8 * g);
  const float4 c1 = *reinterpret_cast<const float4*>(cs + (int64_t)t * half + 8 * g + 4);
  const float4 q0 = *reinterpret_cast<const float4*>(sn + (int64_t)t * half + 8 * g);
  const float4 q1 = *reinterpret_cast<const float4*>(sn + (int64_t)t * half + 8 * g + 4);
  const float co[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
  const float si[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
  const __nv_bfloat162* h1 = reinterpret_cast<const __nv_bfloat162*>(&a1);
  const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&a2);
  uint4 o1, o2;
  __nv_bfloat162* r1 = reinterpret_cast<__nv_bfloat162*>(&o1);
  __nv_bfloat162* r2 = reinterpret_cast<__nv_bfloat162*>(&o2);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 x1 = __bfloat1622float2(h1[k]), x2 = __bfloat1622float2(h2[k]);
    const float s_lo = sign * si[2 * k], s_hi = sign * si[2 * k + 1];
    r1[k] = __floats2bfloat162_rn(fmaf(x1.x, co[2 * k], -x2.x * s_lo),
                                  fmaf(x1.y, co[2 * k + 1], -x2.y * s_hi));
    r2[k] = __floats2bfloat162_rn(fmaf(x2.x, co[2 * k], x1.x * s_lo),
                                  fmaf(x2.y, co[2 * k + 1], x1.y * s_hi));
  }
  *reinterpret_cast<uint4*>(out + off) = o1;
  *reinterpret_cast<uint4*>(out + off + half) = o2;
}

}  // namespace

// n * (d / 16) pieces of a head fit the 32-bit index of the 16-byte kernel.
static bool rope_fast(int B, int n, int d, int dtype) {
  return dtype == SA_BF16 && d % 16 == 0 && B <= 65535 && (int64_t)n * (d / 16) < (1ll << 31) - 256;
}

cudaError_t launch_rope_apply(const void* x, void* out, int B, int H, int n, int d,
                              const int64_t s[3], int dtype, const float* cs, const float* sn,
                              bool inverse, cudaStream_t st) {
  const float sign = inverse ? -1.f : 1.f;
  if (rope_fast(B, n, d, dtype)) {
    const RopeTensor t{(const __nv_bfloat16*)x, (__nv_bfloat16*)out, H, s[0], s[1], s[2]};
    const unsigned blocks = ((unsigned)n * (d / 16) + 255) / 256;
    bump_launches();
    return launch_dependent(rope_apply_bf16_kernel, dim3(blocks, H, B), dim3(256), 0, st, t, t, n, d,
                            cs, sn, sign);
  } else {
    const int64_t total = (int64_t)B * H * n * ((d / 2 + 7) / 8);
    const unsigned blocks = (unsigned)((total + 255) / 256);
    if (dtype == SA_BF16)
      rope_apply_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(
          (const __nv_bfloat16*)x, (__nv_bfloat16*)out, B, H, n, d, s[0], s[1], s[2], cs, sn, sign);
    else
      rope_apply_kernel<float><<<blocks, 256, 0, st>>>((const float*)x, (float*)out, B, H, n, d,
                                                       s[0], s[1], s[2], cs, sn, sign);
  }
  bump_launches();
  return cudaGetLastError();
}

cudaError_t launch_rope_qk(const void* q, void* qr, int Hq, const int64_t qs[3], const void* k,
                           void* kr, int Hkv, const int64_t ks[3], int B, int n, int d, int dtype,
                           const float* cs, const float* sn, cudaStream_t st) {
  if (!rope_fast(B, n, d, dtype) || Hq + Hkv > 65535) {
    const cudaError_t e = launch_rope_apply(q, qr, B, Hq, n, d, qs, dtype, cs, sn, false, st);
    return e != cudaSuccess ? e
                            : launch_rope_apply(k, kr, B, Hkv, n, d, ks, dtype, cs, sn, false, st);
  }
  const RopeTensor a{(const __nv_bfloat16*)q, (__nv_bfloat16*)qr, Hq, qs[0], qs[1], qs[2]};
  const RopeTensor b{(const __nv_bfloat16*)k, (__nv_bfloat16*)kr, Hkv, ks[0], ks[1], ks[2]};
  const unsigned blocks = ((unsigned)n * (d / 16) + 255) / 256;
  bump_launches();
  return launch_dependent(rope_apply_bf16_kernel, dim3(blocks, Hq + Hkv, B), dim3(256), 0, st, a, b, n,
                          d, cs, sn, 1.f);
}

}  // namespace sa

extern "C" sa_status sa_rope_table(int32_t n, int32_t d, double base, float* rope_cos,
                                   float* rope_sin, sa_stream_t stream) {
  using namespace sa;
  if (n < 1 || d < 2 || d % 2 != 0 || !(base > 0.0) || !rope_cos || !rope_sin)
    return SA_ERR_INVALID_ARG;
  const int half = d / 2;
  const int64_t total = (int64_t)n * half;
  rope_table_kernel<<<(unsigned)((total + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      n, half, log2(base) / half, rope_cos, rope_sin);
  bump_launches();
  return cudaGetLastError() == cudaSuccess ? SA_OK : SA_ERR_CUDA;
}

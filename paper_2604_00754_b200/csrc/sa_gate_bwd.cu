// Backward of the projection gates (Eq. 5-6): with z = y w^T, g = sigmoid(z), out = g * y,
//   dz = dout * y * g * (1 - g),   dw = dz^T y,   dy = dout * g + dz w      (per path).
// Three contractions per path, all on the 5th-generation tensor cores through one kernel
// template (128 x 256 output tiles, or 128 x 128 for small products, TMA ring,
// double-buffered fp32 accumulators in tensor memory, eight epilogue warps):
//   kDz: z = y w^T        (both operands K-major);  epilogue writes dz and dout * g
//   kDy: dz w             (w read with its rows as the contraction index: N-major operand);
//                          epilogue adds dout * g and writes dy
//   kDw: dz^T y           (both operands read with their rows as the contraction index);
//                          epilogue writes dw, or fp32 products of parts of the rows
// A plain kernel per step serves fp32 and sizes the tensor-core path does not take.
//
// Every mbarrier wait is bounded; on expiry the CTA records SA_ERR_TIMEOUT in the device
// status word, stops issuing work, drains what it started and returns.
#include "sa_gemm_common.cuh"

namespace sa {
namespace {

// kFwd: the forward's sigmoid(y w^T) * y; kFwdAdd: the same added to what out already holds
enum BwdMode { kDz = 0, kDy = 1, kDw = 2, kFwd = 3, kFwdAdd = 4 };

constexpr int kT = 128, kBK = 64;                  // output tiles of 128 rows, K chunks of 64
constexpr int kATileBytes = kT * kBK * 2;          // A of one K chunk, either major: 16 KB
constexpr int kChunk = 64 * kBK * 2;               // 64 rows x 64 columns: one box of a row-contracted operand
constexpr int kEpiTile = kT * 128;                 // epilogue: 128 rows x 128 bytes, 16 KB
// Shared memory: the operand ring, then the epilogue's tiles, for each half of the output columns
// as many as a chunk of 64 columns has inputs (outputs are written in place): kDz y and dout,
// kFwd y, kFwdAdd y and out, kDy dout * g, kDw a tile for the output alone.
template <int MODE> struct Epi {
  static constexpr int kIn = MODE == kDw ? 0 : MODE == kDy || MODE == kFwd ? 1 : 2;
  static constexpr int kTiles = kIn == 2 ? 2 : 1;                // per half
  static constexpr int kRingBytes = (kIn == 2 ? 9 : 12) * kATileBytes;
};
// TN: columns of the output tile.  256 halves the operand bytes per flop of the B side; which of the
// two a product takes is decided by forward_wide, wide_waves and plan_dw below.  A stage is one K chunk
// of A + B, 48 or 32 KB.
template <int MODE, int TN> struct Tile {
  static constexpr int kBTileBytes = TN * kBK * 2;
  static constexpr int kStageBytes = kATileBytes + kBTileBytes;
  static constexpr int kStages = Epi<MODE>::kRingBytes / kStageBytes;       // 3 to 6
};
constexpr int kMaxStages = 6;
constexpr int kThreadsB = 384;                     // TMA, MMA, eight epilogue warps, two movers
constexpr int kBarFull = 0, kBarEmpty = kMaxStages, kBarAccFull = 2 * kMaxStages,
              kBarAccEmpty = kBarAccFull + 2, kBarIn = kBarAccEmpty + 2, kBarOut = kBarIn + 2,
              kNumBars = kBarOut + 2;
template <int MODE> struct Smem {
  static constexpr int kOffEpi = Epi<MODE>::kRingBytes;
  static constexpr int kOffBars = kOffEpi + 2 * Epi<MODE>::kTiles * kEpiTile;
  static constexpr int kOffMisc = kOffBars + kNumBars * 8;
  static constexpr int kBytes = kOffMisc + 16;
};

struct BwdGateParams {
  int m_rows, n_cols;              // extent of the product
  int tiles_m, tiles_n, k_chunks;  // K chunks of 64
  int splits, per_split;           // kDw: the K chunks go in `splits` parts of `per_split`
  int* status;
};

__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// bit 15: A is MN-major, bit 16: B is MN-major
__host__ __device__ constexpr uint32_t idesc_of(int tn, bool a_mn, bool b_mn) {
  return instr_desc(kT, tn, b_mn) | ((a_mn ? 1u : 0u) << 15);
}
template <int MODE, int TN>
__global__ void __launch_bounds__(kThreadsB, 1)
gate_bwd_kernel(const __grid_constant__ BwdGateParams p, const __grid_constant__ CUtensorMap tm_a,
                const __grid_constant__ CUtensorMap tm_b, const __grid_constant__ CUtensorMap tm_i0,
                const __grid_constant__ CUtensorMap tm_i1, const __grid_constant__ CUtensorMap tm_o0,
                const __grid_constant__ CUtensorMap tm_o1) {
  constexpr bool kAmn = MODE == kDw, kBmn = MODE == kDy || MODE == kDw;
  using TL = Tile<MODE, TN>;
  using SM = Smem<MODE>;
  constexpr int kIn = Epi<MODE>::kIn;
  constexpr int kStages = TL::kStages, kStageBytes = TL::kStageBytes, kTN = TN;
  constexpr int kBlock = 2048 / TN;       // column tiles per block of the tile order
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {
    if (threadIdx.x == 0) atomicCAS(p.status, SA_OK, SA_ERR_CUDA);
    return;
  }
  const uint32_t bar0 = sbase + SM::kOffBars;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + SM::kOffMisc);
  volatile int* gave_up = reinterpret_cast<volatile int*>(smem + SM::kOffMisc + 4);
  if (threadIdx.x == 0) {
    *gave_up = 0;
    grid_dependency_wait();                   // what earlier launches wrote may be read from here on
    note_skip(reinterpret_cast<volatile int*>(smem + SM::kOffMisc + 8), p.status, nullptr);
    for (int i = 0; i < kNumBars; ++i) 
      mbar_init(bar(i), i >= kBarOut ? 128 : i >= kBarIn ? 1 : i >= kBarAccEmpty ? 256 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dependents_launch();
  const uint32_t tmem = *tmem_slot;
  SA_LEAVE_IF_SKIPPED(reinterpret_cast<volatile int*>(smem + SM::kOffMisc + 8), 1, tmem, 512u)
  const int tiles = p.tiles_m * p.tiles_n, total = MODE == kDw ? tiles * p.splits : tiles;
  // blocks of 2048 columns, row tile by row tile inside a block (operand slices stay in L2)
  auto origin = [&](int item, int* m0, int* n0) {
    const int tile = MODE == kDw ? item % tiles : item;
    const int per_block = p.tiles_m * kBlock;
    const int nb = tile / per_block, rem = tile - nb * per_block;
    const int width = min(kBlock, p.tiles_n - nb * kBlock);
    *m0 = (rem / width) * kT;
    *n0 = (nb * kBlock + rem % width) * kTN;
  };
  // the K chunks of an item: all, or (kDw) those of its part
  auto chunks = [&](int item, int* first, int* last) {
    const int part = MODE == kDw ? item / tiles : 0;
    *first = MODE == kDw ? part * p.per_split : 0;
    *last = MODE == kDw ? min(*first + p.per_split, p.k_chunks) : p.k_chunks;
  };
  // the epilogue's chunks: 128 bytes of output columns, the tile's columns in two halves
  const bool parts = MODE == kDw && p.splits > 1;
  const int chunk_cols = parts ? 32 : 64, half_chunks = (kTN / 2) / chunk_cols;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t use = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
        int m0, n0;
        origin(tile, &m0, &n0);
        int kc, k_end;
        chunks(tile, &kc, &k_end);
        for (; kc < k_end && ok; ++kc, ++use) {
          const uint32_t s = use % kStages;
          if (use >= (uint32_t)kStages)
            ok = mbar_wait(bar(kBarEmpty + s), (use / kStages - 1) & 1u, gave_up, p.status);
          if (!ok) break;
          const uint32_t da = sbase + s * kStageBytes, db = da + kATileBytes, fb = bar(kBarFull + s);
          mbar_expect_tx(fb, kStageBytes);
          const int k0 = kc * kBK;                                      // past the end: zeros
          if (kAmn) {
#pragma unroll
            for (int c = 0; c < kT / 64; ++c) tma_load_2d(da + c * kChunk, &tm_a, m0 + 64 * c, k0, fb);
          } else {
            tma_load_2d(da, &tm_a, k0, m0, fb);
          }
          if (kBmn) {
#pragma unroll
            for (int c = 0; c < kTN / 64; ++c) tma_load_2d(db + c * kChunk, &tm_b, n0 + 64 * c, k0, fb);
          } else {
            tma_load_2d(db, &tm_b, k0, n0, fb);
          }
        }
      }
      if (!ok || *gave_up) {   // loads started but never consumed must land before smem goes
        const uint32_t first = use > (uint32_t)kStages ? use - kStages : 0u;
        for (uint32_t u = first; u < use; ++u)
          for (int tries = 0; tries < 100000; ++tries) {
            if (mbar_try(bar(kBarFull + u % kStages), (u / kStages) & 1u)) break;
            __nanosleep(100);
          }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // -------------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_of(TN, kAmn, kBmn);
      constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
      constexpr uint32_t kLoK = (16u >> 4) << 16;                       // K-major operand
      constexpr uint32_t kLoMN = ((uint32_t)kChunk >> 4) << 16;           // next 64 columns
      constexpr uint32_t kStepK = 32u >> 4, kStepMN = 2048u >> 4;         // one K step of 16
      uint32_t use = 0, it = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x, ++it) {
        const uint32_t buf = it & 1u;
        if (it >= 2)
          ok = mbar_wait(bar(kBarAccEmpty + buf), (it / 2 - 1) & 1u, gave_up, p.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * kTN;
        int kc, k_end;
        chunks(tile, &kc, &k_end);
        for (uint32_t acc = 0; kc < k_end && ok; ++kc, ++use, acc = 1) {
          const uint32_t s = use % kStages;
          ok = mbar_wait(bar(kBarFull + s), (use / kStages) & 1u, gave_up, p.status);
          if (!ok) break;
          tc_fence_after();
          const uint32_t la = (sbase + s * kStageBytes) >> 4;
          const uint64_t a0 = desc64(la | (kAmn ? kLoMN : kLoK), kDescHi);
          const uint64_t b0 = desc64((la + (kATileBytes >> 4)) | (kBmn ? kLoMN : kLoK), kDescHi);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            mma_ss(d, a0 + ks * (kAmn ? kStepMN : kStepK), b0 + ks * (kBmn ? kStepMN : kStepK),
                   idesc, ks > 0 ? 1u : acc);
          tc_commit(bar(kBarEmpty + s));
        }
        if (ok) tc_commit(bar(kBarAccFull + buf));
      }
    }
    __syncwarp();
  } else if (warp >= 10) {
    // --------------------------------- movers: the epilogue's tiles of one half of the columns
    // A thread holds a row, so reading and writing global memory from the registers touches 32
    // lines per instruction (30000 cycles for a 128 x 256 tile of kDz, whose products take 8200).
    // TMA brings a chunk of 64 columns x 128 rows of every input into shared memory, the row
    // threads write the outputs in their place, and TMA takes them out; the next chunk comes as
    // soon as this one has been read.
    if (lane == 0) {
      const int hf = warp - 10;
      const uint32_t buf0 = sbase + SM::kOffEpi + hf * Epi<MODE>::kTiles * kEpiTile;
      const uint32_t in_bar = bar(kBarIn + hf), out_bar = bar(kBarOut + hf);
      uint32_t e = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total && ok; tile += gridDim.x) {
        int m0, n0;
        origin(tile, &m0, &n0);
        for (int c = 0; c < half_chunks && ok; ++c, ++e) {
          const int col = n0 + hf * (kTN / 2) + c * chunk_cols;
          if (col >= p.n_cols) break;
          if (e) bulk_wait_read();
          if (kIn) {
            mbar_expect_tx(in_bar, kIn * kEpiTile);
            tma_load_2d(buf0, &tm_i0, col, m0, in_bar);
            if (kIn > 1) tma_load_2d(buf0 + kEpiTile, &tm_i1, col, m0, in_bar);
          } else {
            mbar_arrive(in_bar);
          }
          ok = mbar_wait(out_bar, e & 1u, gave_up, p.status);
          if (!ok) break;
          if (parts) tma_store_3d(&tm_o0, buf0, col, m0, tile / tiles);
          else tma_store_2d(&tm_o0, buf0, col, m0);
          if (MODE == kDz) tma_store_2d(&tm_o1, buf0 + kEpiTile, col, m0);
          bulk_commit();
        }
      }
      if (!ok && kIn)          // the last inputs must land before the shared memory goes away
        for (int tries = 0; tries < 100000 && !mbar_try(in_bar, e & 1u); ++tries) __nanosleep(100);
      bulk_wait();
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------- epilogue (warps 2-9)
    // one row per thread; warps 2-5 take the first half of the tile's columns, 6-9 the other
    const int half = (warp - 2) >> 2;
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t own = sbase + SM::kOffEpi + half * Epi<MODE>::kTiles * kEpiTile + row * 128;
    auto piece = [&](int j) { return own + ((j ^ (row & 7)) << 4); };   // 16 bytes of the row
    uint32_t it = 0, e = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total; tile += gridDim.x, ++it) {
      const uint32_t buf = it & 1u;
      int m0, n0;
      origin(tile, &m0, &n0);
      ok = mbar_wait(bar(kBarAccFull + buf), (it / 2) & 1u, gave_up, p.status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < half_chunks; ++c, ++e) {
        const int col = half * (kTN / 2) + c * chunk_cols;
        if (n0 + col >= p.n_cols) break;
        const uint32_t acc_at = tmem + lane_addr + buf * kTN + col;
        uint32_t acc[32];
        tmem_ld32(acc_at, acc);
        ok = mbar_wait(bar(kBarIn + half), e & 1u, gave_up, p.status);
        ok = __all_sync(0xffffffffu, ok);
        tmem_wait_ld();
        if (!ok) break;
        if (parts) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t st[4] = {acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]};
            sts128(piece(j), st);
          }
        } else {
#pragma unroll
          for (int s2 = 0; s2 < 2; ++s2) {
            if (s2) {
              tmem_ld32(acc_at + 32, acc);
              tmem_wait_ld();
            }
#pragma unroll
            for (int x8 = 0; x8 < 4; ++x8) {
              const uint32_t at = piece(4 * s2 + x8);
              float v8[8];
#pragma unroll
              for (int x = 0; x < 8; ++x) v8[x] = __uint_as_float(acc[8 * x8 + x]);
              uint32_t f0[4], f1[4], st[4];
              if (kIn) lds128(f0, at);
              if (kIn > 1) lds128(f1, at + kEpiTile);
              __nv_bfloat162* hs = reinterpret_cast<__nv_bfloat162*>(st);
              const __nv_bfloat162* h0 = reinterpret_cast<const __nv_bfloat162*>(f0);
              const __nv_bfloat162* h1 = reinterpret_cast<const __nv_bfloat162*>(f1);
              if (MODE == kDz) {
                uint32_t st2[4];
                __nv_bfloat162* hs2 = reinterpret_cast<__nv_bfloat162*>(st2);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                  const float g0 = logistic(v8[2 * x]), g1 = logistic(v8[2 * x + 1]);
                  const float d0 = __low2float(h1[x]), d1 = __high2float(h1[x]);
                  hs[x] = __floats2bfloat162_rn(d0 * __low2float(h0[x]) * g0 * (1.f - g0),
                                                d1 * __high2float(h0[x]) * g1 * (1.f - g1));
                  hs2[x] = __floats2bfloat162_rn(d0 * g0, d1 * g1);
                }
                sts128(at + kEpiTile, st2);
              } else {
                if (MODE == kFwd || MODE == kFwdAdd) {
#pragma unroll
                  for (int x = 0; x < 4; ++x) {
                    v8[2 * x] = logistic(v8[2 * x]) * __low2float(h0[x]);
                    v8[2 * x + 1] = logistic(v8[2 * x + 1]) * __high2float(h0[x]);
                  }
                }
                if (MODE == kDy || MODE == kFwdAdd) {
                  const __nv_bfloat162* ha = MODE == kDy ? h0 : h1;
#pragma unroll
                  for (int x = 0; x < 4; ++x) {
                    v8[2 * x] += __low2float(ha[x]);
                    v8[2 * x + 1] += __high2float(ha[x]);
                  }
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) hs[x] = __floats2bfloat162_rn(v8[2 * x], v8[2 * x + 1]);
              }
              sts128(at, st);
            }
          }
        }
        fence_proxy_async();
        mbar_arrive(bar(kBarOut + half));
      }
      if (!ok) break;
      tc_fence_before();
      mbar_arrive(bar(kBarAccEmpty + buf));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// dw = the sum of its parts, added in their order; 8 columns per thread.
__global__ void dw_sum_kernel(const float4* __restrict__ part, int splits, int64_t eights,
                              uint4* __restrict__ dw) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  grid_dependency_wait();
  grid_dependents_launch();
  if (i >= eights) return;
  float4 a = part[2 * i], b = part[2 * i + 1];
#pragma unroll 4
  for (int s = 1; s < splits; ++s) {
    const float4 c = part[2 * (s * eights + i)], d = part[2 * (s * eights + i) + 1];
    a.x += c.x; a.y += c.y; a.z += c.z; a.w += c.w;
    b.x += d.x; b.y += d.y; b.z += d.z; b.w += d.w;
  }
  uint4 st;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&st);
  h[0] = __floats2bfloat162_rn(a.x, a.y); h[1] = __floats2bfloat162_rn(a.z, a.w);
  h[2] = __floats2bfloat162_rn(b.x, b.y); h[3] = __floats2bfloat162_rn(b.z, b.w);
  dw[i] = st;
}

// ------------------------------------------------- plain kernels (fp32, other sizes)

template <typename T>
__global__ void dz_simt_kernel(int64_t rows, int dm, const T* __restrict__ dout, int64_t ld_dout,
                               const T* __restrict__ y, int64_t ld_y, const T* __restrict__ w,
                               float* __restrict__ dz, float* __restrict__ dyd) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= rows * dm) return;
  const int64_t r = idx / dm;
  const int o = (int)(idx % dm);
  const T* yr = y + r * ld_y;
  const T* wo = w + (int64_t)o * dm;
  float z = 0.f;
  for (int i = 0; i < dm; ++i) z = fmaf(to_f32(yr[i]), to_f32(wo[i]), z);
  const float g = 1.f / (1.f + expf(-z)), d = to_f32(dout[r * ld_dout + o]);
  dz[idx] = d * to_f32(yr[o]) * g * (1.f - g);
  dyd[idx] = d * g;
}

template <typename T>
__global__ void dy_simt_kernel(int64_t rows, int dm, const float* __restrict__ dz,
                               const float* __restrict__ dyd, const T* __restrict__ w,
                               T* __restrict__ dy, int64_t ld_dy) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= rows * dm) return;
  const int64_t r = idx / dm;
  const int i = (int)(idx % dm);
  float acc = dyd[idx];
  for (int o = 0; o < dm; ++o) acc = fmaf(dz[r * dm + o], to_f32(w[(int64_t)o * dm + i]), acc);
  dy[r * ld_dy + i] = from_f32<T>(acc);
}

template <typename T>
__global__ void dw_simt_kernel(int64_t rows, int dm, const float* __restrict__ dz,
                               const T* __restrict__ y, int64_t ld_y, T* __restrict__ dw) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)dm * dm) return;
  const int o = (int)(idx / dm), i = (int)(idx % dm);
  float acc = 0.f;
  for (int64_t r = 0; r < rows; ++r) acc = fmaf(dz[r * dm + o], to_f32(y[r * ld_y + i]), acc);
  dw[idx] = from_f32<T>(acc);
}

// ------------------------------------------------------------------------------ host

// 128 x 256 tiles take less time than 128 x 128 by their waves: a wide tile's K chunk takes 512
// cycles, a narrow one's `narrow` (about 300, with 64 columns of operands per product more).
bool wide_waves(int64_t rows, int dm, int sms, int narrow) {
  const int64_t tm = (rows + kT - 1) / kT;
  return (tm * ((dm + 255) / 256) + sms - 1) / sms * 512 <=
         (tm * ((dm + 127) / 128) + sms - 1) / sms * narrow;
}

// Forward: the wide kernel, one launch per path, or (false) the fused 128 x 128 one.  One path: from
// half a wide tile per SM on (8000 x 1024: 25.9 -> 19.9 us, 1300 x 2048: 23.0 -> 18.5, 9000 x 768: 19.8
// -> 17.2; even at 5000 x 512, 80 tiles: 13.3 -> 12.7).  Two paths: the fused kernel adds them in fp32
// and rounds once, the wide one rounds the first path before the second launch adds to it (2-norm of
// the error 2.03e-3 of the result's against 1.66e-3), so it serves only from two tiles per SM
// (32768 x 1024: 170 -> 162 us), although it would be faster at some smaller sizes (2000 x 4096: 155 -> 138).
bool forward_wide(int64_t rows, int dm, bool dual, int sms) {
  const int64_t tiles = ((rows + kT - 1) / kT) * ((dm + 255) / 256);
  return dual ? tiles >= 2 * (int64_t)sms : 2 * tiles >= sms;
}

struct Maps { CUtensorMap a, b, i0, i1, o0, o1; };

template <int MODE, int TN>
cudaError_t launch_mode(BwdGateParams p, const Maps& m, int64_t k, int sms, cudaStream_t st) {
  p.tiles_m = (p.m_rows + kT - 1) / kT;
  p.tiles_n = (p.n_cols + TN - 1) / TN;
  p.k_chunks = (int)((k + kBK - 1) / kBK);
  if (p.splits < 1) p.splits = 1;
  p.per_split = (p.k_chunks + p.splits - 1) / p.splits;
  cudaError_t e = cudaFuncSetAttribute(gate_bwd_kernel<MODE, TN>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Smem<MODE>::kBytes);
  if (e != cudaSuccess) return e;
  const int64_t total = (int64_t)p.tiles_m * p.tiles_n * p.splits;
  const unsigned grid = (unsigned)(total < sms ? total : sms);
  bump_launches();
  return launch_dependent(gate_bwd_kernel<MODE, TN>, dim3(grid), dim3(kThreadsB), Smem<MODE>::kBytes,
                          st, p, m.a, m.b, m.i0, m.i1, m.o0, m.o1);
}

// dw contracts over all rows and has few tiles (64 of 128 x 128 at dm = 1024, 148 SMs), so the rows
// go in parts, whose fp32 products dw_sum_kernel adds up.  Tile width and number of parts: the
// cheapest by the cycles that a K chunk (512 or 300, by tile width), an item's start and end (3000)
// and the parts' way through memory (8 bytes per element, 3000 bytes a cycle; 4000 for the launch)
// take.  The parts use the half of the workspace that bf16 dz and dout * g leave, so they are at
// most rows / dm.
// 32768 rows, dm = 1024, nine parts of 128 x 256 tiles: 60 us and 7 us for the sum; the whole
// backward of one path 332 -> 246 us, with the epilogue's tiles by TMA (dm = 512: 224 -> 103).
struct DwPlan { int tn, splits; };
DwPlan plan_dw(int64_t rows, int dm, int sms) {
  const int64_t kc = (rows + kBK - 1) / kBK;
  DwPlan best{128, 1};
  double least = 1e300;
  for (int tn = 128; tn <= 256; tn += 128) {
    const int64_t tiles = (int64_t)((dm + kT - 1) / kT) * ((dm + tn - 1) / tn);
    for (int64_t s = 1; s <= 64 && s <= kc && (s == 1 || s * dm <= rows); ++s) {
      const int64_t per = (kc + s - 1) / s;
      if ((kc + per - 1) / per != s) continue;          // an empty part
      const double waves = (double)((tiles * s + sms - 1) / sms);
      const double cost = waves * (per * (tn == 256 ? 512. : 300.) + 3000.) +
                          (s > 1 ? 4000. + s * (double)dm * dm * 8. / 3000. : 0.);
      if (cost < least) { least = cost; best = {tn, (int)s}; }
    }
  }
  return best;
}

}  // namespace

// Forward of one or two paths with 128 x 256 tiles, one launch per path (the second adds to
// the first's rounded result); false where forward_wide says so, and the caller's fused kernel
// should run instead.
bool gate_forward_wide(int64_t rows, int dm, const void* y_sa, const void* y_swa, int64_t ld_y,
                       const void* w_sa, const void* w_swa, void* out, int64_t ld_out,
                       int* status, int sms, cudaStream_t st, cudaError_t* err) {
  *err = cudaSuccess;
  if (!forward_wide(rows, dm, y_swa != nullptr, sms)) return false;
  for (int x = 0; x < (y_swa ? 2 : 1); ++x) {
    const void* y = x ? y_swa : y_sa;
    const void* w = x ? w_swa : w_sa;
    Maps m;
    if (!make_map(&m.a, y, rows, dm, ld_y, 128) || !make_map(&m.b, w, dm, dm, dm, 256) ||
        !make_map(&m.o0, out, rows, dm, ld_out, 128)) {
      *err = cudaErrorUnknown;
      return true;
    }
    m.i0 = m.a;
    m.i1 = m.o1 = m.o0;
    BwdGateParams p{};
    p.status = status;
    p.m_rows = (int)rows; p.n_cols = dm;
    *err = x ? launch_mode<kFwdAdd, 256>(p, m, dm, sms, st)
             : launch_mode<kFwd, 256>(p, m, dm, sms, st);
    if (*err != cudaSuccess) return true;
  }
  return true;
}

}  // namespace sa

extern "C" size_t sa_gate_projection_backward_ws_bytes(int64_t rows, int32_t dm) {
  if (rows < 1 || dm < 1) return (size_t)-1;
  return (size_t)rows * (size_t)dm * 2u * sizeof(float);    // dz and dout * g, fp32 at most
}

extern "C" sa_status sa_gate_projection_backward(
    int64_t rows, int32_t dm, int32_t dtype, const void* dout, int64_t ld_dout, const void* y_sa,
    const void* y_swa, int64_t ld_y, const void* w_sa, const void* w_swa, void* dy_sa,
    void* dy_swa, int64_t ld_dy, void* dw_sa, void* dw_swa, void* ws, size_t ws_bytes,
    sa_stream_t stream) {
  using namespace sa;
  if (rows < 1 || dm < 1 || ld_y < dm || ld_dout < dm || ld_dy < dm) return SA_ERR_INVALID_ARG;
  if (!dout || !y_sa || !w_sa || !dy_sa || !dw_sa || !ws) return SA_ERR_INVALID_ARG;
  if (y_swa && (!w_swa || !dy_swa || !dw_swa)) return SA_ERR_INVALID_ARG;
  if (dtype != SA_F32 && dtype != SA_BF16) return SA_ERR_INVALID_ARG;
  if (ws_bytes < sa_gate_projection_backward_ws_bytes(rows, dm)) return SA_ERR_WORKSPACE;
  if (rows * (int64_t)dm > (1ll << 40)) return SA_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  const bool tc_off = debug_option(SA_DEBUG_TENSOR_CORES) == 0;
  bool tc = !tc_off && dtype == SA_BF16 && dm % 64 == 0 && ld_y % 8 == 0 && ld_dout % 8 == 0 &&
            ld_dy % 8 == 0 && rows < (1ll << 31) - 256 && aligned16(ws) && aligned16(dout);
  const void* ptrs[] = {y_sa, w_sa, dy_sa, dw_sa, y_swa, w_swa, dy_swa, dw_swa};
  for (const void* q : ptrs) tc = tc && aligned16(q);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return SA_ERR_CUDA;
  int* status = status_ptr();
  if (!status) return SA_ERR_CUDA;

  for (int x = 0; x < (y_swa ? 2 : 1); ++x) {
    const void* y = x ? y_swa : y_sa;
    const void* w = x ? w_swa : w_sa;
    void* dy = x ? dy_swa : dy_sa;
    void* dw = x ? dw_swa : dw_sa;
    if (tc) {
      __nv_bfloat16* dz = (__nv_bfloat16*)ws;
      __nv_bfloat16* dyd = dz + rows * (int64_t)dm;
      float* part = (float*)(dyd + rows * (int64_t)dm);
      // (With a long contraction the narrow tiles' operand stream counts for more.  Both widths at 67
      // sizes, 300 ... 20000 rows x 512 ... 4096: the one taken is the faster at all but four, where they
      // are within 4 %.  The lines between: 8000 x 768 57.7 us wide / 55.6, 12000 x 512 51.1 / 47.0, but
      // 5000 x 1024 61.5 / 63.3, 2500 x 2048 85.0 / 92.8, 1500 x 4096 175 / 179.)
      const bool wide = wide_waves(rows, dm, sms, dm >= 1024 ? 350 : 300);
      const DwPlan dwp = plan_dw(rows, dm, sms);
      CUtensorMap y_k, w_k, dz_k, w_mn, dz_mn, y_mn, dout_k, dyd_k, dy_k, dw_o;
      if (!make_map(&y_k, y, rows, dm, ld_y, 128) ||
          !make_map(&w_k, w, dm, dm, dm, wide ? 256 : 128) ||
          !make_map(&dz_k, dz, rows, dm, dm, 128) || !make_map(&w_mn, w, dm, dm, dm, 64) ||
          !make_map(&dz_mn, dz, rows, dm, dm, 64) || !make_map(&y_mn, y, rows, dm, ld_y, 64) ||
          !make_map(&dout_k, dout, rows, dm, ld_dout, 128) ||
          !make_map(&dyd_k, dyd, rows, dm, dm, 128) || !make_map(&dy_k, dy, rows, dm, ld_dy, 128) ||
          !(dwp.splits > 1 ? make_map_f32(&dw_o, part, dwp.splits, dm, dm)
                           : make_map(&dw_o, dw, dm, dm, dm, 128)))
        return SA_ERR_CUDA;
      BwdGateParams p{};
      p.status = status;
      // z = y w^T; epilogue: dz, dout * g
      p.m_rows = (int)rows; p.n_cols = dm;
      Maps m{y_k, w_k, y_k, dout_k, dz_k, dyd_k};
      if ((wide ? launch_mode<kDz, 256>(p, m, dm, sms, st)
                : launch_mode<kDz, 128>(p, m, dm, sms, st)) != cudaSuccess)
        return SA_ERR_CUDA;
      // dy = dz w + dout * g
      m = Maps{dz_k, w_mn, dyd_k, dyd_k, dy_k, dy_k};
      if ((wide ? launch_mode<kDy, 256>(p, m, dm, sms, st)
                : launch_mode<kDy, 128>(p, m, dm, sms, st)) != cudaSuccess)
        return SA_ERR_CUDA;
      // dw = dz^T y
      p.m_rows = dm;
      p.splits = dwp.splits;
      m = Maps{dz_mn, y_mn, y_mn, y_mn, dw_o, dw_o};
      if ((dwp.tn == 256 ? launch_mode<kDw, 256>(p, m, rows, sms, st)
                         : launch_mode<kDw, 128>(p, m, rows, sms, st)) != cudaSuccess)
        return SA_ERR_CUDA;
      if (dwp.splits > 1) {
        const int64_t eights = (int64_t)dm * dm / 8;
        bump_launches();
        if (launch_dependent(dw_sum_kernel, dim3((unsigned)((eights + 255) / 256)), dim3(256), 0, st,
                             (const float4*)part, dwp.splits, eights, (uint4*)dw) != cudaSuccess)
          return SA_ERR_CUDA;
      }
    } else {
      float* dz = (float*)ws;
      float* dyd = dz + rows * (int64_t)dm;
      const unsigned b1 = (unsigned)((rows * dm + 255) / 256);
      const unsigned b2 = (unsigned)(((int64_t)dm * dm + 255) / 256);
      if (dtype == SA_BF16) {
        typedef __nv_bfloat16 T;
        dz_simt_kernel<T><<<b1, 256, 0, st>>>(rows, dm, (const T*)dout, ld_dout, (const T*)y, ld_y,
                                              (const T*)w, dz, dyd);
        dy_simt_kernel<T><<<b1, 256, 0, st>>>(rows, dm, dz, dyd, (const T*)w, (T*)dy, ld_dy);
        dw_simt_kernel<T><<<b2, 256, 0, st>>>(rows, dm, dz, (const T*)y, ld_y, (T*)dw);
      } else {
        typedef float T;
        dz_simt_kernel<T><<<b1, 256, 0, st>>>(rows, dm, (const T*)dout, ld_dout, (const T*)y, ld_y,
                                              (const T*)w, dz, dyd);
        dy_simt_kernel<T><<<b1, 256, 0, st>>>(rows, dm, dz, dyd, (const T*)w, (T*)dy, ld_dy);
        dw_simt_kernel<T><<<b2, 256, 0, st>>>(rows, dm, dz, (const T*)y, ld_y, (T*)dw);
      }
      bump_launches(3);
      if (cudaGetLastError() != cudaSuccess) return SA_ERR_CUDA;
    }
  }
  return SA_OK;
}

// Permutation generation (Alg. 1 line 1): Philox4x32-10 sort keys, a segmented sort by
// (key, token) with one segment per sequence -- one radix pass on the leading key bits,
// then ranking inside each bucket -- and the inverse written with the permutation.  Sequences
// of up to 16384 tokens are sorted by one launch, each in the shared memory of one thread-block
// cluster; longer ones by four launches through global memory.
#include <cooperative_groups.h>

#include <atomic>

#include "sa_common.cuh"

namespace sa {
namespace {

// Sorting n 64-bit keys that are uniform random bits does not need eight radix passes:
// one pass on the leading bits puts every key into a bucket of about 32 keys, and inside a
// bucket the final place of a key is the number of bucket members that precede it in
// (key, token) order, found by direct counting.  Four launches, no assumption on the bucket
// sizes (an unlucky bucket only costs more comparisons), and the order inside a bucket after
// the scatter does not matter, so the scatter may use atomics and the result is still the
// unique ordering by (key, token).
constexpr int kThreadsPerBlock = 256;
constexpr int kMaxBucketBits = 16;

__host__ __device__ inline int bucket_bits_for(int n) {
  int bits = 0;
  while (bits < kMaxBucketBits && (n >> (bits + 5)) > 0) ++bits;   // about 32 keys per bucket
  return bits;
}

__device__ __forceinline__ void philox_round(uint32_t (&c)[4], uint32_t k0, uint32_t k1) {
  const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
  const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
  const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
  c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
}

// Philox4x32 with 10 rounds (Salmon et al., SC'11); the key follows a Weyl sequence.
__device__ __forceinline__ uint64_t sort_key(uint32_t seed_lo, uint32_t seed_hi, uint32_t layer,
                                             uint32_t b, uint32_t i) {
  uint32_t c[4] = {i, b, layer, 0u};
  uint32_t k0 = seed_lo, k1 = seed_hi;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    philox_round(c, k0, k1);
  }
  return ((uint64_t)c[0] << 32) | c[1];
}

__device__ __forceinline__ uint32_t bucket_of(uint64_t key, int bits) {
  return bits ? (uint32_t)(key >> (64 - bits)) : 0u;
}

// keys[b][i] and the size of every bucket.  counts must be zero on entry.
__global__ void keys_kernel(uint32_t seed_lo, uint32_t seed_hi, uint32_t layer, int n, int bits,
                            uint64_t* __restrict__ keys, uint32_t* __restrict__ counts) {
  const int b = blockIdx.y;
  grid_dependents_launch();
  uint32_t* cb = counts + ((size_t)b << bits);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint64_t key = sort_key(seed_lo, seed_hi, layer, b, i);
    keys[(size_t)b * n + i] = key;
    atomicAdd(&cb[bucket_of(key, bits)], 1u);
  }
}

// Exclusive scan of the bucket sizes of one sequence, in place, and a copy that the
// scatter advances.  One block per sequence.
__global__ void __launch_bounds__(kThreadsPerBlock)
scan_kernel(uint32_t* __restrict__ counts, uint32_t* __restrict__ cursor, int nbuckets) {
  __shared__ uint32_t part[kThreadsPerBlock];
  grid_dependency_wait();
  grid_dependents_launch();
  uint32_t* c = counts + (size_t)blockIdx.x * nbuckets;
  uint32_t* cur = cursor + (size_t)blockIdx.x * nbuckets;
  const int per = (nbuckets + kThreadsPerBlock - 1) / kThreadsPerBlock;
  const int lo = threadIdx.x * per, hi = min(lo + per, nbuckets);
  uint32_t s = 0;
  for (int j = lo; j < hi; ++j) s += c[j];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < kThreadsPerBlock; o <<= 1) {
    const uint32_t add = threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
    __syncthreads();
    part[threadIdx.x] += add;
    __syncthreads();
  }
  uint32_t run = part[threadIdx.x] - s;
  for (int j = lo; j < hi; ++j) {
    const uint32_t v = c[j];
    c[j] = run;
    cur[j] = run;
    run += v;
  }
}

// Every (key, token) into its bucket's range, in arbitrary order inside the range.
__global__ void scatter_kernel(const uint64_t* __restrict__ keys, uint32_t* __restrict__ cursor,
                               uint64_t* __restrict__ bkeys, int32_t* __restrict__ btoks, int n,
                               int bits) {
  const int b = blockIdx.y;
  grid_dependency_wait();
  grid_dependents_launch();
  uint32_t* cur = cursor + ((size_t)b << bits);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint64_t key = keys[(size_t)b * n + i];
    const uint32_t pos = atomicAdd(&cur[bucket_of(key, bits)], 1u);
    bkeys[(size_t)b * n + pos] = key;
    btoks[(size_t)b * n + pos] = i;
  }
}

// Slot of every token: start of its bucket plus the number of bucket members that come
// first in (key, token) order.  Writes perm and its inverse.
__global__ void rank_kernel(const uint64_t* __restrict__ bkeys, const int32_t* __restrict__ btoks,
                            const uint32_t* __restrict__ starts, int32_t* __restrict__ perm,
                            int32_t* __restrict__ inv, int n, int bits) {
  const int b = blockIdx.y;
  grid_dependency_wait();
  grid_dependents_launch();
  const uint64_t* kb = bkeys + (size_t)b * n;
  const int32_t* tb = btoks + (size_t)b * n;
  const uint32_t* st = starts + ((size_t)b << bits);
  const uint32_t nbuckets = 1u << bits;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const uint64_t key = kb[e];
    const int32_t tok = tb[e];
    const uint32_t bk = bucket_of(key, bits);
    const uint32_t lo = st[bk], hi = bk + 1 < nbuckets ? st[bk + 1] : (uint32_t)n;
    uint32_t rank = 0;
    for (uint32_t j = lo; j < hi; ++j) {
      const uint64_t kj = kb[j];
      rank += (kj < key) || (kj == key && tb[j] < tok);
    }
    const int32_t pos = (int32_t)(lo + rank);
    perm[(size_t)b * n + pos] = tok;
    inv[(size_t)b * n + tok] = pos;
  }
}

// ------------------------------------------------- one launch, one cluster per sequence
//
// The keys are uniform bits, so the leading bits of a key name, evenly, the CTA of the cluster
// that ranks it and, inside that CTA, a bucket of about eight keys.  Each CTA draws the keys of
// its share of the tokens (in registers), sends every (key, token) to its owner's shared memory
// (places reserved with one remote atomic per CTA pair), and the owner sorts what arrived into
// buckets and ranks it there.  Bound: latency (launch, two cluster barriers, a handful of block
// barriers).  Back to back, before launches started under one another (one launch against the four and
// a memset): n = 256 2.8 against 12.4 us, n = 4096 x 8 sequences 7.7 against 13.0, n = 8192 10.1 against
// 15.2, n = 16384 14.0 against 16.5 (with eight CTAs of 4096 tokens, n = 32768: 22.0 against 16.1).  Now,
// overlapping: n = 8192 3.3, n = 16384 4.4, and the four launches at n = 32768 18.4.
// An owner has room for cap entries; its expected share is n / C with a standard deviation
// below sqrt(n / C), and cap leaves 10 of those (an eighth of the share, 3 of them at 512 tokens,
// was passed by one call in twelve with 8 sequences of 4096, at 760 us instead of 8).  If a share is larger all the same, every CTA
// ranks its own tokens by comparing with every key of the sequence: slow, and still exact.
constexpr int kClusterThreads = 1024;
constexpr int kShareMax = 2048;                                   // tokens per CTA
constexpr int kPerThread = kShareMax / kClusterThreads + 1;       // entries of an owner, per thread

struct ClusterPlan { int log2_c, bits, cap, threads, smem; };

// CTAs per sequence: one up to 1024 tokens (the cluster steps cost 2 us), then so many that a CTA
// keeps 512 (at most eight, the portable cluster size, with up to 2048 each).  Past 16384 tokens eight SMs per sequence are
// too few and the four launches, which use all of them, are faster again.
__host__ inline ClusterPlan cluster_plan(int n) {
  ClusterPlan p;
  p.log2_c = 0;
  while (n > 1024 && p.log2_c < 3 && ((n - 1) >> p.log2_c) >= 512) ++p.log2_c;
  const int share = (n + (1 << p.log2_c) - 1) >> p.log2_c;
  p.bits = 0;
  while (p.bits < 10 && (share >> (p.bits + 3)) > 0) ++p.bits;    // about 8 keys per bucket
  int sd = 1;
  while (sd * sd < share) ++sd;
  p.cap = p.log2_c ? share + 10 * sd : share;
  p.threads = share >= kClusterThreads ? kClusterThreads : (share + 31) / 32 * 32;
  if (p.threads < 64) p.threads = 64;
  p.cap = (p.cap + 3) / 4 * 4;
  p.smem = p.cap * 12 + 2 * (1 << p.bits) * 4 + 16;
  return p;
}

__global__ void __launch_bounds__(kClusterThreads)
perm_cluster_kernel(uint32_t seed_lo, uint32_t seed_hi, uint32_t layer, int n, int log2_c, int bits,
                    int cap, int32_t* __restrict__ perm, int32_t* __restrict__ inv) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t* keys = reinterpret_cast<uint64_t*>(smem);
  int32_t* toks = reinterpret_cast<int32_t*>(keys + cap);
  uint32_t* start = reinterpret_cast<uint32_t*>(toks + cap);      // bucket sizes, then starts
  uint32_t* cursor = start + (1 << bits);
  __shared__ uint32_t received, sent[8], base[8], all[8], wtot[32];
  const int C = 1 << log2_c, nb = 1 << bits, tid = threadIdx.x, T = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x & (C - 1), b = blockIdx.x >> log2_c;
  const int share = (n + C - 1) >> log2_c, t0 = r * share, t1 = min(n, t0 + share);
  perm += (size_t)b * n;
  inv += (size_t)b * n;
  // The sort touches no memory that another kernel uses until it writes its result, so it runs under
  // the tail of the launch before, and the next launch's preamble under it.
  grid_dependents_launch();
  auto bucket = [&](uint64_t key) {
    return bits ? (uint32_t)((key << log2_c) >> (64 - bits)) : 0u;
  };

  uint64_t key[kPerThread];
  int32_t tok[kPerThread];
  int mine = 0, m = t1 - t0;
  uint32_t goff = 0;
  if (C == 1) {
#pragma unroll
    for (int x = 0; x < kPerThread - 1; ++x) {
      const int i = tid + x * T;
      if (i < n) {
        key[x] = sort_key(seed_lo, seed_hi, layer, b, i);
        tok[x] = i;
        mine = x + 1;
      }
    }
    for (int j = tid; j < nb; j += T) start[j] = 0;
    __syncthreads();
  } else {
    cg::cluster_group cl = cg::this_cluster();
    if (tid == 0) received = 0;
    if (tid < C) sent[tid] = 0;
    __syncthreads();
    uint32_t at[kPerThread - 1];
#pragma unroll
    for (int x = 0; x < kPerThread - 1; ++x) {
      tok[x] = -1;
      if (x * T >= share) continue;       // the same for the whole block
      const int i = t0 + tid + x * T;
      const bool have = i < t1;
      const uint64_t k = sort_key(seed_lo, seed_hi, layer, b, i);
      const int owner = have ? (int)(k >> (64 - log2_c)) : -1;
      at[x] = 0;
      for (int o = 0; o < C; ++o) {       // one shared-memory atomic per warp and owner
        const uint32_t who = __ballot_sync(0xffffffffu, owner == o);
        uint32_t first = 0;
        if (lane == 0 && who) first = atomicAdd(&sent[o], __popc(who));
        first = __shfl_sync(0xffffffffu, first, 0);
        if (owner == o) at[x] = first + __popc(who & ((1u << lane) - 1));
      }
      key[x] = k;
      tok[x] = have ? i : -1;
    }
    cl.sync();                            // every `received` is zero, every `sent` complete
    if (tid < C) base[tid] = atomicAdd(cl.map_shared_rank(&received, tid), sent[tid]);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < kPerThread - 1; ++x) {
      if (tok[x] < 0) continue;
      const int owner = (int)(key[x] >> (64 - log2_c));
      const uint32_t p = base[owner] + at[x];
      if (p < (uint32_t)cap) {
        cl.map_shared_rank(keys, owner)[p] = key[x];
        cl.map_shared_rank(toks, owner)[p] = tok[x];
      }
    }
    for (int j = tid; j < nb; j += T) start[j] = 0;
    cl.sync();
    if (tid < C) all[tid] = *cl.map_shared_rank(&received, tid);
    cl.sync();                            // nobody's counter is read after this
    bool over = false;
    for (int o = 0; o < C; ++o) {
      over |= all[o] > (uint32_t)cap;
      if (o < r) goff += all[o];
    }
    if (over) {                           // the exact slow way, see above
      grid_dependency_wait();
      for (int i = t0 + tid; i < t1; i += T) {
        const uint64_t k = sort_key(seed_lo, seed_hi, layer, b, i);
        int pos = 0;
        for (int j = 0; j < n; ++j) {
          const uint64_t kj = sort_key(seed_lo, seed_hi, layer, b, j);
          pos += kj < k || (kj == k && j < i);
        }
        perm[pos] = i;
        inv[i] = pos;
      }
      return;
    }
    m = (int)all[r];
#pragma unroll
    for (int x = 0; x < kPerThread; ++x) {
      const int e = tid + x * T;
      if (e < m) {
        key[x] = keys[e];
        tok[x] = toks[e];
        mine = x + 1;
      }
    }
    __syncthreads();                      // the lists are in registers: the arrays may be rewritten
  }

  // bucket sizes, their exclusive scan, and every entry into its bucket's range
#pragma unroll
  for (int x = 0; x < kPerThread; ++x)
    if (x < mine) atomicAdd(&start[bucket(key[x])], 1u);
  __syncthreads();
  uint32_t carry = 0;
  for (int j0 = 0; j0 < nb; j0 += T) {    // one round unless the block is small
    const int j = j0 + tid;
    const uint32_t v = j < nb ? start[j] : 0u;
    uint32_t s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += up;
    }
    if (lane == 31) wtot[warp] = s;
    __syncthreads();
    uint32_t before = carry, total = 0;
    for (int x = 0; x < T / 32; ++x) {
      if (x < warp) before += wtot[x];
      total += wtot[x];
    }
    carry += total;
    if (j < nb) start[j] = cursor[j] = before + s - v;
    __syncthreads();
  }
#pragma unroll
  for (int x = 0; x < kPerThread; ++x)
    if (x < mine) {
      const uint32_t p = atomicAdd(&cursor[bucket(key[x])], 1u);
      keys[p] = key[x];
      toks[p] = tok[x];
    }
  __syncthreads();
  grid_dependency_wait();
  // rank inside the bucket; cursor[] now holds the bucket ends
#pragma unroll 1
  for (int e = tid; e < m; e += T) {
    const uint64_t k = keys[e];
    const int32_t t = toks[e];
    const uint32_t bk = bucket(k), lo = start[bk], hi = cursor[bk];
    uint32_t rank = 0;
    for (uint32_t j = lo; j < hi; ++j) {
      const uint64_t kj = keys[j];
      rank += (kj < k) || (kj == k && toks[j] < t);
    }
    const int32_t pos = (int32_t)(goff + lo + rank);
    perm[pos] = t;
    inv[t] = pos;
  }
}

__global__ void validate_perm_kernel(const int32_t* __restrict__ perm,
                                     const int32_t* __restrict__ inv, int n, int* status) {
  const int b = blockIdx.y;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const int32_t t = perm[(size_t)b * n + p];
    bool ok = t >= 0 && t < n;
    if (ok) ok = inv[(size_t)b * n + t] == p;
    if (!ok) atomicCAS(status, SA_OK, SA_ERR_BAD_PERM);
  }
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Built-in scratch of sa_make_perm_static: part of the library image, so every GPU that
// loads the library holds these bytes until the process exits.  In host code this name is
// only a host-side stand-in for the symbol, never a device address: the launcher below
// resolves the real address with cudaGetSymbolAddress and hands that to the kernels.
static __device__ __align__(256) unsigned char g_static_scratch[SA_STATIC_SCRATCH_BYTES];

// Device address of g_static_scratch on the current device, resolved once per device.
unsigned char* static_scratch_ptr() {
  static std::atomic<unsigned char*> ptrs[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  unsigned char* q = ptrs[dev].load(std::memory_order_acquire);
  if (!q) {
    if (cudaGetSymbolAddress((void**)&q, g_static_scratch) != cudaSuccess) return nullptr;
    ptrs[dev].store(q, std::memory_order_release);
  }
  return q;
}

}  // namespace

size_t make_perm_ws_bytes(int B, int n) {
  const size_t bn = (size_t)B * n;
  const size_t nb = (size_t)B << bucket_bits_for(n);
  return 2 * align_up(bn * 8, 256) + align_up(bn * 4, 256) + 2 * align_up(nb * 4, 256);
}

cudaError_t launch_make_perm(uint64_t seed, uint32_t layer, int B, int n, int32_t* perm,
                             int32_t* inv, void* ws, cudaStream_t st) {
  if (n <= 8 * kShareMax) {
    const ClusterPlan c = cluster_plan(n);
    if (c.smem > 48 * 1024) {
      const cudaError_t e = cudaFuncSetAttribute(perm_cluster_kernel,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, c.smem);
      if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)B << c.log2_c);
    cfg.blockDim = dim3(c.threads);
    cfg.dynamicSmemBytes = c.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << c.log2_c;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, perm_cluster_kernel, (uint32_t)seed, (uint32_t)(seed >> 32), layer,
                           n, c.log2_c, c.bits, c.cap, perm, inv);
    if (e != cudaSuccess) return reported(e);
    bump_launches();
    return cudaGetLastError();
  }
  const size_t bn = (size_t)B * n;
  const int bits = bucket_bits_for(n);
  const size_t nb = (size_t)B << bits;
  char* p = (char*)ws;
  uint64_t* keys = (uint64_t*)p; p += align_up(bn * 8, 256);
  uint64_t* bkeys = (uint64_t*)p; p += align_up(bn * 8, 256);
  int32_t* btoks = (int32_t*)p; p += align_up(bn * 4, 256);
  uint32_t* counts = (uint32_t*)p; p += align_up(nb * 4, 256);
  uint32_t* cursor = (uint32_t*)p;

  cudaError_t e = cudaMemsetAsync(counts, 0, nb * 4, st);   // bucket sizes start at zero
  if (e != cudaSuccess) return e;
  const int kb = min((n + kThreadsPerBlock - 1) / kThreadsPerBlock, 1024);
  keys_kernel<<<dim3(kb, B), kThreadsPerBlock, 0, st>>>((uint32_t)seed, (uint32_t)(seed >> 32),
                                                        layer, n, bits, keys, counts);
  e = launch_dependent(scan_kernel, dim3(B), dim3(kThreadsPerBlock), 0, st, counts, cursor, 1 << bits);
  if (e == cudaSuccess)
    e = launch_dependent(scatter_kernel, dim3(kb, B), dim3(kThreadsPerBlock), 0, st, keys, cursor, bkeys,
                         btoks, n, bits);
  if (e == cudaSuccess)
    e = launch_dependent(rank_kernel, dim3(kb, B), dim3(kThreadsPerBlock), 0, st, bkeys, btoks, counts,
                         perm, inv, n, bits);
  if (e != cudaSuccess) return e;
  bump_launches(4);
  return cudaGetLastError();
}

cudaError_t launch_validate_perm(const int32_t* perm, const int32_t* inv, int B, int n,
                                 cudaStream_t st) {
  int* status = status_ptr();
  if (!status) return cudaErrorUnknown;
  const int kb = min((n + 255) / 256, 1024);
  validate_perm_kernel<<<dim3(kb, B), 256, 0, st>>>(perm, inv, n, status);
  bump_launches();
  return cudaGetLastError();
}

}  // namespace sa

extern "C" sa_status sa_make_perm_static(uint64_t seed, uint32_t layer, int32_t B, int32_t n,
                                         int32_t* perm, int32_t* inv, sa_stream_t stream) {
  using namespace sa;
  if (B < 1 || n < 1) return SA_ERR_INVALID_ARG;
  if (B > 32767 || n > (1 << 30)) return SA_ERR_UNSUPPORTED;
  if (!perm || !inv || ((uintptr_t)perm & 15u) || ((uintptr_t)inv & 15u)) return SA_ERR_INVALID_ARG;
  if (make_perm_ws_bytes(B, n) > (size_t)SA_STATIC_SCRATCH_BYTES) return SA_ERR_TOO_LARGE;
  unsigned char* scratch = static_scratch_ptr();
  if (!scratch) return SA_ERR_CUDA;
  // Only the bucket counters have to start at zero, and the launcher clears them on the
  // stream itself; the key and token arrays are written in full before anything reads
  // them, so whatever the previous call left behind is never seen.
  return launch_make_perm(seed, layer, B, n, perm, inv, scratch, (cudaStream_t)stream) ==
                 cudaSuccess ? SA_OK : SA_ERR_CUDA;
}

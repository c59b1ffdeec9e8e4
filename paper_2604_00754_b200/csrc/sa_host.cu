// Gated SA + SWA forward for tensors that live in HOST memory (Alg. 2 / Eq. 5 end to end:
// fresh permutation, both branches, gates), as one C-ABI call.
//
// The attention of one KV head (and of the query heads that share it) reads nothing of the
// other heads, so the heads travel through the GPU in pieces: while one piece is being
// computed, the next one is on its way in over PCIe and the previous result is on its way out.
// Three streams (copy in, compute, copy out) and one event pair per piece do the ordering;
// every piece is computed by the same entry points a device-resident caller uses, on strided
// views of whole-size device buffers carved out of the caller's workspace.  The permutation is
// drawn once per call and shared by all pieces.
#include <initializer_list>
#include <mutex>

#include "sa_common.cuh"

namespace sa {
namespace {

constexpr int kMaxPieces = 256;
constexpr int kPlanSms = 148;       // SMs of the GPU planned for: a plan is the same without one at hand

struct Piece { int ka, kb, qa, qb, with_kv, b0, b1; };

// KV heads in at most n_groups contiguous ranges.  The first and the last range, when they hold
// one KV head, are cut further into q_parts ranges of query heads if those divide evenly (only
// the first part carries K/V): the copy in of the first piece and the kernels and copy out of
// the last one are what cannot overlap, so those pieces are small; the pieces in between are
// large, because every piece costs launches and events.
int plan(int Hq, int Hkv, int n_groups, int q_parts, Piece* out, int max_out) {
  if (Hq < 1 || Hkv < 1 || Hq % Hkv != 0 || !out) return -1;
  const int G = Hq / Hkv;
  n_groups = n_groups < 1 ? 1 : (n_groups > Hkv ? Hkv : n_groups);
  int cnt = 0;
  for (int i = 0; i < n_groups; ++i) {
    const int a = (int)((int64_t)i * Hkv / n_groups), b = (int)((int64_t)(i + 1) * Hkv / n_groups);
    if (b <= a) continue;
    const bool edge = i == 0 || i == n_groups - 1;
    if (edge && b - a == 1 && q_parts > 1 && G % q_parts == 0) {
      const int step = G / q_parts;
      for (int j = 0; j < q_parts; ++j) {
        if (cnt >= max_out) return -1;
        out[cnt++] = Piece{a, b, a * G + j * step, a * G + (j + 1) * step, j == 0, 0, 0};
      }
    } else {
      if (cnt >= max_out) return -1;
      out[cnt++] = Piece{a, b, a * G, b * G, 1, 0, 0};
    }
  }
  return cnt;
}

// The same for B sequences: the sequences are divided first, into at most n_groups or `most` ranges (whole
// sequences are one block of memory, so a piece is one copy per tensor where a range of heads is one
// per tensor and sequence), then the heads of each range until there are about n_groups pieces.
// Only the last range's ends are cut by query heads.  With heads alone, 8 sequences of one head
// (n = 3248, d = 64) were a single piece whose copies and kernels followed one another (580 -> 410 us); 16 x 12 heads of
// 64, n = 700: 2880 -> 1280 us, 2 x 32/8 heads of 128, n = 3727: 2680 -> 2150.
int plan_batch(int most, int B, int Hq, int Hkv, int n_groups, int q_parts, Piece* out, int max_out) {
  n_groups = n_groups < 1 ? 1 : n_groups;
  const int parts = most < n_groups ? most : n_groups;
  int cnt = 0;
  for (int i = 0; i < parts; ++i) {
    const int got = plan(Hq, Hkv, n_groups / parts, i == parts - 1 ? q_parts : 1, out + cnt,
                         max_out - cnt);
    if (got < 0) return -1;
    for (int j = 0; j < got; ++j) {
      out[cnt + j].b0 = (int)((int64_t)i * B / parts);
      out[cnt + j].b1 = (int)((int64_t)(i + 1) * B / parts);
    }
    cnt += got;
  }
  return cnt;
}

// Input bytes on the device (q, k, v, each rounded up to 256 bytes).
size_t align256(size_t x) { return (x + 255) / 256 * 256; }
size_t tensor_bytes(const sa_problem* p, int heads) {
  return align256((size_t)p->B * heads * p->n * p->d * (p->dtype == SA_BF16 ? 2 : 4));
}

// The pieces of one call; -1 for what plan() refuses for the heads alone.  Any number of groups that
// it takes for the heads is taken for a batch too: below 1 means 1, and more pieces than there are
// events are not made.
int plan_call(const sa_problem* p, int n_groups, int q_parts, Piece* out) {
  if (plan(p->Hq, p->Hkv, n_groups, q_parts, out, kMaxPieces) < 1) return -1;
  n_groups = n_groups < 1 ? 1 : (n_groups > kMaxPieces ? kMaxPieces : n_groups);
  // a range's permutation may have to move to an aligned place in the scratch, which is as large as Q:
  // one range if that is too small (rows of a few bytes)
  const size_t per_seq = 2 * align256((size_t)p->n * sizeof(int32_t));
  const int ranged = per_seq * p->B <= tensor_bytes(p, p->Hq) ? p->B : 1;
  // a piece costs the host about 40 us of calls, as long as 2 MB take over PCIe: none smaller
  const size_t most = (tensor_bytes(p, p->Hq) + 2 * tensor_bytes(p, p->Hkv)) >> 21;
  if ((size_t)n_groups > most) {
    n_groups = most ? (int)most : 1;
    q_parts = 1;
  }
  // half of a group's query heads that leave SMs idle (an item is two tiles of 128 rows) take the
  // kernels as long as the whole group: 32/8 heads, n = 8192: 2440 -> 2370 us uncut
  if (q_parts > 1 &&
      (int64_t)(p->Hq / p->Hkv / q_parts) * ((p->n + 127) / 128) < 2 * kPlanSms)
    q_parts = 1;
  const int cnt = plan_batch(ranged, p->B, p->Hq, p->Hkv, n_groups, q_parts, out, kMaxPieces);
  return cnt > 0 ? cnt : plan_batch(ranged, p->B, p->Hq, p->Hkv, n_groups, 1, out, kMaxPieces);
}

// Streams and events of the pipeline, created at the first call on a device and kept.
struct Pipe {
  bool ready = false;
  cudaStream_t s_in = nullptr, s_run = nullptr, s_out = nullptr;
  cudaEvent_t ev_start = nullptr, ev_end = nullptr;
  cudaEvent_t ev_in[kMaxPieces], ev_done[kMaxPieces];
};
Pipe g_pipes[64];
std::mutex g_pipe_mutex;

Pipe* pipe_for_current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(g_pipe_mutex);
  Pipe& p = g_pipes[dev];
  if (p.ready) return &p;
  bool ok = cudaStreamCreateWithFlags(&p.s_in, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&p.s_run, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&p.s_out, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&p.ev_start, cudaEventDisableTiming) == cudaSuccess &&
            cudaEventCreateWithFlags(&p.ev_end, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; ok && i < kMaxPieces; ++i)
    ok = cudaEventCreateWithFlags(&p.ev_in[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&p.ev_done[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) return nullptr;
  p.ready = true;
  return &p;
}

struct Carve {
  size_t q, k, v, y, scratch, gate, perm, inv, perm_ws, total;
  size_t lists, list_bytes, with_lists;   // key lists of the SA branch; bytes with room for them
};

bool carve(const sa_problem* p, Carve* c) {
  if (!p || p->B < 1 || p->Hq < 1 || p->Hkv < 1 || p->n < 1 || p->d < 1) return false;
  const size_t qb = tensor_bytes(p, p->Hq), kb = tensor_bytes(p, p->Hkv);
  size_t o = 0;
  c->q = o; o += qb;
  c->k = o; o += kb;
  c->v = o; o += kb;
  c->y = o; o += qb;
  c->scratch = o; o += qb;
  // the logits as they come ([2, Hq]), then one contiguous [2, heads] block per piece
  c->gate = o; o += 2 * align256((size_t)2 * p->Hq * sizeof(float));
  c->perm = o; o += align256((size_t)p->B * p->n * sizeof(int32_t));
  c->inv = o; o += align256((size_t)p->B * p->n * sizeof(int32_t));
  c->perm_ws = o; o += align256(make_perm_ws_bytes(p->B, p->n));
  c->total = o;
  // The key lists of all sequences go behind the copies of index lists that some ranges need in the scratch
  // (at most one of each per sequence), or behind everything where that is too small.
  sa_problem dp = *p;
  sa_problem_set_contiguous(&dp);
  const size_t lb = sa_workspace_bytes(&dp, SA_OP_KEY_LISTS);
  c->list_bytes = lb == (size_t)-1 ? 0 : lb;
  const size_t copies = 2 * (size_t)p->B * align256((size_t)p->n * sizeof(int32_t));
  const bool fits = copies + c->list_bytes <= qb;
  c->lists = fits ? c->scratch + copies : o;
  c->with_lists = fits ? o : o + c->list_bytes;
  return true;
}

}  // namespace
}  // namespace sa

using namespace sa;

extern "C" {

int32_t sa_host_forward_plan(int32_t Hq, int32_t Hkv, int32_t n_groups, int32_t q_parts,
                             int32_t* pieces, int32_t max_pieces) {
  Piece tmp[kMaxPieces];
  const int cnt = plan(Hq, Hkv, n_groups, q_parts, tmp, kMaxPieces);
  if (cnt < 0 || cnt > max_pieces || !pieces) return -1;
  for (int i = 0; i < cnt; ++i) {
    pieces[5 * i + 0] = tmp[i].ka; pieces[5 * i + 1] = tmp[i].kb;
    pieces[5 * i + 2] = tmp[i].qa; pieces[5 * i + 3] = tmp[i].qb;
    pieces[5 * i + 4] = tmp[i].with_kv;
  }
  return cnt;
}

int32_t sa_host_forward_pieces(const sa_problem* p, int32_t n_groups, int32_t q_parts,
                               int32_t* pieces, int32_t max_pieces) {
  Carve c;
  Piece tmp[kMaxPieces];
  if (!pieces || !carve(p, &c)) return -1;
  const int cnt = plan_call(p, n_groups, q_parts, tmp);
  if (cnt < 0 || cnt > max_pieces) return -1;
  for (int i = 0; i < cnt; ++i) {
    const Piece& g = tmp[i];
    const int row[7] = {g.ka, g.kb, g.qa, g.qb, g.with_kv, g.b0, g.b1};
    for (int x = 0; x < 7; ++x) pieces[7 * i + x] = row[x];
  }
  return cnt;
}

size_t sa_host_forward_ws_bytes(const sa_problem* p) {
  Carve c;
  return carve(p, &c) ? c.with_lists : (size_t)-1;
}

sa_status sa_swa_gated_forward_host(const sa_problem* p, const void* q, const void* k,
                                    const void* v, const float* gate_logits, void* y,
                                    uint64_t seed, uint32_t layer, int32_t n_groups,
                                    int32_t q_parts, void* ws, size_t ws_bytes,
                                    sa_stream_t stream) {
  if (!p || !q || !k || !v || !gate_logits || !y || !ws) return SA_ERR_INVALID_ARG;
  if (((uintptr_t)ws & 255u) != 0) return SA_ERR_INVALID_ARG;
  Carve c;
  if (!carve(p, &c)) return SA_ERR_INVALID_ARG;
  if (ws_bytes < c.total) return SA_ERR_WORKSPACE;
  Piece pieces[kMaxPieces];
  const int cnt = plan_call(p, n_groups, q_parts, pieces);
  if (cnt < 1) return SA_ERR_INVALID_ARG;
  // device-side problem: contiguous [B,H,n,d] buffers, whatever the strides field says
  sa_problem dp = *p;
  sa_problem_set_contiguous(&dp);
  dp.flags &= ~(uint32_t)SA_SAVE_FOR_BWD;
  // validate the shape once through the ordinary sizing call
  if (sa_workspace_bytes(&dp, SA_OP_GATED_FORWARD) == (size_t)-1) return SA_ERR_INVALID_ARG;
  Pipe* pipe = pipe_for_current_device();
  if (!pipe) return SA_ERR_CUDA;

  char* base = (char*)ws;
  const size_t es = p->dtype == SA_BF16 ? 2 : 4;
  const size_t head_bytes = (size_t)p->n * p->d * es;
  char *dq = base + c.q, *dk = base + c.k, *dv = base + c.v, *dyv = base + c.y;
  float* dgate_all = (float*)(base + c.gate);
  float* dgate = (float*)(base + c.gate + align256((size_t)2 * p->Hq * sizeof(float)));
  int32_t* dperm = (int32_t*)(base + c.perm);
  int32_t* dinv = (int32_t*)(base + c.inv);
  cudaStream_t cur = (cudaStream_t)stream;
  bool ok = true;
  auto chk = [&](cudaError_t e) { ok = ok && e == cudaSuccess; };

  // everything below is ordered after what the caller's stream has queued so far
  chk(cudaEventRecord(pipe->ev_start, cur));
  chk(cudaStreamWaitEvent(pipe->s_in, pipe->ev_start, 0));
  chk(cudaStreamWaitEvent(pipe->s_run, pipe->ev_start, 0));
  chk(cudaStreamWaitEvent(pipe->s_out, pipe->ev_start, 0));

  // copy in: all logits in one small copy (a copy of a few bytes holds the copy engine as long
  // as one of a few hundred kilobytes, and two per piece stood between the large ones), then
  // the heads of each piece; the [2, heads] block of a piece is cut out on the compute stream
  chk(cudaMemcpyAsync(dgate_all, gate_logits, (size_t)2 * p->Hq * sizeof(float),
                      cudaMemcpyHostToDevice, pipe->s_in));
  // heads [a, b) of a piece's sequences, out of H heads per sequence: one block where the piece has
  // all heads, else one per sequence
  auto copy_heads = [&](const Piece& g, int H, int a, int e, char* dst, const char* src,
                        cudaMemcpyKind kind, cudaStream_t st) {
    const int step = e - a == H ? g.b1 - g.b0 : 1;
    for (int b = g.b0; b < g.b1; b += step) {
      const size_t off = ((size_t)b * H + a) * head_bytes;
      chk(cudaMemcpyAsync(dst + off, src + off, (size_t)step * (e - a) * head_bytes, kind, st));
    }
  };
  for (int i = 0; i < cnt && ok; ++i) {
    const Piece& g = pieces[i];
    if (g.with_kv) {
      copy_heads(g, p->Hkv, g.ka, g.kb, dk, (const char*)k, cudaMemcpyHostToDevice, pipe->s_in);
      copy_heads(g, p->Hkv, g.ka, g.kb, dv, (const char*)v, cudaMemcpyHostToDevice, pipe->s_in);
    }
    copy_heads(g, p->Hq, g.qa, g.qb, dq, (const char*)q, cudaMemcpyHostToDevice, pipe->s_in);
    chk(cudaEventRecord(pipe->ev_in[i], pipe->s_in));
  }

  // compute: fresh permutation, then piece by piece as the inputs arrive
  sa_status st = SA_OK;
  if (ok)
    st = sa_make_perm(seed, layer, p->B, p->n, dperm, dinv, base + c.perm_ws,
                      make_perm_ws_bytes(p->B, p->n), (sa_stream_t)pipe->s_run);
  // the SA branch's key lists are made once per range of sequences, by its first piece
  void* lists = c.list_bytes && ws_bytes >= c.with_lists ? base + c.lists : nullptr;
  const int32_t *rperm = dperm, *rinv = dinv;     // of the range at hand
  bool lists_ready = false;
  int range_at = 0;
  size_t spare = c.scratch;
  for (int i = 0; i < cnt && ok && st == SA_OK; ++i) {
    const Piece& g = pieces[i];
    if (g.b0 != range_at) {
      // the kernels' entry points take index lists that start on 16 bytes
      const size_t at = (size_t)g.b0 * p->n, len = (size_t)(g.b1 - g.b0) * p->n * sizeof(int32_t);
      range_at = g.b0;
      lists_ready = false;
      rperm = dperm + at;
      rinv = dinv + at;
      if (at % 4 != 0) {
        for (const int32_t** list : {&rperm, &rinv}) {
          chk(cudaMemcpyAsync(base + spare, *list, len, cudaMemcpyDeviceToDevice, pipe->s_run));
          *list = (const int32_t*)(base + spare);
          spare += align256(len);
        }
      }
    }
    chk(cudaStreamWaitEvent(pipe->s_run, pipe->ev_in[i], 0));
    const int hq = g.qb - g.qa;
    float* gates = dgate_all;
    if (hq < p->Hq) {                       // each range of query heads has its own place
      gates = dgate + 2 * g.qa;
      chk(cudaMemcpy2DAsync(gates, (size_t)hq * sizeof(float), dgate_all + g.qa,
                            (size_t)p->Hq * sizeof(float), (size_t)hq * sizeof(float), 2,
                            cudaMemcpyDeviceToDevice, pipe->s_run));
    }
    sa_problem gp = dp;                     // a view of the whole-size buffers: same strides
    gp.B = g.b1 - g.b0;
    gp.Hq = hq;
    gp.Hkv = g.kb - g.ka;
    const size_t qoff = ((size_t)g.b0 * p->Hq + g.qa) * head_bytes;
    const size_t koff = ((size_t)g.b0 * p->Hkv + g.ka) * head_bytes;
    st = gated_forward(&gp, dq + qoff, dk + koff, dv + koff, rperm, rinv, gates, dyv + qoff, nullptr, nullptr,
                       nullptr, nullptr, lists, lists_ready, pipe->s_run);
    lists_ready = lists != nullptr;
    chk(cudaEventRecord(pipe->ev_done[i], pipe->s_run));
  }

  // copy out
  for (int i = 0; i < cnt && ok && st == SA_OK; ++i) {
    const Piece& g = pieces[i];
    chk(cudaStreamWaitEvent(pipe->s_out, pipe->ev_done[i], 0));
    copy_heads(g, p->Hq, g.qa, g.qb, (char*)y, dyv, cudaMemcpyDeviceToHost, pipe->s_out);
  }
  // the caller's stream resumes when all three streams are done (also after an error, so
  // that nothing of this call is still in flight when the caller goes on)
  cudaEventRecord(pipe->ev_end, pipe->s_in);
  cudaStreamWaitEvent(cur, pipe->ev_end, 0);
  cudaEventRecord(pipe->ev_end, pipe->s_run);
  cudaStreamWaitEvent(cur, pipe->ev_end, 0);
  cudaEventRecord(pipe->ev_end, pipe->s_out);
  cudaStreamWaitEvent(cur, pipe->ev_end, 0);
  if (st != SA_OK) return st;
  return ok ? SA_OK : SA_ERR_CUDA;
}

}  // extern "C"

// Host side of the library: descriptor validation, position IDs and slots (integer rules of
// Eq. 4 and Section 3.3), the split-K work list, plan life cycle and the C entry points.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <functional>
#include <mutex>
#include <new>
#include <vector>

#include "aspd_internal.cuh"

using namespace aspd;

namespace {

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---- device blocks of destroyed plans are kept for the next plan --------------------------------
// A decode loop makes a new plan every step; cudaMalloc and cudaFree (which waits for the whole
// device) would cost more than the step's host work.  aspd_plan_destroy therefore parks the plan's
// block together with an event recorded on every stream the plan was used on, and
// aspd_plan_create takes a parked block of fitting size and makes its stream wait for those events
// before the new tables are uploaded -- no host synchronisation on either side.  With the block goes
// the page-locked host buffer the tables are assembled in (a copy from pageable memory would make
// the host wait for everything queued before it on the stream).
// upload_done: recorded right after the plan's table copy; the host may write the buffer again only
// once it has completed, so a block whose copy is still queued is passed over (a fresh one is
// allocated instead and the pool settles at the depth the loop needs).
// The events live as long as the block: recording one again costs half of creating and destroying one.
std::mutex g_blocks_mu;
std::vector<PlanBlock> g_blocks;
constexpr size_t kParkedMax = 8;                       // blocks kept per process
constexpr size_t kParkedMaxBytes = 2048ull << 20;     // all parked blocks together

bool block_free(PlanBlock& b) {
  for (cudaEvent_t e : b.events) cudaEventDestroy(e);
  if (b.upload_done) cudaEventDestroy(b.upload_done);
  const bool ok = b.ptr == nullptr || cudaFree(b.ptr) == cudaSuccess;    // waits for the device: the host buffer's last copy is done after it
  if (b.host) cudaFreeHost(b.host);
  b = PlanBlock();
  return ok;
}

// Sizes are rounded up (to a quarter of their power of two), so that the plans of steps that differ a little
// share one size of block.
size_t rounded_size(size_t bytes, size_t least) {
  size_t p2 = least;
  while (2 * p2 <= bytes) p2 *= 2;
  return align_up(std::max(bytes, least), std::max(least, p2 / 4));
}

// Into the park, as the latest block or as the one parked longest ago.  It keeps the blocks of the latest plans: the ones
// parked longest ago make room.  (A park that kept the earliest ones -- a batch whose size has changed since never
// fits them -- turned every later plan into cudaMalloc + cudaFree, i.e. a device synchronisation per step: a
// serving mix step of 28 layers took 2.2 ms instead of 1.5 once eight other sizes had been planned.)
void block_park(const PlanBlock& b, bool latest) {
  std::vector<PlanBlock> evicted;
  {
    std::lock_guard<std::mutex> lock(g_blocks_mu);
    g_blocks.insert(latest ? g_blocks.end() : g_blocks.begin(), b);
    size_t parked = 0;
    for (const PlanBlock& x : g_blocks) parked += x.bytes;
    while (g_blocks.size() > kParkedMax || parked > kParkedMaxBytes) {
      parked -= g_blocks.front().bytes;
      evicted.push_back(g_blocks.front());
      g_blocks.erase(g_blocks.begin());
    }
  }
  for (PlanBlock& x : evicted) block_free(x);
}

// (The lock is held for the list alone: what waits for the GPU, allocates or frees does so with the block taken out of
// it, so that plans of other threads, streams and devices go on.)
int block_acquire(size_t bytes, size_t host_need, cudaStream_t s, PlanBlock* out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ASPD_ERR_CUDA;
  const size_t least = bytes;
  bytes = rounded_size(bytes, 4u << 20); host_need = rounded_size(host_need, 64u << 10);
  if (bytes > kParkedMaxBytes) bytes = least;      // never parked, so there is nobody to share a size with
  PlanBlock b;
  int fitting = 0;
  bool ready = false;                              // b's copy is through
  {
    std::lock_guard<std::mutex> lock(g_blocks_mu);
    int best = -1, oldest = -1;
    for (int i = 0; i < (int)g_blocks.size(); ++i) {
      if (g_blocks[i].device != dev || g_blocks[i].bytes < bytes || g_blocks[i].bytes > 4 * bytes) continue;
      ++fitting;
      if (oldest < 0) oldest = i;
      if ((best < 0 || g_blocks[i].bytes < g_blocks[best].bytes) && cudaEventQuery(g_blocks[i].upload_done) == cudaSuccess) best = i;
    }
    ready = best >= 0;
    if (best < 0) best = oldest;
    if (best >= 0) {
      std::swap(b, g_blocks[best]);
      g_blocks.erase(g_blocks.begin() + best);
    }
  }
  // Every fitting block still has its copy queued.  A new block (device and page-locked memory) takes the host the
  // better part of a millisecond, so a copy that is about to finish is waited for first; and with a couple of
  // blocks parked the host is simply ahead of the GPU and waits for the oldest one instead of allocating more.
  if (!ready && fitting == 1) {
    const auto until = std::chrono::steady_clock::now() + std::chrono::microseconds(300);
    do {
      ready = cudaEventQuery(b.upload_done) == cudaSuccess;
    } while (!ready && std::chrono::steady_clock::now() < until);
  }
  if (!ready && fitting >= 2) ready = cudaEventSynchronize(b.upload_done) == cudaSuccess;
  if (ready) {
    int rc = ASPD_OK;
    for (int i = 0; i < b.n_wait; ++i)
      if (cudaStreamWaitEvent(s, b.events[i], 0) != cudaSuccess) rc = ASPD_ERR_CUDA;
    b.n_wait = 0;
    if (rc == ASPD_OK && b.host_bytes < host_need) {             // too small for the new tables (its last copy has completed)
      cudaFreeHost(b.host);
      b.host = nullptr; b.host_bytes = 0;
      if (cudaMallocHost(&b.host, host_need) != cudaSuccess) { b.host = nullptr; rc = ASPD_ERR_NOMEM; }
      else b.host_bytes = host_need;
    }
    if (rc) { block_free(b); return rc; }
    *out = b;
    return ASPD_OK;
  }
  if (fitting > 0) block_park(b, false);
  b = PlanBlock();
  b.device = dev; b.bytes = bytes; b.host_bytes = host_need;
  if (cudaMalloc(&b.ptr, bytes) != cudaSuccess) {
    b.ptr = nullptr;
    cudaGetLastError();                            // (the next launch's check would find it)
    b.bytes = least;                               // what was added for the sake of other plans may be what does not fit
    if (cudaMalloc(&b.ptr, least) != cudaSuccess) { b.ptr = nullptr; return ASPD_ERR_NOMEM; }
  }
  if (cudaMallocHost(&b.host, host_need) != cudaSuccess) { b.host = nullptr; block_free(b); return ASPD_ERR_NOMEM; }
  if (cudaEventCreateWithFlags(&b.upload_done, cudaEventDisableTiming) != cudaSuccess) { b.upload_done = nullptr; block_free(b); return ASPD_ERR_CUDA; }
  *out = b;
  return ASPD_OK;
}

int block_release(PlanBlock& b, const std::vector<cudaStream_t>& streams) {
  int dev = 0;
  bool park = cudaGetDevice(&dev) == cudaSuccess && dev == b.device && b.bytes <= kParkedMaxBytes;   // not from another device's context
  b.n_wait = 0;
  for (size_t i = 0; park && i < streams.size(); ++i) {
    if (i == b.events.size()) {
      cudaEvent_t e;
      if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) { park = false; break; }
      b.events.push_back(e);
    }
    if (cudaEventRecord(b.events[i], streams[i]) != cudaSuccess) park = false;   // e.g. the stream is gone
    else b.n_wait = (int)i + 1;
  }
  if (!park) return block_free(b) ? ASPD_OK : ASPD_ERR_CUDA;
  block_park(b, true);
  return ASPD_OK;
}

int block_cache_clear() {
  std::vector<PlanBlock> all;
  {
    std::lock_guard<std::mutex> lock(g_blocks_mu);
    all.swap(g_blocks);
  }
  int rc = ASPD_OK;
  for (PlanBlock& b : all)
    if (!block_free(b)) rc = ASPD_ERR_CUDA;
  return rc;
}

// every stream a plan's work was enqueued on (a handful at most): what its block must wait for when reused
inline void note_stream(aspd_plan* p, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (std::find(p->streams.begin(), p->streams.end(), s) == p->streams.end()) p->streams.push_back(s);
}

int check_shape(const aspd_shape_t* s) {
  if (!s) return ASPD_ERR_INVALID_ARG;
  if (s->n_q_heads <= 0 || s->n_kv_heads <= 0 || s->n_q_heads % s->n_kv_heads) return ASPD_ERR_INVALID_ARG;
  if (s->head_dim != 64 && s->head_dim != 128) return ASPD_ERR_UNSUPPORTED;
  if (s->dtype != ASPD_DTYPE_F32 && s->dtype != ASPD_DTYPE_BF16) return ASPD_ERR_UNSUPPORTED;
  if (s->page_size != 8 && s->page_size != 16 && s->page_size != 32) return ASPD_ERR_UNSUPPORTED;
  if (s->n_q_heads / s->n_kv_heads > kMaxRowsPerItem) return ASPD_ERR_UNSUPPORTED;
  if (!(s->rope_theta > 0.f) || !(s->sm_scale > 0.f)) return ASPD_ERR_INVALID_ARG;
  return ASPD_OK;
}

// Structural checks that need no page table: counts, q_len <= kv_len, tail in serial mode.
int check_counts(const aspd_request_t* req, const aspd_branch_t* br, int n_req, int mode) {
  if (n_req < 0 || (n_req > 0 && !req)) return ASPD_ERR_INVALID_ARG;
  if (mode != ASPD_MODE_BRANCH && mode != ASPD_MODE_SERIAL) return ASPD_ERR_INVALID_ARG;
  for (int r = 0; r < n_req; ++r) {
    const aspd_request_t& q = req[r];
    if (q.prefix_len < 0 || q.n_branches < 0 || q.branch_begin < 0 || q.tail_len < 0 || q.tail_off < 0)
      return ASPD_ERR_BAD_DESCRIPTOR;
    if (q.n_branches > 0 && !br) return ASPD_ERR_INVALID_ARG;
    for (int b = 0; b < q.n_branches; ++b) {
      const aspd_branch_t& x = br[q.branch_begin + b];
      if (x.kv_off < 0 || x.kv_len < 0 || x.q_len < ASPD_Q_SHARED || x.q_len > x.kv_len || x.pos_start < ASPD_POS_AUTO)
        return ASPD_ERR_BAD_DESCRIPTOR;
    }
    if (mode == ASPD_MODE_SERIAL && q.tail_len < 1) return ASPD_ERR_BAD_DESCRIPTOR;
  }
  return ASPD_OK;
}

struct Region { int lo, hi; };

// Regions inside the page table, page alignment, overlap, page ids.
int check_layout(const aspd_shape_t* s, const aspd_request_t* req, const aspd_branch_t* br, const int32_t* page_ids,
                 int n_req, int64_t n_pool_pages, int mode) {
  if (n_req > 0 && !page_ids) return ASPD_ERR_INVALID_ARG;
  if (n_pool_pages < 0) return ASPD_ERR_INVALID_ARG;
  std::vector<uint8_t> used((size_t)n_pool_pages, 0);
  std::vector<Region> regs;
  for (int r = 0; r < n_req; ++r) {
    const aspd_request_t& q = req[r];
    if (q.page_begin < 0 || q.n_pages < 0) return ASPD_ERR_BAD_DESCRIPTOR;
    const long cap = (long)q.n_pages * s->page_size;
    regs.clear();
    regs.push_back({0, q.prefix_len});
    for (int b = 0; b < q.n_branches; ++b) {
      const aspd_branch_t& x = br[q.branch_begin + b];
      if (x.kv_off % s->page_size) return ASPD_ERR_BAD_DESCRIPTOR;
      regs.push_back({x.kv_off, x.kv_off + x.kv_len});
    }
    if (mode == ASPD_MODE_SERIAL || q.tail_len > 0) {
      if (q.tail_off % s->page_size) return ASPD_ERR_BAD_DESCRIPTOR;
      regs.push_back({q.tail_off, q.tail_off + q.tail_len});
    }
    for (const Region& g : regs)
      if (g.hi > cap) return ASPD_ERR_BAD_DESCRIPTOR;
    regs.erase(std::remove_if(regs.begin(), regs.end(), [](const Region& g) { return g.hi <= g.lo; }), regs.end());
    std::sort(regs.begin(), regs.end(), [](const Region& a, const Region& b) { return a.lo < b.lo; });
    for (size_t i = 1; i < regs.size(); ++i)
      if (regs[i].lo < regs[i - 1].hi) return ASPD_ERR_BAD_DESCRIPTOR;
    for (int p = 0; p < q.n_pages; ++p) {
      int32_t id = page_ids[q.page_begin + p];
      if (id < 0 || id >= n_pool_pages) return ASPD_ERR_BAD_DESCRIPTOR;
      if (used[id]) return ASPD_ERR_BAD_DESCRIPTOR;
      used[id] = 1;
    }
  }
  return ASPD_OK;
}

}  // namespace

extern "C" {

const char* aspd_strerror(int status) {
  switch (status) {
    case ASPD_OK: return "ok";
    case ASPD_ERR_INVALID_ARG: return "invalid argument";
    case ASPD_ERR_BAD_DESCRIPTOR: return "bad descriptor (overlap, out-of-table slot, alignment, q_len > kv_len or page id)";
    case ASPD_ERR_UNSUPPORTED: return "unsupported shape (head_dim, page_size or dtype)";
    case ASPD_ERR_CUDA: return "CUDA runtime or launch error";
    case ASPD_ERR_TIMEOUT: return "a bounded device-side wait ran out";
    case ASPD_ERR_NOMEM: return "out of memory";
    case ASPD_ERR_TOO_LARGE: return "size exceeds a stated maximum";
    default: return "unknown status";
  }
}

size_t aspd_pool_bytes(const aspd_shape_t* shape, int64_t n_pages) {
  if (check_shape(shape) != ASPD_OK || n_pages < 0) return 0;
  return (size_t)n_pages * shape->n_kv_heads * tile_bytes(shape->page_size, shape->head_dim, esize_of(shape->dtype));
}

int aspd_count_new_tokens(const aspd_request_t* req, const aspd_branch_t* br, int n_req, int mode) {
  int rc = check_counts(req, br, n_req, mode);
  if (rc != ASPD_OK) return rc;
  long n = 0;
  for (int r = 0; r < n_req; ++r) {
    if (mode == ASPD_MODE_SERIAL) { ++n; continue; }
    for (int b = 0; b < req[r].n_branches; ++b) n += std::max(0, br[req[r].branch_begin + b].q_len);
  }
  if (n > (1 << 24)) return ASPD_ERR_TOO_LARGE;
  return (int)n;
}

int aspd_positions(const aspd_request_t* req, const aspd_branch_t* br, int n_req, int mode, int32_t* pos_out,
                   int32_t* slot_out, int32_t* req_out) {
  int n = aspd_count_new_tokens(req, br, n_req, mode);
  if (n < 0) return n;
  if (n > 0 && (!pos_out || !slot_out)) return ASPD_ERR_INVALID_ARG;
  int t = 0;
  for (int r = 0; r < n_req; ++r) {
    const aspd_request_t& q = req[r];
    if (mode == ASPD_MODE_BRANCH) {
      // Eq. 4, stage_start: every token cached before the stage counts -- the prefix and the regions
      // of earlier stages (merged branches, serial tokens between stages); all branches share it
      long stage_start = q.prefix_len;
      for (int b = 0; b < q.n_branches; ++b)
        if (br[q.branch_begin + b].q_len == ASPD_Q_SHARED) stage_start += br[q.branch_begin + b].kv_len;
      for (int b = 0; b < q.n_branches; ++b) {
        const aspd_branch_t& x = br[q.branch_begin + b];
        const long first = x.pos_start == ASPD_POS_AUTO ? stage_start : (long)x.pos_start;
        for (int i = 0; i < x.q_len; ++i, ++t) {
          int k = x.kv_len - x.q_len + i;        // index of the token inside its branch
          if (first + k > INT32_MAX) return ASPD_ERR_TOO_LARGE;
          pos_out[t] = (int32_t)(first + k);     // Eq. 4: stage_start + delta
          slot_out[t] = x.kv_off + k;
          if (req_out) req_out[t] = r;
        }
      }
    } else {
      long total = q.prefix_len;                  // Eq. 4, main branch: every cached token counts
      for (int b = 0; b < q.n_branches; ++b) total += br[q.branch_begin + b].kv_len;
      pos_out[t] = (int32_t)(total + q.tail_len - 1);
      slot_out[t] = q.tail_off + q.tail_len - 1;
      if (req_out) req_out[t] = r;
      ++t;
    }
  }
  return ASPD_OK;
}

int aspd_visible_slots(const aspd_request_t* req, const aspd_branch_t* br, int n_req, int mode, int n_slots,
                       uint8_t* vis_out) {
  return aspd_visible_slots_masked(req, br, n_req, mode, ASPD_MASK_BRANCH_INVISIBLE, n_slots, vis_out);
}

int aspd_visible_slots_masked(const aspd_request_t* req, const aspd_branch_t* br, int n_req, int mode, int mask, int n_slots,
                              uint8_t* vis_out) {
  int n = aspd_count_new_tokens(req, br, n_req, mode);
  if (n < 0) return n;
  if (!vis_out || n_slots < 0 || (mask != ASPD_MASK_BRANCH_INVISIBLE && mask != ASPD_MASK_SHARED)) return ASPD_ERR_INVALID_ARG;
  memset(vis_out, 0, (size_t)n * n_slots);
  int t = 0;
  auto mark = [&](int tok, int lo, int hi) -> int {
    if (hi > n_slots) return ASPD_ERR_INVALID_ARG;
    for (int s = lo; s < hi; ++s) vis_out[(size_t)tok * n_slots + s] = 1;
    return ASPD_OK;
  };
  for (int r = 0; r < n_req; ++r) {
    const aspd_request_t& q = req[r];
    if (mode == ASPD_MODE_BRANCH) {
      for (int b = 0; b < q.n_branches; ++b) {
        const aspd_branch_t& x = br[q.branch_begin + b];
        for (int i = 0; i < x.q_len; ++i, ++t) {
          if (mark(t, 0, q.prefix_len)) return ASPD_ERR_INVALID_ARG;
          for (int s2 = 0; s2 < q.n_branches; ++s2) {          // regions of earlier stages (Eq. 3, third case)
            const aspd_branch_t& y = br[q.branch_begin + s2];
            if (y.q_len == ASPD_Q_SHARED && mark(t, y.kv_off, y.kv_off + y.kv_len)) return ASPD_ERR_INVALID_ARG;
          }
          const int k = x.kv_len - x.q_len + i;                // the token's offset in its branch
          if (mark(t, x.kv_off, x.kv_off + k + 1)) return ASPD_ERR_INVALID_ARG;
          if (mask == ASPD_MASK_SHARED)                         // smaller offsets of the stage's other branches
            for (int s2 = 0; s2 < q.n_branches; ++s2) {
              const aspd_branch_t& y = br[q.branch_begin + s2];
              if (s2 != b && y.q_len != ASPD_Q_SHARED && mark(t, y.kv_off, y.kv_off + std::min(k, y.kv_len))) return ASPD_ERR_INVALID_ARG;
            }
        }
      }
    } else {
      if (mark(t, 0, q.prefix_len)) return ASPD_ERR_INVALID_ARG;
      for (int b = 0; b < q.n_branches; ++b) {
        const aspd_branch_t& x = br[q.branch_begin + b];
        if (mark(t, x.kv_off, x.kv_off + x.kv_len)) return ASPD_ERR_INVALID_ARG;
      }
      if (mark(t, q.tail_off, q.tail_off + q.tail_len)) return ASPD_ERR_INVALID_ARG;
      ++t;
    }
  }
  return ASPD_OK;
}

static int plan_to_device(aspd_plan* p, cudaStream_t s);

// like: the plan that this one is to take the place of (aspd_plan_update re-plans on the host for the device that
// plan lives on): the grid of its device, its way of splitting the streams and, as far as possible, of writing new rows
// coarse: fewer and longer items, for host-only plans whose records would not fit into the static scratch otherwise
static int plan_create_impl(const aspd_shape_t* shape, const aspd_request_t* req, const aspd_branch_t* br,
                            const int32_t* page_ids, int n_req, int64_t n_pool_pages, int mode, const int32_t* q_pos,
                            const aspd_tuning_t* tuning, void* stream, const aspd_plan* like, bool coarse, aspd_plan_t** plan_out) {
  if (!plan_out) return ASPD_ERR_INVALID_ARG;
  *plan_out = nullptr;
  int rc = check_shape(shape);
  if (rc) return rc;
  rc = check_counts(req, br, n_req, mode);
  if (rc) return rc;
  rc = check_layout(shape, req, br, page_ids, n_req, n_pool_pages, mode);
  if (rc) return rc;
  const int n_new = aspd_count_new_tokens(req, br, n_req, mode);
  if (n_new < 0) return n_new;

  aspd_tuning_t tune = {ASPD_KERNEL_AUTO, 0, 0, 0, 0, ASPD_MASK_BRANCH_INVISIBLE, 0, ASPD_COMBINE_AUTO, 0, 0};
  if (tuning) tune = *tuning;
  const int ps = shape->page_size, d = shape->head_dim, Hq = shape->n_q_heads, Hkv = shape->n_kv_heads;
  const int G = Hq / Hkv, es = esize_of(shape->dtype);
  if (tune.chunk_tokens < 0 || tune.chunk_tokens % ps || tune.n_ctas < 0) return ASPD_ERR_INVALID_ARG;
  if (tune.mask != ASPD_MASK_BRANCH_INVISIBLE && tune.mask != ASPD_MASK_SHARED) return ASPD_ERR_INVALID_ARG;
  if (tune.wide_rows != 0 && tune.wide_rows != 128 && tune.wide_rows != 256) return ASPD_ERR_INVALID_ARG;
  if (tune.mma_m != 0 && tune.mma_m != 64 && tune.mma_m != 96 && tune.mma_m != 128) return ASPD_ERR_INVALID_ARG;
  if (tune.combine != ASPD_COMBINE_AUTO && tune.combine != ASPD_COMBINE_KERNEL && tune.combine != ASPD_COMBINE_FUSED) return ASPD_ERR_INVALID_ARG;
  const bool shared_mask = tune.mask == ASPD_MASK_SHARED && mode == ASPD_MODE_BRANCH;
  const bool mma_ok = shape->dtype == ASPD_DTYPE_BF16;
  const bool wide_ok = mma_ok && d == 128 && ps == 16;                 // aspd_attn_tc.cu; the other bf16 shapes: aspd_attn_dec.cu
  int kernel = tune.kernel;
  if (kernel == ASPD_KERNEL_AUTO) kernel = mma_ok ? ASPD_KERNEL_MMA : ASPD_KERNEL_GENERIC;
  if (kernel == ASPD_KERNEL_MMA && !mma_ok) return ASPD_ERR_UNSUPPORTED;
  if (kernel != ASPD_KERNEL_MMA && kernel != ASPD_KERNEL_GENERIC) return ASPD_ERR_INVALID_ARG;

  aspd_plan* p = new (std::nothrow) aspd_plan();
  if (!p) return ASPD_ERR_NOMEM;
  p->shape = *shape; p->mode = mode; p->n_req = n_req; p->n_new = n_new; p->kernel = kernel;
  p->stable_cache = tune.stable_cache ? 1 : 0;
  p->shared_mask = (tune.mask == ASPD_MASK_SHARED && mode == ASPD_MODE_BRANCH) ? 1 : 0;
  p->dec = kernel == ASPD_KERNEL_MMA && !wide_ok;
  p->host_only = tune.host_only; p->n_pool_pages = n_pool_pages; p->device_base = nullptr; p->device_bytes = 0;
  memset(&p->dev, 0, sizeof(p->dev));
  p->tune = tune;
  p->sm_count = like ? like->sm_count : 148;
  if (!tune.host_only && !like) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      delete p; return ASPD_ERR_CUDA;
    }
    p->sm_count = sms;
  }

  // ---- new-token table --------------------------------------------------------------
  std::vector<int32_t> pos(n_new), slot(n_new), treq(n_new), tok_page(n_new), tok_row(n_new);
  rc = aspd_positions(req, br, n_req, mode, pos.data(), slot.data(), treq.data());
  if (rc) { delete p; return rc; }
  for (int t = 0; t < n_new; ++t) {
    tok_page[t] = page_ids[req[treq[t]].page_begin + slot[t] / ps];
    tok_row[t] = slot[t] % ps;
    if (q_pos) { if (q_pos[t] < 0) { delete p; return ASPD_ERR_INVALID_ARG; } pos[t] = q_pos[t]; }
  }

  // ---- key streams -------------------------------------------------------------------
  // Per request, the pages the step must read, in one sequence: the prefix, then every branch
  // that has queries (branch mode) or every branch and the tail (serial mode).  Each entry is
  // (physical page, valid rows); the padding rows of partly filled pages are masked by the
  // kernels.  A new token sees stream keys [0, pe) (the prefix) and [lo, hi) (its own branch up
  // to itself); a serial token sees the whole stream.
  // With block_tok > 0 (plans that deal whole streams) every run of block_tok query tokens of a
  // request gets a sequence of its own: the prefix and, of the branches, only the pages that one
  // of the run's tokens can see.
  const int max_tok = std::max(1, kMaxRowsPerItem / G);
  struct Block { int request, tok0, n_tok, visit0, n_pages; };
  std::vector<int2> visit;
  std::vector<Block> blocks;
  std::vector<int4> tok_vis(n_new);
  int64_t kv_tokens = 0;
  const bool tok_field_fits = n_new < (1 << 18);      // the 18 bits above bit 13 of a page entry hold a token index
  bool counts_fit = true;                             // the 5 bits before them every page's number of new rows
  auto build_visit = [&](int block_tok) {
    visit.clear(); blocks.clear();
    counts_fit = true;
    int64_t kv_count = 0;
    int t = 0;
    // new_key0 / new_tok0: the keys [new_key0, len) of the region are this step's new tokens
    // new_tok0, new_tok0 + 1, ...; a page entry carries (valid rows | new rows << 8 | first new
    // token << 13) so that a fused step can write those rows just before it reads the page.
    // Under the shared mask the upper bits carry the page's index inside its branch instead (its
    // first key's offset / page_size; such plans never fuse the append): a token at offset k
    // also sees the keys of other branches whose offset is below k.
    auto push_region = [&](const aspd_request_t& q, int slot0, int len, int new_key0, int new_tok0, bool branch_pages = false) {
      const size_t at = visit.size();
      const int32_t* ids = page_ids + q.page_begin + slot0 / ps;
      const int n_old = (shared_mask && branch_pages) ? 0 : std::min(len, new_key0) / ps;       // full pages without new rows
      visit.resize(at + (len + ps - 1) / ps);
      int2* out = visit.data() + at;
      for (int i = 0; i < n_old; ++i) out[i] = make_int2(ids[i], ps);
      for (int s0 = n_old * ps; s0 < len; s0 += ps) {
        const int nv = std::min(ps, len - s0), first_new = std::max(s0, new_key0);
        const int n_newrows = std::max(0, s0 + nv - first_new);
        int y = nv;
        // 5 bits: a page of 32 new rows says 31, which is enough to tell that it has some, but not to write them
        if (n_newrows > 31) counts_fit = false;
        if (n_newrows > 0) y |= (std::min(n_newrows, 31) << 8);
        if (shared_mask) y |= branch_pages ? (s0 / ps) << 13 : 0;
        else if (n_newrows > 0 && tok_field_fits) y |= (new_tok0 + first_new - new_key0) << 13;
        out[s0 / ps] = make_int2(ids[s0 / ps], y);
      }
    };
    auto push_shared = [&](const aspd_request_t& q) {            // prefix and regions of earlier stages: seen by every branch
      push_region(q, 0, q.prefix_len, q.prefix_len, 0);
      for (int b = 0; b < q.n_branches; ++b) {
        const aspd_branch_t& x = br[q.branch_begin + b];
        if (x.q_len == ASPD_Q_SHARED) push_region(q, x.kv_off, x.kv_len, x.kv_len, 0);
      }
    };
    for (int r = 0; r < n_req; ++r) {
      const aspd_request_t& q = req[r];
      const int t_req = t, v0 = (int)visit.size();
      if (mode == ASPD_MODE_BRANCH) {
        int nq = 0;
        int64_t kv_req = q.prefix_len;                         // keys of this request that the step reads
        for (int b = 0; b < q.n_branches; ++b) {
          const aspd_branch_t& x = br[q.branch_begin + b];
          nq += std::max(0, x.q_len);
          if (x.q_len != 0 || shared_mask) kv_req += x.kv_len;
        }
        if (nq == 0) continue;
        kv_count += kv_req;
        if (block_tok == 0) {
          push_shared(q);
          const int pe = ((int)visit.size() - v0) * ps;
          for (int b = 0; b < q.n_branches; ++b) {
            const aspd_branch_t& x = br[q.branch_begin + b];
            if (x.q_len < 0 || (x.q_len == 0 && !shared_mask)) continue;     // shared mask: also branches without queries
            const int lo = ((int)visit.size() - v0) * ps, prior = x.kv_len - x.q_len;
            push_region(q, x.kv_off, x.kv_len, prior, t, true);
            for (int i = 0; i < x.q_len; ++i) tok_vis[t++] = make_int4(pe, lo, lo + prior + i + 1, shared_mask ? prior + i : 0);
          }
          blocks.push_back({r, t_req, nq, v0, (int)visit.size() - v0});
        } else {
          int n_shared = 0;                                    // pages that every block of the request lists
          for (int blk0 = 0; blk0 < nq; blk0 += block_tok) {
            const int blk1 = std::min(nq, blk0 + block_tok), bv0 = (int)visit.size();
            if (blk0 == 0) {
              push_shared(q);
              n_shared = (int)visit.size() - bv0;
            } else {                                           // as in the request's first block
              visit.resize((size_t)bv0 + n_shared);
              std::copy(visit.begin() + v0, visit.begin() + v0 + n_shared, visit.begin() + bv0);
            }
            const int pe = n_shared * ps;
            int off = 0;                                       // index, among the request's new tokens, of the branch's first
            for (int b = 0; b < q.n_branches; ++b) {
              const aspd_branch_t& x = br[q.branch_begin + b];
              if (x.q_len <= 0) continue;
              const int a = std::max(blk0, off), e = std::min(blk1, off + x.q_len);
              if (a < e) {
                const int lo = ((int)visit.size() - bv0) * ps, prior = x.kv_len - x.q_len;
                push_region(q, x.kv_off, prior + (e - off), prior, t_req + off);   // up to the run's last token of this branch
                for (int i = a - off; i < e - off; ++i) tok_vis[t_req + off + i] = make_int4(pe, lo, lo + prior + i + 1, 0);
              }
              off += x.q_len;
            }
            blocks.push_back({r, t_req + blk0, blk1 - blk0, bv0, (int)visit.size() - bv0});
          }
          t += nq;
        }
      } else {
        push_region(q, 0, q.prefix_len, q.prefix_len, 0);
        kv_count += q.prefix_len + q.tail_len;
        for (int b = 0; b < q.n_branches; ++b) {
          const aspd_branch_t& x = br[q.branch_begin + b];
          push_region(q, x.kv_off, x.kv_len, x.kv_len, 0);
          kv_count += x.kv_len;
        }
        push_region(q, q.tail_off, q.tail_len, q.tail_len - 1, t);
        tok_vis[t++] = make_int4(kCausalAll, 0, 0, 0);
        blocks.push_back({r, t_req, 1, v0, (int)visit.size() - v0});
      }
    }
    kv_tokens = kv_count;
  };
  build_visit(0);

  // ---- work items: a contiguous, equal share of all pages for every CTA -----------------
  // Streams are walked in the order (request, row block, KV head); the concatenation of all
  // streams is cut at the CTA boundaries (and, if asked for, every chunk_tokens keys).
  struct Stream { int request, tok0, n_tok, head, page0, n_pages, row_block; };
  std::vector<int2> row_blocks;
  std::vector<Stream> streams;
  long total_pages = 0;
  auto build_streams = [&](int tok_per_block) {
    row_blocks.clear(); streams.clear(); total_pages = 0;
    for (const Block& bk : blocks) {
      if (bk.n_tok == 0 || bk.n_pages == 0) continue;
      for (int i0 = 0; i0 < bk.n_tok; i0 += tok_per_block) {
        row_blocks.push_back(make_int2(bk.tok0 + i0, std::min(tok_per_block, bk.n_tok - i0)));
        for (int h = 0; h < Hkv; ++h) {
          streams.push_back({bk.request, bk.tok0 + i0, std::min(tok_per_block, bk.n_tok - i0), h, bk.visit0, bk.n_pages,
                             (int)row_blocks.size() - 1});
          total_pages += bk.n_pages;
        }
      }
    }
  };
  build_streams(max_tok);
  const bool cores = kernel == ASPD_KERNEL_GENERIC;
  // pages that a CTA gets at least, and the grain of cuts inside a stream
  const int cta_pages = coarse ? 8 : std::max(1, (cores ? 32 : 128) / ps), tile_pages = !coarse ? cta_pages : ps == 16 ? 8 : 1;
  auto ctas_for = [&](long pages) {
    // do not cut finer than one 128-key tile per CTA (measured on a 2.5 k-token step: 80 CTAs with a
    // full tile each take 10.6 us per layer, 148 CTAs with half a tile 11.9: fewer records to combine);
    // the CUDA-core kernel takes 32 keys at a time and two of its CTAs fit an SM
    const int want = tune.n_ctas > 0 ? tune.n_ctas : p->sm_count * (cores && !coarse ? 2 : 1);
    return (int)std::max(1L, std::min((long)want, (pages + cta_pages - 1) / cta_pages));
  };
  // Dealing the streams out whole, largest first, each to the CTA with the least so far.  A stream costs its pages and
  // kDealItem more.  Returned: the largest share over the mean one.  (Rounds back and forth over the CTAs, as they were
  // dealt before, left the first CTAs with a stream more and 8 to 12 % more pages: 160 requests, 212 us a layer
  // against 204; the streams of masked prefill are so many that both come out even.)
  std::vector<std::vector<int>> mine;
  auto deal_out = [&](int n_ctas) {
    constexpr double kDealItem = 8.0;
    std::vector<int> order(streams.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return streams[a].n_pages > streams[b].n_pages; });
    mine.assign(n_ctas, {});
    std::vector<std::pair<double, int>> load(n_ctas);                    // a heap, the CTA with the least on top
    for (int c = 0; c < n_ctas; ++c) load[c] = {0.0, c};
    double all = 0.0, most = 0.0;
    for (int si : order) {
      std::pop_heap(load.begin(), load.end(), std::greater<>());
      auto& [cost, c] = load.back();
      mine[c].push_back(si);
      cost += kDealItem + streams[si].n_pages;
      all += kDealItem + streams[si].n_pages;
      most = std::max(most, cost);
      std::push_heap(load.begin(), load.end(), std::greater<>());
    }
    return most * n_ctas / std::max(1.0, all);
  };
  // With many more streams than CTAs (a step with many query tokens per branch: masked prefill,
  // teacher forcing; a step of many requests) nothing is cut: every stream is one item whose CTA writes the output,
  // and no records go through memory to a combine launch.  The longest requests come first, so that at any moment
  // all CTAs read the K/V pages of the same one or two requests (which then stay in L2).
  // Every row block then gets a page sequence of its own, without the branch pages none of its
  // tokens sees, and the tensor-core kernel takes row blocks of up to 128 rows (its wide variant).
  // (only where the step fills the grid, or the caller chose the grid: a step of a few pages has few CTAs and many streams by default)
  // From four streams per CTA on always; from two on where the shares come out even.  Requests of 0.5-8 k tokens, four
  // KV heads, largest share over the mean one, us a layer dealt and cut: 100 requests 1.05, 134 and 146; 80 requests
  // 1.08, 105 and 120; 60 requests 1.41 to 1.52, 87 to 93 and 85 to 87; 40 requests 1.97 to 2.3, 79 and 56 to 61.
  constexpr double kDealSkew = 1.2;
  bool deal_streams = mode == ASPD_MODE_BRANCH && !shared_mask && tune.chunk_tokens == 0 &&
                      (long)streams.size() >= 2L * ctas_for(total_pages) && (tune.n_ctas > 0 || ctas_for(total_pages) >= p->sm_count);
  if (deal_streams && (long)streams.size() < 4L * ctas_for(total_pages)) deal_streams = !coarse && deal_out(ctas_for(total_pages)) <= kDealSkew;
  if (like) deal_streams = like->dealt != 0;
  p->wide = 0;
  if (deal_streams) {
    p->wide = (kernel == ASPD_KERNEL_MMA && wide_ok && kMaxRowsWide / G > max_tok) ? 1 : 0;
    // A step in which some request has more query tokens than one 128-row tile holds takes row blocks
    // of two tiles (the two-tile variant of the kernel: both tiles are scored against every K/V tile
    // the CTA fetches, one softmax group per tile), unless the caller asked for single tiles.
    if (p->wide && tune.wide_rows != 128) {
      int most_q = 0;
      for (const Block& bk : blocks) most_q = std::max(most_q, bk.n_tok);
      if (most_q > kMaxRowsWide / G || tune.wide_rows == 256) p->wide = 2;
    }
    const int tok_per_block = p->wide ? p->wide * (kMaxRowsWide / G) : max_tok;
    build_visit(tok_per_block);
    build_streams(tok_per_block);
  }
  p->max_rows = 0;
  for (const int2& rb : row_blocks) p->max_rows = std::max(p->max_rows, rb.y * G);
  const int base_ctas = ctas_for(total_pages);
  int n_ctas = like && like->tile_cut ? like->n_ctas : base_ctas;
  const int chunk_pages = tune.chunk_tokens > 0 ? tune.chunk_tokens / ps : (1 << 28);
  p->chunk_tokens = tune.chunk_tokens; p->base_ctas = base_ctas;
  std::vector<int32_t> n_parts((size_t)n_new * Hkv, 0), part_base((size_t)n_new * Hkv + 1, 0), cta_item0(n_ctas + 1, 0);
  p->dealt = deal_streams ? 1 : 0;
  std::vector<int> fresh;                          // entries of `visit` with new rows, ascending
  for (size_t i = 0; i < visit.size(); ++i)
    if ((visit[i].y >> 8) & 31) fresh.push_back((int)i);
  p->patch_tiles = (!deal_streams && total_pages <= 2L * 8 * base_ctas) ? 1 : 0;
  if (deal_streams) {
    deal_out(n_ctas);
    for (int c = 0; c < n_ctas; ++c) {
      cta_item0[c] = (int)p->items.size();
      for (int si : mine[c]) {
        const Stream& st = streams[si];
        DeviceItem it;
        it.q_tok0 = st.tok0; it.n_q_tok = st.n_tok; it.kv_head = st.head; it.page0 = st.page0; it.n_pages = st.n_pages;
        it.key0 = 0; it.part_slot = 0; it.request = st.request; it.row_block = st.row_block; it.n_parts = 1;
        p->items.push_back(it);
        for (int i = 0; i < st.n_tok; ++i) n_parts[(size_t)(st.tok0 + i) * Hkv + st.head] = 1;
      }
    }
    cta_item0[n_ctas] = (int)p->items.size();
  } else {
    // Every CTA gets the same cost, cost = pages + kItemCost per item it starts: an item boundary
    // (new query tile, ragged last tile, epilogue) costs about as much as streaming a dozen pages,
    // so CTAs that end up with several short items get fewer pages.
    const double kItemCost = coarse ? 12.0 : (cores ? 64.0 : 192.0) / ps;
    // a page costs a little more the more query rows are scored against it (best measured balance:
    // 0.35 % per row), so streams of requests with many branches weigh more
    const double kRowCost = 0.0035;
    auto page_cost = [&](const Stream& st) { return 1.0 + kRowCost * st.n_tok * G; };
    // A CTA that comes to a page with new rows within its first 160 keys waits for them (its first tiles arrive while
    // the kernel before this one still runs, the rows are written after it), unless the rows are put into the tiles
    // (patch_tiles): it gets fewer pages, as many as it could have had by then.  Cuts lie on tile boundaries, so a
    // single step can gain or lose a tile: judged over many.  At 0 / 96 / 128 / 160 / 192 / 256 keys, mean us a layer: six
    // requests of 9 to 16 k tokens with eight branches 16.1 / 15.8 / 15.5 / 15.4 / 15.1 / 15.5 (one of them 16.9 / 16.6 /
    // 16.4 / 16.0 / 15.8 / 16.4), steps of 3 to 20 requests 18.9 / 18.8 / 18.7 / 18.5 / 18.5 / 18.5 (worst step against 0:
    // at 160 2.6 % slower, at 192 3.5 %, at 256 the 12 k request 11 %); 32 requests, whose CTAs have two dozen tiles
    // each, come out the same.
    const double kWait = (kernel == ASPD_KERNEL_MMA && !p->patch_tiles && !coarse) ? 160.0 / ps : 0.0;
    // the share is re-derived from what is left whenever a CTA is closed, so rounding does not pile up
    // (the sum of the waits is not known before the cuts are: made twice where there are any)
    auto cut = [&](double waits_left) {
      double cost_left = 0.0, waits = 0.0;
      for (const Stream& st : streams) cost_left += page_cost(st) * st.n_pages;
      long streams_left = (long)streams.size();
      auto share_now = [&](int ctas_left) {
        return (cost_left + std::max(0.0, waits_left) + kItemCost * ((double)streams_left + ctas_left)) / std::max(1, ctas_left);
      };
      double share = share_now(n_ctas);
      int cta = 0;
      double acc = 0.0;                              // cost already given to the current CTA
      int done = 0;                                  // its pages
      bool waited = false;                           // it has come to a page with new rows
      p->items.clear();
      auto next_cta = [&]() { cta_item0[++cta] = (int)p->items.size(); acc = 0.0; done = 0; waited = false; share = share_now(n_ctas - cta); };
      // what the CTA waits, in pages, when it goes on with `take` pages from entry `from` of `visit`
      auto wait_for = [&](int from, long take) {
        if (waited || done >= kWait) return 0.0;
        const auto e = std::lower_bound(fresh.begin(), fresh.end(), from);
        return e == fresh.end() || *e >= from + take ? 0.0 : std::max(0.0, kWait - done - (*e - from));
      };
      for (const Stream& st : streams) {
        int at = 0, slot = 0;
        const size_t first_item = p->items.size();
        const double pc = page_cost(st);
        --streams_left;
        while (at < st.n_pages) {
          double room = (share - acc - kItemCost) / pc;   // pages that still fit if an item starts here
          if (room < 1.0 && acc > 0.0 && cta + 1 < n_ctas) { next_cta(); continue; }
          long take = std::min<long>(st.n_pages - at, chunk_pages);
          if (cta + 1 < n_ctas) take = std::min<long>(take, std::max<long>(1, (long)(room + 0.5)));
          // a cut inside a stream goes on a tile boundary (128 keys; CUDA cores: 32) where the item is long
          // enough: the item's last tile is then a full one (measured on the serving mix: 0.4 % on the step)
          if (take < st.n_pages - at && tune.chunk_tokens == 0 && take >= tile_pages + tile_pages / 2)
            take = std::min<long>((take + tile_pages / 2) / tile_pages * tile_pages, st.n_pages - at);
          double wait = wait_for(st.page0 + at, take);
          if (wait > 0.0 && cta + 1 < n_ctas) {
            room -= wait / pc;
            if (room < 1.0 && acc > 0.0) { next_cta(); continue; }
            if (tune.chunk_tokens == 0 && room < (double)take) {
              take = std::max<long>(1, (long)(room + 0.5));
              if (take >= tile_pages + tile_pages / 2) take = (take + tile_pages / 2) / tile_pages * tile_pages;
              take = std::min<long>(take, st.n_pages - at);
              wait = wait_for(st.page0 + at, take);
            }
          }
          DeviceItem it;
          it.q_tok0 = st.tok0; it.n_q_tok = st.n_tok; it.kv_head = st.head; it.page0 = st.page0 + at;
          it.n_pages = (int)take; it.key0 = at * ps; it.part_slot = slot++; it.request = st.request;
          it.row_block = st.row_block; it.n_parts = 0;
          p->items.push_back(it);
          at += (int)take;
          cost_left -= pc * take;
          acc += kItemCost + pc * (double)take + wait;
          waits += wait; waits_left -= wait; waited |= wait > 0.0; done += (int)take;
          if (acc >= share - 0.5 && cta + 1 < n_ctas) next_cta();
        }
        for (int i = 0; i < st.n_tok; ++i) n_parts[(size_t)(st.tok0 + i) * Hkv + st.head] = slot;
        for (size_t i = first_item; i < p->items.size(); ++i) p->items[i].n_parts = slot;
      }
      while (cta < n_ctas) cta_item0[++cta] = (int)p->items.size();
      return waits;
    };
    if (!(like && like->tile_cut)) {
      const double waits = cut(0.0);
      if (waits > 0.0) cut(waits);
    }
    // A step of a few tiles per CTA takes as long as its slowest CTA, and that is a chain of tiles, whatever they hold, and
    // of items.  The cut above counts pages: one request of 2.5 k keys became 71 CTAs of one tile and 11 of nine pages,
    // which are two.  So such a step is also cut by tiles: every CTA one item of at most T tiles, the least T for which
    // the SMs suffice, fewer where it would wait for new rows within its first kWaitKeys keys; and that cut is taken if
    // its longest CTA has fewer tiles, or (up to four) as many where the other has CTAs of several items and there are
    // hardly fewer of them.  us a pass, cut by pages and by tiles: 2 tiles and 1: one request of 2.5 k keys 244 and 235,
    // a serial step over 1.1 k 196 and 185; 4 and 3: two requests opened with up to 26 tokens a branch 393 and 381; 4
    // with two items and 4: 17 k keys 418 and 406.  Not where the tiles come out the same (four requests of 2.2 k: 461
    // and 498 by tiles) and not with several items to a CTA (six branches opened with twelve tokens, 3 and 2 tiles: 395
    // and 408).  Over 51 random steps that are cut by tiles so, of all three tensor-core shapes, the cut by pages takes
    // 4.3 % longer in the mean, 27 % at most, and is never faster by more than 1 %.  Both numbers of kept lines against
    // others, steps that come out differently: "up to four" against two, five steps 4.7 % slower; against six, nine 2.5 %
    // faster (two of them slower); nine tenths as many items against as many, three 7 % slower; against eight tenths,
    // seven 3.4 % faster.  kWaitKeys between 160 and 640 makes the same cuts.
    constexpr int kWaitKeys = 480, kTileCost = 320;          // a tile is 128 keys and a chain as long as 192 more
    const int tp = 128 / ps;                                 // pages of a tile
    if (kernel == ASPD_KERNEL_MMA && !coarse && tune.chunk_tokens == 0 && tune.n_ctas == 0 && !streams.empty() && !(like && !like->tile_cut) &&
        (like || total_pages <= 6L * tp * base_ctas)) {
      const int most = like ? n_ctas : p->sm_count;
      if ((long)streams.size() > most && like) { delete p; return ASPD_ERR_UNSUPPORTED; }      // an item each at least
      // Pages of the items, an item of at most T tiles to every CTA, fewer for one that comes to new rows within its first
      // `wait_keys` keys; false: too few SMs.  Row block by row block: its streams, one to a KV head, are cut alike.
      std::vector<int> takes;
      auto pack = [&](int T, int wait_keys) {
        takes.clear();
        for (size_t s = 0; s < streams.size(); s += Hkv) {
          const Stream& st = streams[s];
          for (int at = 0; at < st.n_pages; at += takes.back()) {
            int take = std::min(T * tp, st.n_pages - at);
            if (wait_keys > 0) {
              const auto e = std::lower_bound(fresh.begin(), fresh.end(), st.page0 + at);
              const int before = e == fresh.end() ? take : *e - st.page0 - at;         // pages before the first with new rows
              const long wait = wait_keys - (long)kTileCost * (before / tp);
              if (before < take && wait > 0) take = (int)std::min<long>(take, std::max(1L, ((long)T * kTileCost - wait) / kTileCost) * tp);
            }
            takes.push_back(take);
          }
          if ((long)takes.size() * Hkv > most) return false;
        }
        return true;
      };
      // of those: f(pages, first page in `visit`, stream) for every row block's items
      auto each_take = [&](auto f) {
        size_t i = 0;
        for (size_t s = 0; s < streams.size(); s += Hkv)
          for (int at = 0; at < streams[s].n_pages; at += takes[i++]) f(takes[i], streams[s].page0 + at, streams[s]);
      };
      long tiles = 0;
      int longest_stream = 0;
      for (const Stream& st : streams) {
        tiles += (st.n_pages + tp - 1) / tp;
        longest_stream = std::max(longest_stream, (st.n_pages + tp - 1) / tp);
      }
      // items of T tiles, which no wait makes fewer
      auto least_items = [&](int T) {
        long n = 0;
        for (size_t s = 0; s < streams.size(); s += Hkv) n += (streams[s].n_pages + T * tp - 1) / (T * tp);
        return n * Hkv;
      };
      int longest = 0;                               // of the cut by pages
      for (int c = 0; !like && c < n_ctas; ++c) {
        int n = 0;
        for (int i = cta_item0[c]; i < cta_item0[c + 1]; ++i) n += (p->items[i].n_pages + tp - 1) / tp;
        longest = std::max(longest, n);
      }
      const int several = (int)p->items.size() > n_ctas && longest <= 4 ? 1 : 0;
      // new rows that come to a CTA, and whether some CTA would have more than it writes itself
      auto rows_of = [&](int from, int n_pages) {
        int n = 0;
        for (auto e = std::lower_bound(fresh.begin(), fresh.end(), from); e != fresh.end() && *e < from + n_pages; ++e) n += (visit[*e].y >> 8) & 31;
        return n;
      };
      auto many_rows = [&]() {
        bool many = false;
        each_take([&](int take, int from, const Stream&) { many |= rows_of(from, take) > kMostFusedRows; });
        return many;
      };
      auto many_rows_by_pages = [&]() {
        for (int c = 0; c < n_ctas; ++c) {
          int n = 0;
          for (int i = cta_item0[c]; i < cta_item0[c + 1]; ++i) n += rows_of(p->items[i].page0, p->items[i].n_pages);
          if (n > kMostFusedRows) return true;
        }
        return false;
      };
      // an update has the room of the plan that it updates, and its launches
      auto fits_plan = [&]() {
        long records = 0;
        each_take([&](int, int, const Stream& st) { records += (long)st.n_tok * Hkv; });
        return takes.size() * Hkv <= like->layout.cap_items && records <= (long)like->layout.cap_partials &&
               !(like->fuse_append && like->patch_tiles && many_rows());
      };
      bool done = false;
      int T = (int)std::max(1L, (tiles + most - 1) / most);
      if (like) T = std::max(T, like->tile_cut);
      // (an update's streams have an item each at the latest with as many tiles as the longest has)
      const int last = like ? std::max(T, longest_stream) : longest + several - 1;
      for (; !done && T <= last; ++T)
        for (int w = least_items(T) > most ? -1 : p->patch_tiles ? 0 : kWaitKeys; !done && w >= 0; w -= kTileCost / 2) done = pack(T, w) && (!like || fits_plan());
      if (done && !like) {
        int now = 0;
        for (int take : takes) now = std::max(now, (take + tp - 1) / tp);
        done = now < longest || 10 * takes.size() * Hkv >= 9 * (size_t)n_ctas;
      }
      // not where a CTA gets more new rows than it writes itself and none has them by pages: such a step would take a
      // launch more.  Nor, if the plan is to be updated, the other way round: updates have to keep the plan's launches.
      if (done && !like) {
        const bool by_tiles = many_rows();
        if (by_tiles || tune.updatable) done = by_tiles == many_rows_by_pages();
      }
      if (done && tune.updatable && !like) {
        p->room_items = p->items.size();
        for (const DeviceItem& it : p->items) p->room_partials += it.n_q_tok;
      }
      if (!done && like) {                             // an update that no cut by tiles fits is cut by pages
        const double waits = cut(0.0);
        if (waits > 0.0) cut(waits);
      }
      if (done) {
        p->tile_cut = T - 1;
        p->items.clear();
        size_t i0 = 0;
        for (size_t s = 0; s < streams.size(); s += Hkv) {
          size_t i1 = i0;
          for (int h = 0; h < Hkv; ++h) {
            const Stream& st = streams[s + h];
            int at = 0;
            for (i1 = i0; at < st.n_pages; at += takes[i1++]) {
              DeviceItem it;
              it.q_tok0 = st.tok0; it.n_q_tok = st.n_tok; it.kv_head = st.head; it.page0 = st.page0 + at; it.n_pages = takes[i1]; it.key0 = at * ps;
              it.part_slot = (int)(i1 - i0); it.request = st.request; it.row_block = st.row_block; it.n_parts = 0;
              p->items.push_back(it);
            }
            const int parts = (int)(i1 - i0);
            for (size_t i = p->items.size() - parts; i < p->items.size(); ++i) p->items[i].n_parts = parts;
            for (int i = 0; i < st.n_tok; ++i) n_parts[(size_t)(st.tok0 + i) * Hkv + st.head] = parts;
          }
          i0 = i1;
        }
        // (a plan to be updated in place has a CTA to spare for every stream, whose number of tiles may grow)
        if (!like) n_ctas = tune.updatable ? (int)std::min<long>(p->sm_count, std::max<long>((long)p->items.size(), base_ctas + (long)streams.size())) : (int)p->items.size();
        cta_item0.assign(n_ctas + 1, (int)p->items.size());
        for (int c = 0; c < (int)p->items.size(); ++c) cta_item0[c] = c;
      }
    }
  }
  p->n_ctas = n_ctas;
  // Rows that are new this step, per CTA: what a fused step must write before the CTA reads.  The fused step
  // writes them in batches at the start of the kernel; with many new rows per CTA (a branch-open step) the
  // separate append kernel is the faster way, and such plans carry no list.  (The few pages that hold new rows
  // are found once, not once per KV head and CTA.)
  std::vector<int4> dirty;
  std::vector<int32_t> cta_dirty0(n_ctas + 1, 0);
  p->fuse_append = (!shared_mask && tok_field_fits && counts_fit && p->wide != 2 && !(like && !like->fuse_append)) ? 1 : 0;
  // A CTA with that many tiles has its rows written long before it comes to the pages that hold them, so there more are
  // written at its start, as long as that does not take longer than the tiles: up to 2.5 to a tile over the step where
  // the streams are dealt, which begin with a prefix, and one to a tile in any CTA where they are cut, since a CTA may
  // then begin with the new rows.  8 layers from the host, us with the rows written here and by the append kernel:
  // dealt, 0.25 to 1 a tile 1540 and 1594, 858 and 896; 1.7 to 1.8 382 and 414, 772 and 788; 2.4 585 and 569; 4.3 1250
  // and 1103; 6 and 8 795 and 665, 765 and 630.  Cut, 0.6 to 0.7 a tile 638 and 648, 606 and 613, 608 and 614; 1.3 478
  // and 456; 1.6 569 and 563; 5 to 8 523 and 419, 968 and 645, 1333 and 809 (branches of up to 100 tokens, 640 rows to a CTA).
  // Not where the tiles are patched: patch_tiles goes by the mean over the CTAs, so that one of them may be long (a
  // forced cut every chunk_tokens keys leaves the last CTA with dozens of short tiles), and the rows' place in shared
  // memory is kMostFusedRows long.
  constexpr int kLongCta = 16;
  long all_tiles = 0;
  bool many = false;                               // a CTA has more than kMostFusedRows
  const bool patches = like ? like->patch_tiles != 0 : p->patch_tiles != 0;      // an update's launches are the old plan's
  if (p->fuse_append) {
    for (int c = 0; c < n_ctas && p->fuse_append; ++c) {
      cta_dirty0[c] = (int)dirty.size();
      const int ppt = 128 / ps;                    // pages of a tile
      int tile0 = 0;                               // number of the item's first tile among the CTA's
      for (int i = cta_item0[c]; i < cta_item0[c + 1]; ++i) {
        const DeviceItem& it = p->items[i];
        for (auto e = std::lower_bound(fresh.begin(), fresh.end(), it.page0); e != fresh.end() && *e < it.page0 + it.n_pages; ++e) {
          const int2 v = visit[*e];
          const int cnt = (v.y >> 8) & 31, tok0 = v.y >> 13, row0 = (v.y & 255) - cnt;
          const int pg = *e - it.page0, place = (pg % ppt) << 8 | (tile0 + pg / ppt) << 16;
          for (int k = 0; k < cnt; ++k) dirty.push_back(make_int4(v.x, it.kv_head, tok0 + k, (row0 + k) | place));
        }
        tile0 += (it.n_pages + ppt - 1) / ppt;
      }
      // (32 767 tiles: what the number's field holds)
      const int rows = (int)dirty.size() - cta_dirty0[c];
      const bool more = !patches && !cores && (like || (tile0 >= kLongCta && !p->dec && (deal_streams || rows <= tile0)));
      if ((rows > kMostFusedRows && !more) || tile0 > 32767) p->fuse_append = 0;
      many |= rows > kMostFusedRows; all_tiles += tile0;
    }
    cta_dirty0[n_ctas] = (int)dirty.size();
    if (many && deal_streams && !like && dirty.size() > 2.5 * all_tiles) p->fuse_append = 0;
    if (!p->fuse_append) { dirty.clear(); std::fill(cta_dirty0.begin(), cta_dirty0.end(), 0); }
  }
  // the merge of a token's records inside the attention kernel: stream-K plans of the tensor-core kernel
  // 1: both MMAs with M = 64; 2: only P.V (the default: at most 64 of P.V's 128 rows are ever read, a quarter
  // less tensor work lifts the power-capped clock and the softmax layout, which M = 64 scores would slow
  // down, stays as it is); 0: both with M = 128
  p->m64 = (kernel == ASPD_KERNEL_MMA && !deal_streams && !p->dec) ? (tune.mma_m == 64 ? 1 : tune.mma_m == 128 ? 0 : 2) : 0;
  p->stagger_start = (!deal_streams && total_pages <= 6L * 8 * n_ctas) ? 1 : 0;       // at most six 128-key tiles per CTA
  // Merging inside the attention kernel is an option, not the default.  Measured on every workload of
  // the benchmark, the CTA that stores a pair's last record is a CTA at the very end of its own work,
  // so its fence, count and merge (1.5 us + one memory round trip per 16 rows of the pairs it ended
  // up with; all rows of a stream cut into dozens of parts land on one CTA) lengthen the kernel by
  // more than the combine launch costs, whose blocks are resident and waiting when the pass ends.
  p->single_launch = (kernel == ASPD_KERNEL_MMA && !deal_streams && !p->dec && tune.combine == ASPD_COMBINE_FUSED && max_tok <= 16) ? 1 : 0;   // 16: an item's tokens in the merge queue
  for (size_t i = 0; i < n_parts.size(); ++i) part_base[i + 1] = part_base[i] + n_parts[i];
  int max_parts = 0;                               // (not the plan's own in the loop, where it would be stored and read again every time)
  for (int n : n_parts) max_parts = std::max(max_parts, n);
  p->max_parts = max_parts;
  p->n_items = (int)p->items.size();
  p->n_partials = part_base[n_parts.size()];
  p->kv_tokens_read = kv_tokens;
  p->algorithmic_bytes = 2LL * Hkv * d * es * kv_tokens + 2LL * es * Hq * d * n_new + 2LL * Hkv * d * es * n_new;
  p->n_row_blocks = (int)row_blocks.size();
  p->visit.swap(visit); p->cta_item0.swap(cta_item0); p->part_base.swap(part_base); p->row_blocks.swap(row_blocks); p->q_pos.swap(pos);
  p->tok_vis.swap(tok_vis); p->tok_page.swap(tok_page); p->tok_row.swap(tok_row); p->dirty.swap(dirty); p->cta_dirty0.swap(cta_dirty0);
  if (tune.host_only) { *plan_out = p; return ASPD_OK; }
  rc = plan_to_device(p, (cudaStream_t)stream);
  if (rc) { delete p; return rc; }
  *plan_out = p;
  return ASPD_OK;
}

int aspd_plan_create(const aspd_shape_t* shape, const aspd_request_t* req, const aspd_branch_t* br,
                     const int32_t* page_ids, int n_req, int64_t n_pool_pages, int mode, const int32_t* q_pos,
                     const aspd_tuning_t* tuning, void* stream, aspd_plan_t** plan_out) {
  const int rc = plan_create_impl(shape, req, br, page_ids, n_req, n_pool_pages, mode, q_pos, tuning, stream, nullptr, false, plan_out);
  if (rc || !tuning || !tuning->host_only || fits_static_scratch(*plan_out)) return rc;
  // Cut for speed, the CUDA-core kernel's steps have up to two items per SM and so twice the records of steps that
  // give every SM one share: 28/4 heads of 128 in fp32, 16 tokens over 3 k, 9.9 MB instead of 5.0.  A host-only plan
  // that aspd_attn_static could not take is made again with those.
  aspd_plan_t* longer = nullptr;
  if (plan_create_impl(shape, req, br, page_ids, n_req, n_pool_pages, mode, q_pos, tuning, stream, nullptr, true, &longer) != ASPD_OK) return rc;
  if (fits_static_scratch(longer)) std::swap(longer, *plan_out);
  delete longer;
  return rc;
}

// ---- one device allocation, one staging blob ----------------------------------------------
// Offsets of the plan's tables inside its device block.  The tables whose size depends on the
// lengths of the step (items, page list, new-row list, partial records) get `slack` times the room
// they need now, so that aspd_plan_update can re-plan into the same addresses.
static void plan_layout(const aspd_plan* p, double slack, aspd::PlanLayout* L) {
  const aspd_shape_t& sh = p->shape;
  const int d = sh.head_dim, Hq = sh.n_q_heads, Hkv = sh.n_kv_heads, G = Hq / Hkv, es = esize_of(sh.dtype), n_new = p->n_new;
  auto cap = [&](size_t n) { return std::max<size_t>(1, (size_t)((double)n * slack) + (slack > 1.0 ? 64 : 0)); };
  L->cap_items = cap(std::max(p->items.size(), p->room_items)); L->cap_visit = cap(p->visit.size()); L->cap_dirty = cap(p->dirty.size());
  L->cap_partials = p->wide == 2 ? 1 : cap(std::max((size_t)p->n_partials, p->room_partials));      // (the two-tile kernel never writes records)
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  L->o_items = take(sizeof(DeviceItem) * L->cap_items);
  L->o_cta = take(2 * sizeof(int4) * std::max(1, p->n_ctas));
  L->o_visit = take(sizeof(int2) * L->cap_visit);
  L->o_dirty = take(sizeof(int4) * L->cap_dirty);
  L->o_tpage = take(sizeof(int32_t) * std::max(1, n_new));
  L->o_trow = take(sizeof(int32_t) * std::max(1, n_new));
  L->o_tpos = take(sizeof(int32_t) * std::max(1, n_new));
  L->o_tvis = take(sizeof(int4) * std::max(1, n_new));
  L->o_rb = take(sizeof(int2) * std::max<size_t>(1, p->row_blocks.size()));
  L->o_pbase = take(sizeof(int32_t) * p->part_base.size());
  L->o_freq = take(sizeof(double) * (d / 2));
  L->upload_bytes = off;
  // the status word is zeroed when the plan is created and never uploaded again, so that a time-out
  // recorded by an earlier launch survives aspd_plan_update until aspd_plan_status reads it
  L->o_status = take(sizeof(int32_t) * 2);
  L->o_arrive = take(p->single_launch ? sizeof(int32_t) * std::max(1, n_new) * Hkv : 0);   // right behind the status word: cleared with it
  L->cleared_end = off;
  L->o_qcs = take(sizeof(float2) * std::max(1, n_new) * (d / 2));   // filled on the device from tok_pos and inv_freq
  L->o_wso = take(sizeof(float) * L->cap_partials * G * d);
  L->o_wsml = take(sizeof(float2) * L->cap_partials * G);
  L->o_stq = take((size_t)es * std::max(1, n_new) * Hq * d);
  L->o_stk = take((size_t)es * std::max(1, n_new) * Hkv * d);
  L->o_stv = take((size_t)es * std::max(1, n_new) * Hkv * d);
  L->o_sto = take((size_t)es * std::max(1, n_new) * Hq * d);
  L->o_stp = take(sizeof(int32_t) * std::max(1, n_new));
  L->device_bytes = off;
  L->n_row_blocks = p->row_blocks.size(); L->n_part_base = p->part_base.size();
}

// Assembles the tables in the plan's page-locked buffer, sends them to the device block and fills
// the cos/sin table there.  The caller has made sure that the buffer's previous copy has completed.
static int plan_upload(aspd_plan* p, cudaStream_t s, bool clear) {
  const aspd::PlanLayout& L = p->layout;
  const int n_new = p->n_new, d = p->shape.head_dim;
  uint8_t* blob = static_cast<uint8_t*>(p->block.host);
  if (!p->items.empty()) memcpy(blob + L.o_items, p->items.data(), sizeof(DeviceItem) * p->items.size());
  fill_cta_head(p, reinterpret_cast<int4*>(blob + L.o_cta));
  if (!p->visit.empty()) memcpy(blob + L.o_visit, p->visit.data(), sizeof(int2) * p->visit.size());
  if (!p->dirty.empty()) memcpy(blob + L.o_dirty, p->dirty.data(), sizeof(int4) * p->dirty.size());
  if (n_new) {
    memcpy(blob + L.o_tpage, p->tok_page.data(), sizeof(int32_t) * n_new);
    memcpy(blob + L.o_trow, p->tok_row.data(), sizeof(int32_t) * n_new);
    memcpy(blob + L.o_tpos, p->q_pos.data(), sizeof(int32_t) * n_new);
    memcpy(blob + L.o_tvis, p->tok_vis.data(), sizeof(int4) * n_new);
  }
  if (!p->row_blocks.empty()) memcpy(blob + L.o_rb, p->row_blocks.data(), sizeof(int2) * p->row_blocks.size());
  memcpy(blob + L.o_pbase, p->part_base.data(), sizeof(int32_t) * p->part_base.size());
  double* freq = reinterpret_cast<double*>(blob + L.o_freq);
  for (int i = 0; i < d / 2; ++i) freq[i] = pow((double)p->shape.rope_theta, -2.0 * i / d);
  size_t bytes = L.upload_bytes;
  if (clear) {                                     // the status word and the counters lie right behind the tables: one copy
    memset(blob + L.o_status, 0, L.cleared_end - L.o_status);
    bytes = L.cleared_end;
  }
  if (cudaMemcpyAsync(p->device_base, blob, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return ASPD_ERR_CUDA;
  if (cudaEventRecord(p->block.upload_done, s) != cudaSuccess) return ASPD_ERR_CUDA;
  if (std::find(p->streams.begin(), p->streams.end(), s) == p->streams.end()) p->streams.push_back(s);
  // cos/sin of every new token's position (query rotation, fused append): on the device, after the upload
  return n_new > 0 ? launch_qcs(p, s) : ASPD_OK;
}

static int plan_to_device(aspd_plan* p, cudaStream_t s) {
  plan_layout(p, p->tune.updatable ? 1.25 : 1.0, &p->layout);
  const aspd::PlanLayout& L = p->layout;
  p->device_bytes = L.device_bytes;
  int rc = block_acquire(L.device_bytes, L.cleared_end, s, &p->block);
  if (rc) return rc;
  uint8_t* b8 = (uint8_t*)p->block.ptr;
  p->device_base = b8;
  p->dev.items = (const DeviceItem*)(b8 + L.o_items);
  p->dev.cta_head = (const int4*)(b8 + L.o_cta);
  p->dev.visit = (const int2*)(b8 + L.o_visit);
  p->dev.dirty = (const int4*)(b8 + L.o_dirty);
  p->dev.tok_vis = (const int4*)(b8 + L.o_tvis);
  p->dev.row_blocks = (const int2*)(b8 + L.o_rb);
  p->dev.tok_page = (const int32_t*)(b8 + L.o_tpage);
  p->dev.tok_row = (const int32_t*)(b8 + L.o_trow);
  p->dev.tok_pos = (const int32_t*)(b8 + L.o_tpos);
  p->dev.q_cs = (const float2*)(b8 + L.o_qcs);
  p->dev.part_base = (const int32_t*)(b8 + L.o_pbase);
  p->dev.inv_freq = (const double*)(b8 + L.o_freq);
  p->dev.status = (int32_t*)(b8 + L.o_status);
  p->dev.work_counter = p->dev.status + 1;
  p->dev.arrive = (int32_t*)(b8 + L.o_arrive);
  p->dev.ws_o = (float*)(b8 + L.o_wso);
  p->dev.ws_ml = (float2*)(b8 + L.o_wsml);
  p->dev.st_q = b8 + L.o_stq; p->dev.st_k = b8 + L.o_stk; p->dev.st_v = b8 + L.o_stv; p->dev.st_out = b8 + L.o_sto;
  p->dev.st_pos = (int32_t*)(b8 + L.o_stp);
  p->dev.pool_limit = (int32_t)std::min<int64_t>(p->n_pool_pages, INT32_MAX);
  rc = plan_upload(p, s, true);
  if (rc) { block_free(p->block); p->device_base = nullptr; }
  return rc;
}

int aspd_plan_update(aspd_plan_t* p, const aspd_request_t* req, const aspd_branch_t* br, const int32_t* page_ids, int n_req,
                     const int32_t* q_pos, void* stream) {
  if (!p || p->host_only || !p->device_base) return ASPD_ERR_INVALID_ARG;
  aspd_tuning_t tune = p->tune;
  tune.host_only = 1;
  aspd_plan* t = nullptr;
  int rc = plan_create_impl(&p->shape, req, br, page_ids, n_req, p->n_pool_pages, p->mode, q_pos, &tune, nullptr, p, false, &t);
  if (rc) return rc;
  const aspd::PlanLayout& L = p->layout;
  if (t->n_new != p->n_new || t->n_ctas != p->n_ctas || t->base_ctas != p->base_ctas || t->kernel != p->kernel || t->wide != p->wide || t->dealt != p->dealt ||
      t->fuse_append != p->fuse_append || t->shared_mask != p->shared_mask || t->single_launch != p->single_launch || t->m64 != p->m64 || (p->dec && padded_rows(t->max_rows) != padded_rows(p->max_rows)) || t->kernel != ASPD_KERNEL_MMA ||
      t->row_blocks.size() != L.n_row_blocks || t->part_base.size() != L.n_part_base) {
    delete t;
    return ASPD_ERR_UNSUPPORTED;
  }
  if (t->items.size() > L.cap_items || t->visit.size() > L.cap_visit || t->dirty.size() > L.cap_dirty ||
      (p->wide != 2 && (size_t)t->n_partials > L.cap_partials)) {
    delete t;
    return ASPD_ERR_TOO_LARGE;
  }
  // the page-locked buffer is written again: its previous copy must be through
  if (cudaEventSynchronize(p->block.upload_done) != cudaSuccess) { delete t; return ASPD_ERR_CUDA; }
  p->n_req = t->n_req; p->n_items = t->n_items; p->n_partials = t->n_partials; p->n_row_blocks = t->n_row_blocks; p->max_parts = t->max_parts;
  p->kv_tokens_read = t->kv_tokens_read; p->algorithmic_bytes = t->algorithmic_bytes;
  p->items.swap(t->items); p->visit.swap(t->visit); p->tok_vis.swap(t->tok_vis); p->cta_item0.swap(t->cta_item0);
  p->part_base.swap(t->part_base); p->q_pos.swap(t->q_pos); p->row_blocks.swap(t->row_blocks);
  p->tok_page.swap(t->tok_page); p->tok_row.swap(t->tok_row); p->cta_dirty0.swap(t->cta_dirty0); p->dirty.swap(t->dirty);
  delete t;
  return plan_upload(p, (cudaStream_t)stream, false);
}

int aspd_plan_destroy(aspd_plan_t* plan) {
  if (!plan) return ASPD_OK;
  int rc = ASPD_OK;
  if (plan->device_base) rc = block_release(plan->block, plan->streams);
  delete plan;
  return rc;
}

int aspd_release_cached_memory(void) { return block_cache_clear(); }

int aspd_plan_info(const aspd_plan_t* p, aspd_plan_info_t* info) {
  if (!p || !info) return ASPD_ERR_INVALID_ARG;
  info->n_new = p->n_new; info->n_items = p->n_items; info->n_partials = p->n_partials;
  info->n_stream_pages = (int32_t)p->visit.size(); info->kernel = p->kernel;
  info->chunk_tokens = p->chunk_tokens; info->n_ctas = p->n_ctas; info->fused_append = (p->kernel == ASPD_KERNEL_MMA && p->fuse_append) ? 1 : 0;
  info->direct_output = attn_mma_direct(p) ? 1 : 0; info->max_rows_per_item = p->wide ? p->wide * kMaxRowsWide : kMaxRowsPerItem;
  info->dealt = p->dealt; info->single_launch = p->single_launch;
  info->mma_m = p->kernel == ASPD_KERNEL_MMA ? (p->m64 == 1 ? 64 : p->m64 == 2 ? 96 : 128) : 0;
  info->patch_tiles = (info->fused_append && p->patch_tiles && !p->dec && p->m64 != 1 && !p->single_launch) ? 1 : 0;
  info->workspace_bytes = (int64_t)p->device_bytes;
  info->kv_tokens_read = p->kv_tokens_read; info->algorithmic_bytes = p->algorithmic_bytes;
  return ASPD_OK;
}

int aspd_plan_items(const aspd_plan_t* p, aspd_item_t* items, int max_items) {
  if (!p || (max_items > 0 && !items) || max_items < 0) return ASPD_ERR_INVALID_ARG;
  int n = std::min(max_items, p->n_items);
  static_assert(sizeof(aspd_item_t) == sizeof(DeviceItem) && sizeof(DeviceItem) == 40, "item layouts must match");
  if (n) memcpy(items, p->items.data(), sizeof(DeviceItem) * n);
  return p->n_items;
}

int aspd_plan_cta_ranges(const aspd_plan_t* p, int32_t* first, int max_entries) {
  if (!p || max_entries < 0 || (max_entries > 0 && !first)) return ASPD_ERR_INVALID_ARG;
  const int n = std::min<int>(max_entries, (int)p->cta_item0.size());
  for (int i = 0; i < n; ++i) first[i] = p->cta_item0[i];
  return p->n_ctas;
}

int aspd_plan_stream_pages(const aspd_plan_t* p, int32_t* page_ids, int32_t* n_valid, int max_pages) {
  if (!p || max_pages < 0 || (max_pages > 0 && (!page_ids || !n_valid))) return ASPD_ERR_INVALID_ARG;
  const int n = std::min<int>(max_pages, (int)p->visit.size());
  for (int i = 0; i < n; ++i) { page_ids[i] = p->visit[i].x; n_valid[i] = p->visit[i].y & 255; }
  return (int)p->visit.size();
}

int aspd_plan_token_ranges(const aspd_plan_t* p, int32_t* pe, int32_t* lo, int32_t* hi, int max_tokens) {
  if (!p || max_tokens < 0 || (max_tokens > 0 && (!pe || !lo || !hi))) return ASPD_ERR_INVALID_ARG;
  const int n = std::min<int>(max_tokens, (int)p->tok_vis.size());
  for (int i = 0; i < n; ++i) { pe[i] = p->tok_vis[i].x; lo[i] = p->tok_vis[i].y; hi[i] = p->tok_vis[i].z; }
  return (int)p->tok_vis.size();
}

int aspd_plan_shared_mask_tables(const aspd_plan_t* p, int32_t* below, int32_t* page_in_branch) {
  if (!p || !p->shared_mask || !below || !page_in_branch) return ASPD_ERR_INVALID_ARG;
  for (size_t i = 0; i < p->tok_vis.size(); ++i) below[i] = p->tok_vis[i].w;
  for (size_t i = 0; i < p->visit.size(); ++i) page_in_branch[i] = p->visit[i].y >> 13;
  return ASPD_OK;
}

int aspd_plan_status(aspd_plan_t* p, void* stream) {
  if (!p || p->host_only) return ASPD_ERR_INVALID_ARG;
  int32_t st = 0;
  if (cudaMemcpyAsync(&st, p->dev.status, sizeof(st), cudaMemcpyDeviceToHost, (cudaStream_t)stream) != cudaSuccess)
    return ASPD_ERR_CUDA;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return ASPD_ERR_CUDA;
  return st;
}

int aspd_kv_append(aspd_plan_t* p, const void* k_new, const void* v_new, const int32_t* pos, void* k_pool,
                   void* v_pool, void* stream) {
  if (!p || p->host_only) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!k_new || !v_new || !pos || !k_pool || !v_pool || misaligned16(k_new, v_new, k_pool, v_pool)) return ASPD_ERR_INVALID_ARG;
  note_stream(p, stream);
  return launch_append(p, k_new, v_new, pos, k_pool, v_pool, (cudaStream_t)stream);
}

int aspd_attn_partials(aspd_plan_t* p, const void* q, const void* k_pool, const void* v_pool, void* stream) {
  if (!p || p->host_only) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!q || !k_pool || !v_pool || misaligned16(q, k_pool, v_pool)) return ASPD_ERR_INVALID_ARG;
  if (p->wide == 2) return ASPD_ERR_UNSUPPORTED;       // the two-tile variant only writes final outputs
  cudaStream_t s = (cudaStream_t)stream;
  note_stream(p, stream);
  return p->kernel == ASPD_KERNEL_MMA ? launch_attn_mma(p, q, k_pool, v_pool, nullptr, s)
                                      : launch_attn_generic(p, q, nullptr, nullptr, k_pool, v_pool, s);
}

int aspd_step_partials(aspd_plan_t* p, const void* q, const void* k_new, const void* v_new, void* k_pool, void* v_pool,
                       void* stream) {
  if (!p || p->host_only) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!q || !k_new || !v_new || !k_pool || !v_pool || misaligned16(q, k_new, v_new, k_pool, v_pool)) return ASPD_ERR_INVALID_ARG;
  if (!(p->kernel == ASPD_KERNEL_MMA && p->fuse_append) || attn_mma_direct(p)) return ASPD_ERR_UNSUPPORTED;
  note_stream(p, stream);
  return launch_attn_mma_step(p, q, k_new, v_new, k_pool, v_pool, nullptr, (cudaStream_t)stream);
}

int aspd_attn_combine(aspd_plan_t* p, void* out, void* stream) {
  if (!p || p->host_only) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!out || misaligned16(out)) return ASPD_ERR_INVALID_ARG;
  note_stream(p, stream);
  return launch_combine(p, out, (cudaStream_t)stream);
}

static int run_attn(aspd_plan_t* p, int mode, const void* q, const void* k_pool, const void* v_pool, void* out,
                    void* stream) {
  if (!p || p->host_only || p->mode != mode) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!q || !k_pool || !v_pool || !out || misaligned16(q, k_pool, v_pool, out)) return ASPD_ERR_INVALID_ARG;
  note_stream(p, stream);
  // a plan with one item per (token, KV head) needs no records: the kernel normalises and writes the output;
  // a single-launch plan's kernel merges its records itself
  if (attn_mma_writes_output(p)) return launch_attn_mma(p, q, k_pool, v_pool, out, (cudaStream_t)stream);
  int rc = aspd_attn_partials(p, q, k_pool, v_pool, stream);
  if (rc) return rc;
  return aspd_attn_combine(p, out, stream);
}

int aspd_branch_attn(aspd_plan_t* p, const void* q, const void* k_pool, const void* v_pool, void* out, void* stream) {
  return run_attn(p, ASPD_MODE_BRANCH, q, k_pool, v_pool, out, stream);
}

int aspd_serial_attn(aspd_plan_t* p, const void* q, const void* k_pool, const void* v_pool, void* out, void* stream) {
  return run_attn(p, ASPD_MODE_SERIAL, q, k_pool, v_pool, out, stream);
}

static int run_step(aspd_plan_t* p, int mode, const void* q, const void* k_new, const void* v_new, void* k_pool,
                    void* v_pool, void* out, void* stream) {
  if (!p || p->host_only || p->mode != mode) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!q || !k_new || !v_new || !k_pool || !v_pool || !out || misaligned16(q, k_new, v_new, k_pool, v_pool, out)) return ASPD_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  note_stream(p, stream);
  int rc;
  if (p->kernel == ASPD_KERNEL_MMA && p->fuse_append) {
    rc = launch_attn_mma_step(p, q, k_new, v_new, k_pool, v_pool, out, s);
  } else if (p->kernel == ASPD_KERNEL_MMA) {
    rc = launch_append(p, k_new, v_new, p->dev.tok_pos, k_pool, v_pool, s);
    if (rc == ASPD_OK) rc = launch_attn_mma(p, q, k_pool, v_pool, out, s);
  } else if (p->fuse_append) {
    rc = launch_attn_generic(p, q, k_new, v_new, k_pool, v_pool, s);
  } else {
    rc = launch_append(p, k_new, v_new, p->dev.tok_pos, k_pool, v_pool, s);
    if (rc == ASPD_OK) rc = launch_attn_generic(p, q, nullptr, nullptr, k_pool, v_pool, s);
  }
  if (rc || attn_mma_writes_output(p)) return rc;
  return launch_combine(p, out, s);
}

int aspd_branch_step(aspd_plan_t* p, const void* q, const void* k_new, const void* v_new, void* k_pool, void* v_pool,
                     void* out, void* stream) {
  return run_step(p, ASPD_MODE_BRANCH, q, k_new, v_new, k_pool, v_pool, out, stream);
}

int aspd_serial_step(aspd_plan_t* p, const void* q, const void* k_new, const void* v_new, void* k_pool, void* v_pool,
                     void* out, void* stream) {
  return run_step(p, ASPD_MODE_SERIAL, q, k_new, v_new, k_pool, v_pool, out, stream);
}

int aspd_step_host_async(aspd_plan_t* p, const void* q, const void* k_new, const void* v_new, const int32_t* pos,
                         void* k_pool, void* v_pool, void* out, void* stream) {
  if (!p || p->host_only) return ASPD_ERR_INVALID_ARG;
  if (p->n_new == 0) return ASPD_OK;
  if (!q || !k_new || !v_new || !pos || !k_pool || !v_pool || !out || misaligned16(k_pool, v_pool)) return ASPD_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  note_stream(p, stream);
  const aspd_shape_t& sh = p->shape;
  const size_t es = esize_of(sh.dtype);
  const size_t qb = es * p->n_new * sh.n_q_heads * sh.head_dim, kb = es * p->n_new * sh.n_kv_heads * sh.head_dim;
  // The staging areas of q, k_new and v_new lie back to back in the plan's block; when the caller's
  // three buffers do too (one packed host buffer), one copy moves them all.
  const char* qh = static_cast<const char*>(q);
  const bool packed = static_cast<const char*>(k_new) == qh + qb && static_cast<const char*>(v_new) == qh + qb + kb &&
                      static_cast<char*>(p->dev.st_k) == static_cast<char*>(p->dev.st_q) + qb &&
                      static_cast<char*>(p->dev.st_v) == static_cast<char*>(p->dev.st_q) + qb + kb;
  if (packed) {
    if (cudaMemcpyAsync(p->dev.st_q, q, qb + 2 * kb, cudaMemcpyHostToDevice, s) != cudaSuccess) return ASPD_ERR_CUDA;
  } else if (cudaMemcpyAsync(p->dev.st_q, q, qb, cudaMemcpyHostToDevice, s) != cudaSuccess ||
             cudaMemcpyAsync(p->dev.st_k, k_new, kb, cudaMemcpyHostToDevice, s) != cudaSuccess ||
             cudaMemcpyAsync(p->dev.st_v, v_new, kb, cudaMemcpyHostToDevice, s) != cudaSuccess) {
    return ASPD_ERR_CUDA;
  }
  int rc;
  if (memcmp(pos, p->q_pos.data(), sizeof(int32_t) * p->n_new) == 0) {
    // the caller's position IDs are the plan's (the usual case): they are on the device already,
    // and the step may write the new rows inside the attention pass
    rc = run_step(p, p->mode, p->dev.st_q, p->dev.st_k, p->dev.st_v, k_pool, v_pool, p->dev.st_out, stream);
  } else {
    if (cudaMemcpyAsync(p->dev.st_pos, pos, sizeof(int32_t) * p->n_new, cudaMemcpyHostToDevice, s) != cudaSuccess) return ASPD_ERR_CUDA;
    rc = launch_append(p, p->dev.st_k, p->dev.st_v, p->dev.st_pos, k_pool, v_pool, s);
    if (rc == ASPD_OK) rc = run_attn(p, p->mode, p->dev.st_q, k_pool, v_pool, p->dev.st_out, stream);
  }
  if (rc) return rc;
  if (cudaMemcpyAsync(out, p->dev.st_out, qb, cudaMemcpyDeviceToHost, s) != cudaSuccess) return ASPD_ERR_CUDA;
  return ASPD_OK;
}

int aspd_step_host(aspd_plan_t* p, const void* q, const void* k_new, const void* v_new, const int32_t* pos,
                   void* k_pool, void* v_pool, void* out, void* stream) {
  const int rc = aspd_step_host_async(p, q, k_new, v_new, pos, k_pool, v_pool, out, stream);
  if (rc) return rc;
  if (p->n_new > 0 && cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return ASPD_ERR_CUDA;
  return ASPD_OK;
}

int aspd_k_rerotate(const aspd_shape_t* shape, void* k_pool, const int32_t* pages, const int32_t* rows,
                    const int32_t* delta, int n, void* stream) {
  int rc = check_shape(shape);
  if (rc) return rc;
  if (n < 0) return ASPD_ERR_INVALID_ARG;
  if (n == 0) return ASPD_OK;
  if (!k_pool || !pages || !rows || !delta || misaligned16(k_pool)) return ASPD_ERR_INVALID_ARG;
  return launch_rerotate(shape, k_pool, pages, rows, delta, n, (cudaStream_t)stream);
}

static int check_ranges(const int32_t* ranges, int n_ranges) {
  for (int i = 0; i < n_ranges; ++i) {
    const int32_t* g = ranges + 4 * (size_t)i;
    if (g[0] < 0 || g[1] < 0 || g[2] < 0 || (long)g[1] + g[2] > INT32_MAX) return ASPD_ERR_BAD_DESCRIPTOR;
  }
  return ASPD_OK;
}

int aspd_k_rerotate_ranges(const aspd_shape_t* shape, void* k_pool, const int32_t* page_table, const int32_t* ranges, int n_ranges,
                           void* stream) {
  return aspd_k_rerotate_ranges_layers(shape, &k_pool, 1, page_table, ranges, n_ranges, stream);
}

int aspd_k_rerotate_ranges_layers(const aspd_shape_t* shape, void* const* k_pools, int n_layers, const int32_t* page_table,
                                  const int32_t* ranges, int n_ranges, void* stream) {
  int rc = check_shape(shape);
  if (rc) return rc;
  if (n_ranges < 0 || n_layers < 0) return ASPD_ERR_INVALID_ARG;
  if (n_ranges == 0 || n_layers == 0) return ASPD_OK;
  if (!k_pools || !page_table || !ranges) return ASPD_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l)
    if (!k_pools[l] || misaligned16(k_pools[l])) return ASPD_ERR_INVALID_ARG;
  if ((rc = check_ranges(ranges, n_ranges))) return rc;
  return launch_rerotate_ranges(shape, k_pools, n_layers, page_table, ranges, n_ranges, (cudaStream_t)stream);
}

int aspd_debug_pool_limit(aspd_plan_t* p, int64_t n_pages) {
  if (!p || p->host_only || n_pages < 0 || n_pages > p->n_pool_pages) return ASPD_ERR_INVALID_ARG;
#ifdef ASPD_DEBUG_BOUNDS
  p->dev.pool_limit = (int32_t)std::min<int64_t>(n_pages, INT32_MAX);
  return ASPD_OK;
#else
  return ASPD_ERR_UNSUPPORTED;
#endif
}

int aspd_debug_profile(void* device_buf, int cta) {
  if (cta < 0) return ASPD_ERR_INVALID_ARG;
  return set_profile_buffer((long long*)device_buf, cta);
}

int aspd_debug_bounded_wait(int64_t limit_cycles, int32_t* status_out, void* stream) {
  if (!status_out || limit_cycles < 0 || limit_cycles > 4000000000LL) return ASPD_ERR_INVALID_ARG;
  int32_t* dev = nullptr;
  if (cudaMalloc(&dev, sizeof(int32_t)) != cudaSuccess) return ASPD_ERR_NOMEM;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = launch_wait_probe(limit_cycles, dev, s);
  if (rc == ASPD_OK && (cudaMemcpyAsync(status_out, dev, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                        cudaStreamSynchronize(s) != cudaSuccess))
    rc = ASPD_ERR_CUDA;
  cudaFree(dev);
  return rc;
}

int aspd_debug_read_token(const aspd_shape_t* shape, const void* pool, int64_t page, int row, int kv_head, float* out,
                          void* stream) {
  int rc = check_shape(shape);
  if (rc) return rc;
  if (!pool || !out || page < 0 || row < 0 || row >= shape->page_size || kv_head < 0 || kv_head >= shape->n_kv_heads)
    return ASPD_ERR_INVALID_ARG;
  float* tmp = nullptr;
  if (cudaMalloc(&tmp, sizeof(float) * shape->head_dim) != cudaSuccess) return ASPD_ERR_NOMEM;
  cudaStream_t s = (cudaStream_t)stream;
  rc = launch_read_token(shape, pool, page, row, kv_head, tmp, s);
  if (rc == ASPD_OK && (cudaMemcpyAsync(out, tmp, sizeof(float) * shape->head_dim, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                        cudaStreamSynchronize(s) != cudaSuccess))
    rc = ASPD_ERR_CUDA;
  cudaFree(tmp);
  return rc;
}

}  // extern "C"

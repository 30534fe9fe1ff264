// Small kernels: RoPE + paged append (a3), the generic CUDA-core attention kernel (any
// supported dtype / head_dim / page_size), the log-sum-exp combine (a7) and a debug reader.
#include "aspd_internal.cuh"
#include "aspd_combine.cuh"

namespace aspd {

namespace {

constexpr float kLog2e = 1.4426950408889634f;

template <typename T> __device__ inline float to_f32(T x);
template <> __device__ inline float to_f32<float>(float x) { return x; }
template <> __device__ inline float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ inline T from_f32(float x);
template <> __device__ inline float from_f32<float>(float x) { return x; }
template <> __device__ inline __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// ------------------------------------------------------------------------------- append
// A thread owns one 16-byte chunk of the first half of a (new token, KV head) row and its partner
// chunk in the second half (the pairs (i, i + d/2)): it rotates that chunk pair of K and copies
// that chunk pair of V.
constexpr int kAppendThreads = 128;
template <typename T>
__global__ void __launch_bounds__(kAppendThreads)
append_kernel(const T* __restrict__ k_new, const T* __restrict__ v_new, const int32_t* __restrict__ pos, const float2* __restrict__ cs_table,
              const int32_t* __restrict__ tok_page, const int32_t* __restrict__ tok_row,
              const double* __restrict__ inv_freq, T* __restrict__ k_pool, T* __restrict__ v_pool,
              int n_new, int n_kv_heads, int head_dim, int page_size, PlanDevice pd) {
  constexpr int VEC = 16 / sizeof(T);
  pdl_launch_dependents();
  const int half = head_dim / 2, chunks = half / VEC;
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long t = gid / (chunks * n_kv_heads);
  const int h = (int)(gid / chunks % n_kv_heads), c = (int)(gid % chunks);
  const int page = t < n_new ? tok_page[t] : 0, row = t < n_new ? tok_row[t] : 0;   // plan data: may be read before the dependency wait
  pdl_wait();
  if (t >= n_new || !bounds_ok(pd, page, row, page_size)) return;
  float sn[VEC], cs[VEC];
  if (cs_table != nullptr) {                       // the plan's own positions: their sines and cosines are there already
    const float4* w = reinterpret_cast<const float4*>(cs_table + t * half + c * VEC);
#pragma unroll
    for (int j = 0; j < VEC; j += 2) {
      const float4 x = w[j / 2];
      cs[j] = x.x; sn[j] = x.y; cs[j + 1] = x.z; sn[j + 1] = x.w;
    }
  } else {
    // angle reduced to [-pi, pi] in fp64, then fp32 sincos: the error stays near 1e-7 rad
    // however large the position is
    const double p = (double)pos[t];
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      double a = p * inv_freq[c * VEC + j];
      a -= rint(a * 0.15915494309189535) * 6.283185307179586;
      sincosf((float)a, &sn[j], &cs[j]);
    }
  }
  const uint32_t rb = head_dim * sizeof(T);
  const size_t tb = tile_bytes(page_size, head_dim, sizeof(T));
  const size_t tile0 = (size_t)page * n_kv_heads * tb;
  const uint32_t o0 = tile_offset(row, c * 16, rb), o1 = tile_offset(row, half * sizeof(T) + c * 16, rb);
  {
    const size_t src = ((size_t)t * n_kv_heads + h) * head_dim;
    uint4 u0 = *reinterpret_cast<const uint4*>(k_new + src + c * VEC);
    uint4 u1 = *reinterpret_cast<const uint4*>(k_new + src + half + c * VEC);
    const uint4 w0 = *reinterpret_cast<const uint4*>(v_new + src + c * VEC);
    const uint4 w1 = *reinterpret_cast<const uint4*>(v_new + src + half + c * VEC);
    T* x0 = reinterpret_cast<T*>(&u0);
    T* x1 = reinterpret_cast<T*>(&u1);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const float a = to_f32(x0[j]), b = to_f32(x1[j]);
      x0[j] = from_f32<T>(a * cs[j] - b * sn[j]);
      x1[j] = from_f32<T>(b * cs[j] + a * sn[j]);
    }
    char* kp = reinterpret_cast<char*>(k_pool) + tile0 + h * tb;
    char* vp = reinterpret_cast<char*>(v_pool) + tile0 + h * tb;
    *reinterpret_cast<uint4*>(kp + o0) = u0;
    *reinterpret_cast<uint4*>(kp + o1) = u1;
    *reinterpret_cast<uint4*>(vp + o0) = w0;
    *reinterpret_cast<uint4*>(vp + o1) = w1;
  }
}

// ------------------------------------------------------------------- cos/sin table of a plan
// q_cs[t][i] = (cos, sin)(pos[t] * inv_freq[i]): the rotation of new token t's query (and, in the
// fused step, of its key).  Same arithmetic as the append kernel: angle reduced in fp64, fp32 sincos.
__global__ void qcs_kernel(const int32_t* __restrict__ pos, const double* __restrict__ inv_freq, float2* __restrict__ q_cs,
                           int n_new, int half) {
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long)n_new * half) return;
  const int t = (int)(gid / half), i = (int)(gid % half);
  double a = (double)pos[t] * inv_freq[i];
  a -= rint(a * 0.15915494309189535) * 6.283185307179586;
  float sn, cs;
  sincosf((float)a, &sn, &cs);
  q_cs[gid] = make_float2(cs, sn);
}

// --------------------------------------------------------------------------- re-rotation
// K'(pos + delta) = RoPE(K'(pos), delta): rotations compose, so cached keys can be moved to new
// position IDs in place, reading and writing each key once, instead of being re-encoded from
// the raw keys.  A thread owns one 16-byte chunk of the first half of a token's row and its
// partner chunk in the second half (the pairs (i, i + d/2)), computes the chunk's sines and
// cosines once and applies them to every KV head of the token.
constexpr int kRerotateThreads = 256;
struct InvFreq {          // theta^(-2i/d), computed by the host in double; by value in the launch
  double f[64];
};
// One thread's share of a token: the 16-byte chunk at o0 and its partner at o1 in every KV head's
// tile.  The loads of four heads are issued before the first store (the stores go to the same pool,
// so the compiler would otherwise keep every head's loads behind the previous head's stores).
template <typename T>
__device__ __forceinline__ void rotate_token_heads(char* tile, size_t tb, uint32_t o0, uint32_t o1, int n_kv_heads,
                                                   const float (&sn)[16 / sizeof(T)], const float (&cs)[16 / sizeof(T)]) {
  constexpr int VEC = 16 / sizeof(T);
  for (int h0 = 0; h0 < n_kv_heads; h0 += 4) {
    uint4 u0[4], u1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int h = min(h0 + k, n_kv_heads - 1);
      u0[k] = *reinterpret_cast<const uint4*>(tile + h * tb + o0);
      u1[k] = *reinterpret_cast<const uint4*>(tile + h * tb + o1);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (h0 + k >= n_kv_heads) break;
      T* x0 = reinterpret_cast<T*>(&u0[k]);
      T* x1 = reinterpret_cast<T*>(&u1[k]);
#pragma unroll
      for (int j = 0; j < VEC; ++j) {
        const float a = to_f32(x0[j]), b = to_f32(x1[j]);
        x0[j] = from_f32<T>(a * cs[j] - b * sn[j]);
        x1[j] = from_f32<T>(b * cs[j] + a * sn[j]);
      }
      *reinterpret_cast<uint4*>(tile + (h0 + k) * tb + o0) = u0[k];
      *reinterpret_cast<uint4*>(tile + (h0 + k) * tb + o1) = u1[k];
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kRerotateThreads)
rerotate_kernel(T* __restrict__ k_pool, const int32_t* __restrict__ pages, const int32_t* __restrict__ rows,
                const int32_t* __restrict__ delta, const InvFreq table, int n, int n_kv_heads, int head_dim, int page_size) {
  constexpr int VEC = 16 / sizeof(T);
  __shared__ double inv_freq[64];
  pdl_launch_dependents();
  const int half = head_dim / 2, chunks = half / VEC;
  if (threadIdx.x < half) inv_freq[threadIdx.x] = table.f[threadIdx.x];
  __syncthreads();
  pdl_wait();
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long t = gid / chunks;
  const int c = (int)(gid % chunks);
  if (t >= n) return;
  float sn[VEC], cs[VEC];
  const double dl = (double)delta[t];
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    double a = dl * inv_freq[c * VEC + j];
    a -= rint(a * 0.15915494309189535) * 6.283185307179586;
    sincosf((float)a, &sn[j], &cs[j]);
  }
  const uint32_t rb = head_dim * sizeof(T);
  const size_t tb = tile_bytes(page_size, head_dim, sizeof(T));
  char* tile = reinterpret_cast<char*>(k_pool) + (size_t)pages[t] * n_kv_heads * tb;
  const uint32_t o0 = tile_offset(rows[t], c * 16, rb), o1 = tile_offset(rows[t], half * sizeof(T) + c * 16, rb);
  rotate_token_heads<T>(tile, tb, o0, o1, n_kv_heads, sn, cs);
}

// The same with the tokens given as ranges of logical slots: range i covers `count` consecutive
// slots from `first` of the request whose page table starts at page_table[base], all moved by the
// same `delta` (a finished branch that is renumbered moves as a whole).  The kernel derives page
// and row itself, so no per-token index arrays are read: a block takes one page of one range.
constexpr int kMaxRanges = 512;         // ranges per launch (they travel in the launch parameters, about 10 KB)
struct RerotateRanges {
  int n;
  int unit0[kMaxRanges + 1];            // first page unit of range i (prefix sum of the pages each range touches)
  int4 r[kMaxRanges];                   // (page-table base, first slot, count, delta)
};
constexpr int kMaxLayerPools = 64;      // K pools (layers) per launch: grid.y, their addresses in the launch parameters
struct PoolList {
  void* p[kMaxLayerPools];
};
template <typename T>
__global__ void __launch_bounds__(512)
rerotate_ranges_kernel(const PoolList pools, const int32_t* __restrict__ page_table, const RerotateRanges rr, const InvFreq table,
                       int n_kv_heads, int head_dim, int page_size) {
  T* __restrict__ k_pool = static_cast<T*>(pools.p[blockIdx.y]);   // the layers share the page tables, so the same pages move in each
  constexpr int VEC = 16 / sizeof(T);
  __shared__ float2 cs_sm[64];          // (cos, sin) of the range's delta for every element pair: the same for all tokens of the page
  pdl_launch_dependents();
  const int half = head_dim / 2, chunks = half / VEC;
  const int u = blockIdx.x;
  int lo = 0, hi = rr.n - 1;            // the range this block's page belongs to: last i with unit0[i] <= u
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (rr.unit0[mid] <= u) lo = mid; else hi = mid - 1;
  }
  const int4 rg = rr.r[lo];
  const int page = rg.y / page_size + (u - rr.unit0[lo]);           // index of the page in the request's table
  const int tok = threadIdx.x / chunks, c = threadIdx.x % chunks, slot = page * page_size + tok;
  const bool active = tok < page_size && slot >= rg.y && slot < rg.y + rg.z;
  // the sines and cosines depend on the launch parameters only: taken before the dependency wait,
  // i.e. while the previous kernel of the stream is still running
  if ((int)threadIdx.x < half) {
    double a = (double)rg.w * table.f[threadIdx.x];
    a -= rint(a * 0.15915494309189535) * 6.283185307179586;
    float sn1, cs1;
    sincosf((float)a, &sn1, &cs1);
    cs_sm[threadIdx.x] = make_float2(cs1, sn1);
  }
  __syncthreads();
  pdl_wait();
  const uint32_t rb = head_dim * sizeof(T);
  const size_t tb = tile_bytes(page_size, head_dim, sizeof(T));
  char* tile = reinterpret_cast<char*>(k_pool) + (size_t)page_table[rg.x + page] * n_kv_heads * tb;
  const uint32_t o0 = tile_offset(tok, c * 16, rb), o1 = tile_offset(tok, half * sizeof(T) + c * 16, rb);
  uint4 u0[4], u1[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    u0[k] = make_uint4(0, 0, 0, 0); u1[k] = u0[k];
    if (active) {
      const int h = min(k, n_kv_heads - 1);
      u0[k] = *reinterpret_cast<const uint4*>(tile + h * tb + o0);
      u1[k] = *reinterpret_cast<const uint4*>(tile + h * tb + o1);
    }
  }
  if (!active) return;
  float sn[VEC], cs[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) { cs[j] = cs_sm[c * VEC + j].x; sn[j] = cs_sm[c * VEC + j].y; }
  for (int h0 = 0; h0 < n_kv_heads; h0 += 4) {
    if (h0 > 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int h = min(h0 + k, n_kv_heads - 1);
        u0[k] = *reinterpret_cast<const uint4*>(tile + h * tb + o0);
        u1[k] = *reinterpret_cast<const uint4*>(tile + h * tb + o1);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (h0 + k >= n_kv_heads) break;
      T* x0 = reinterpret_cast<T*>(&u0[k]);
      T* x1 = reinterpret_cast<T*>(&u1[k]);
#pragma unroll
      for (int j = 0; j < VEC; ++j) {
        const float a = to_f32(x0[j]), b = to_f32(x1[j]);
        x0[j] = from_f32<T>(a * cs[j] - b * sn[j]);
        x1[j] = from_f32<T>(b * cs[j] + a * sn[j]);
      }
      *reinterpret_cast<uint4*>(tile + (h0 + k) * tb + o0) = u0[k];
      *reinterpret_cast<uint4*>(tile + (h0 + k) * tb + o1) = u1[k];
    }
  }
}

// ------------------------------------------------------------------- generic attention
// CUDA-core split-K pass for every dtype, head_dim and page size (fp32 steps, and KERNEL_GENERIC plans).
// A CTA walks its items 32 keys at a time: the pages of the next 32 keys are on their way to shared memory
// (cp.async, the cache's swizzled tile image as it lies) while these are scored.  A warp owns RPW query rows from
// the score to the record -- lane j scores key j against all of them (the key's 16-byte chunk is read once, the
// queries are broadcast), then each lane owns D / 32 output elements -- so that inside a chunk nothing
// crosses warps.  Bound by latency on the steps it serves: 3 branches over 256 tokens (fp32, 4 heads of 64) are
// 10 CTAs of 32 keys, 7.4 us a step (append, this, combine) in a graph; 5 CTAs of 64 keys 10.2; the kernel before, a
// block of four warps to 128 keys, each warp walking one row's keys through memory at a time, 153.7.
// A key of weight 0 for a row is left out of it (its V row may hold Inf or NaN that the row does not see); no measurable time.
constexpr int kGenThreads = 256, kGenWarps = kGenThreads / 32, kGenKeys = 32;
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool there) {   // 16 zero bytes if not there
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(there ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T, int D>
struct GenSmem {
  T k[2][kGenKeys * D], v[2][kGenKeys * D];      // two chunks of 32 keys, tile images
  float q[kMaxRowsPerItem * D];                  // rotated, scaled queries
  float p[kGenWarps][kMaxRowsPerItem / kGenWarps][kGenKeys];
  int4 vis[kMaxRowsPerItem];                     // per token of the item
};

// The 16-byte piece of this lane's D / 32 elements of row `tok` of a tile image, as floats
template <typename T, int D>
__device__ __forceinline__ void lane_elems(const T* tile, int tok, int lane, float (&x)[D / 32]) {
  const char* at = reinterpret_cast<const char*>(tile) + tile_offset(tok, lane * (D / 32) * (int)sizeof(T), D * sizeof(T));
  T e[D / 32];
  if constexpr (sizeof(e) == 16) *reinterpret_cast<uint4*>(e) = *reinterpret_cast<const uint4*>(at);
  else if constexpr (sizeof(e) == 8) *reinterpret_cast<uint2*>(e) = *reinterpret_cast<const uint2*>(at);
  else *reinterpret_cast<uint32_t*>(e) = *reinterpret_cast<const uint32_t*>(at);
#pragma unroll
  for (int i = 0; i < D / 32; ++i) x[i] = to_f32(e[i]);
}

template <typename T, int D, int RPW>
__device__ __forceinline__ void generic_item(const PlanDevice& pd, const DeviceItem& it, GenSmem<T, D>& sm, const T* __restrict__ q,
                                             const T* __restrict__ k_pool, const T* __restrict__ v_pool, int n_q_heads, int n_kv_heads,
                                             int page_size, float scale_log2) {
  constexpr int EPL = D / 32, EPC = 16 / (int)sizeof(T), RB = D * (int)sizeof(T);
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const int G = n_q_heads / n_kv_heads, n_rows = it.n_q_tok * G, ppc = kGenKeys / page_size;   // pages of a chunk (4, 2, 1)
  const int n_chunks = (it.n_pages + ppc - 1) / ppc, page_shift = 31 - __clz(page_size);
  const size_t tb = tile_bytes(page_size, D, sizeof(T));
  // lane l < ppc: entry of page l of a chunk (no valid rows behind the item's pages)
  auto entry_of = [&](int chunk) {
    int2 e = make_int2(0, 0);
    if (lane < ppc && chunk * ppc + lane < it.n_pages) {
      e = pd.visit[it.page0 + chunk * ppc + lane];
      if (!bounds_ok(pd, e.x, 0, page_size)) e = make_int2(0, 0);     // checking builds: flagged, keys left out
    }
    return e;
  };
  auto request = [&](int2 entry, int st) {
    const uint32_t kd = (uint32_t)__cvta_generic_to_shared(sm.k[st]), vd = (uint32_t)__cvta_generic_to_shared(sm.v[st]);
#pragma unroll
    for (int u = 0; u < kGenKeys * RB / 16 / kGenThreads; ++u) {
      const uint32_t b = (tid + u * kGenThreads) * 16u;
      const int pg = (int)(b / (uint32_t)tb);
      const int id = __shfl_sync(0xffffffffu, entry.x, pg), there = __shfl_sync(0xffffffffu, entry.y, pg) & 255;
      const size_t src = ((size_t)id * n_kv_heads + it.kv_head) * tb + (b - pg * (uint32_t)tb);
      cp_async16(kd + b, reinterpret_cast<const char*>(k_pool) + src, there != 0);
      cp_async16(vd + b, reinterpret_cast<const char*>(v_pool) + src, there != 0);
    }
    cp_async_commit();
  };
  int2 cur = entry_of(0), nxt = entry_of(1);
  request(cur, 0);
  // the queries, rotated at their own positions (table of the plan), scale folded in
  for (int e = tid; e < it.n_q_tok; e += kGenThreads) sm.vis[e] = pd.tok_vis[it.q_tok0 + e];
  for (int e = tid; e < n_rows * (D / 2); e += kGenThreads) {
    const int r = e / (D / 2), i = e % (D / 2), tok = it.q_tok0 + r / G;
    const T* qrow = q + ((size_t)tok * n_q_heads + it.kv_head * G + r % G) * D;
    const float2 cs = pd.q_cs[(size_t)tok * (D / 2) + i];
    const float x0 = to_f32(qrow[i]), x1 = to_f32(qrow[i + D / 2]);
    sm.q[r * D + i] = (x0 * cs.x - x1 * cs.y) * scale_log2;
    sm.q[r * D + i + D / 2] = (x1 * cs.x + x0 * cs.y) * scale_log2;
  }
  const int row0 = warp * RPW;                    // rows row0 ... row0 + RPW - 1, those below n_rows
  float m[RPW], l[RPW], acc[RPW][EPL];
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[i][e] = 0.f;
  }
  for (int ch = 0; ch < n_chunks; ++ch) {
    const int st = ch & 1;
    const int2 after = entry_of(ch + 2);
    if (ch + 1 < n_chunks) { request(nxt, st ^ 1); cp_async_wait<1>(); }
    else cp_async_wait<0>();
    __syncthreads();
    if (row0 < n_rows) {
      float s[RPW][2];                            // even and odd chunks of the dot products apart
#pragma unroll
      for (int i = 0; i < RPW; ++i) s[i][0] = s[i][1] = 0.f;
#pragma unroll (RPW < 8 ? 4 : 2)
      for (int c = 0; c < RB / 16; ++c) {
        const uint4 raw = *reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(sm.k[st]) + tile_offset(lane, c * 16, RB));
        const T* e8 = reinterpret_cast<const T*>(&raw);
        float kx[EPC];
#pragma unroll
        for (int e = 0; e < EPC; ++e) kx[e] = to_f32(e8[e]);
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
          const float4* qr = reinterpret_cast<const float4*>(sm.q + min(row0 + i, n_rows - 1) * D + c * EPC);
#pragma unroll
          for (int e = 0; e < EPC / 4; ++e) {
            const float4 w = qr[e];
            float& d = s[i][(EPC == 4 ? c : e) & 1];
            d = fmaf(w.x, kx[4 * e], d); d = fmaf(w.y, kx[4 * e + 1], d); d = fmaf(w.z, kx[4 * e + 2], d); d = fmaf(w.w, kx[4 * e + 3], d);
          }
        }
      }
      // stream keys [0, pe) and [lo, hi) are visible; under the shared mask (w > 0) also keys of other
      // branches whose offset in their branch (page index in the upper bits of the page entry) is below w
      const int ye = __shfl_sync(0xffffffffu, cur.y, lane >> page_shift), row = lane & (page_size - 1), kg = it.key0 + ch * kGenKeys + lane;
      const bool valid = row < (ye & 255);
#pragma unroll
      for (int i = 0; i < RPW; ++i) {
        const int4 vis = sm.vis[min(row0 + i, n_rows - 1) / G];
        const bool seen = valid && (kg < vis.x || (kg >= vis.y && kg < vis.z) || (ye >> 13) * page_size + row < vis.w);
        const float x = seen ? s[i][0] + s[i][1] : -INFINITY;
        float mx = x;
#pragma unroll
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float mn = fmaxf(m[i], mx), base = mn == -INFINITY ? 0.f : mn;      // no key seen so far: every weight is 0
        const float pw = exp2f(x - base), alpha = exp2f(m[i] - base);
        float ps = pw;
#pragma unroll
        for (int o = 16; o; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
        l[i] = l[i] * alpha + ps;
        m[i] = mn;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[i][e] *= alpha;
        sm.p[warp][i][lane] = pw;
      }
      __syncwarp();
#pragma unroll (RPW < 8 ? 2 : 1)
      for (int j = 0; j < kGenKeys; j += 4) {
        float v[4][EPL];
#pragma unroll
        for (int k = 0; k < 4; ++k) lane_elems<T, D>(sm.v[st], j + k, lane, v[k]);
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
          const float4 w4 = *reinterpret_cast<const float4*>(&sm.p[warp][i][j]);
          const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (w[k] != 0.f) {                    // a key that the row does not see may hold anything, Inf and NaN too
#pragma unroll
              for (int e = 0; e < EPL; ++e) acc[i][e] = fmaf(w[k], v[k][e], acc[i][e]);
            }
        }
      }
    }
    __syncthreads();                              // the chunk's buffers (and, after the last one, the queries) are free
    cur = nxt;
    nxt = after;
  }
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = row0 + i;
    if (r >= n_rows) break;
    const size_t rec = (size_t)(pd.part_base[(it.q_tok0 + r / G) * n_kv_heads + it.kv_head] + it.part_slot) * G + r % G;
    if (lane == 0) pd.ws_ml[rec] = make_float2(m[i], l[i]);
#pragma unroll
    for (int e = 0; e < EPL; ++e) pd.ws_o[rec * D + lane * EPL + e] = acc[i][e];
  }
}

// The step's new rows in pages that THIS CTA reads (fused step), K rotated with the plan's sines and cosines, V as is.
// CTAs that read the same page write identical bytes.  A thread takes a chunk pair of K and of V, as the append kernel's do.
// One launch less a step: three branches over 256 tokens (one layer, 4 heads of 64, a plan per step) 29.7 -> 27.5 us, two requests of
// 0.4 k tokens (four layers, 8 heads of 128) 57 -> 49.5.
template <typename T, int D>
__device__ __forceinline__ void generic_append(const PlanDevice& pd, const T* __restrict__ k_new, const T* __restrict__ v_new, char* k_pool, char* v_pool,
                                               int dirty0, int n_rows, int n_kv_heads, int page_size) {
  constexpr int VEC = 16 / (int)sizeof(T), HALF = D / 2, CH = HALF / VEC;
  const size_t tb = tile_bytes(page_size, D, sizeof(T));
#pragma unroll 1
  for (int e = threadIdx.x; e < n_rows * CH; e += kGenThreads) {
    const int4 d = pd.dirty[dirty0 + e / CH];      // (page, KV head, new token, row | ...)
    const int c = e % CH, row = d.w & 255;
    if (!bounds_ok(pd, d.x, row, page_size)) continue;
    const size_t src = ((size_t)d.z * n_kv_heads + d.y) * D + c * VEC;
    uint4 u0 = *reinterpret_cast<const uint4*>(k_new + src), u1 = *reinterpret_cast<const uint4*>(k_new + src + HALF);
    const uint4 w0 = *reinterpret_cast<const uint4*>(v_new + src), w1 = *reinterpret_cast<const uint4*>(v_new + src + HALF);
    const float2* cs = pd.q_cs + (size_t)d.z * HALF + c * VEC;
    T* x0 = reinterpret_cast<T*>(&u0);
    T* x1 = reinterpret_cast<T*>(&u1);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const float2 w = cs[j];
      const float a = to_f32(x0[j]), b = to_f32(x1[j]);
      x0[j] = from_f32<T>(a * w.x - b * w.y);
      x1[j] = from_f32<T>(b * w.x + a * w.y);
    }
    const size_t tile = ((size_t)d.x * n_kv_heads + d.y) * tb;
    const uint32_t o0 = tile_offset(row, c * 16, D * (int)sizeof(T)), o1 = tile_offset(row, HALF * (int)sizeof(T) + c * 16, D * (int)sizeof(T));
    *reinterpret_cast<uint4*>(k_pool + tile + o0) = u0;
    *reinterpret_cast<uint4*>(k_pool + tile + o1) = u1;
    *reinterpret_cast<uint4*>(v_pool + tile + o0) = w0;
    *reinterpret_cast<uint4*>(v_pool + tile + o1) = w1;
  }
}

// (RPW for the plan's largest row block: an instance that chose per item was 65 to 79 KB of code, and a short launch
// waits for its instructions.)
template <typename T, int D, int RPW>
__global__ void __launch_bounds__(kGenThreads, 2) attn_generic_kernel(PlanDevice pd, const T* __restrict__ q, const T* __restrict__ k_new,
                                                                      const T* __restrict__ v_new, T* k_pool, T* v_pool, int n_q_heads,
                                                                      int n_kv_heads, int page_size, float scale_log2) {
  extern __shared__ __align__(1024) uint8_t gen_smem[];
  GenSmem<T, D>& sm = *reinterpret_cast<GenSmem<T, D>*>(gen_smem);
  pdl_launch_dependents();
  const int4 head = pd.cta_head[2 * blockIdx.x], head2 = pd.cta_head[2 * blockIdx.x + 1];
  DeviceItem it = {};
  const int item_begin = uniform(head.x), item_end = uniform(head.y);
  if (item_begin < item_end) it = uniform_item(pd.items[item_begin]);
  pdl_wait();
  if (k_new != nullptr && head2.y > 0) {
    generic_append<T, D>(pd, k_new, v_new, reinterpret_cast<char*>(k_pool), reinterpret_cast<char*>(v_pool), head2.x, head2.y, n_kv_heads, page_size);
    __syncthreads();                              // before the CTA asks for those pages
  }
  for (int idx = item_begin; idx < item_end; ++idx) {
    if (idx > item_begin) it = uniform_item(pd.items[idx]);
    generic_item<T, D, RPW>(pd, it, sm, q, k_pool, v_pool, n_q_heads, n_kv_heads, page_size, scale_log2);
  }
}

// ------------------------------------------------------------------------------ combine
// One warp per (new token, query head): merge the partial records of (token, KV head) by
// log-sum-exp, up to 64 of them against one maximum (combine_row).  Where the records lie is plan
// data and is read before the dependency wait.
// FLAT: the rows of all tokens are numbered through, four to a block; otherwise a token's heads have blocks of their own, a
// grid of (tokens, heads / 4).  FLAT where four does not divide the heads: every fourth block of 14 heads had two idle
// warps, and eight requests' 152 blocks did not fit the chip at a time, which 133 do (24 layers 356 and 344 us).  Not
// where it does: its 64 registers instead of 72 let eight instead of seven waiting blocks onto an SM, so that a large grid
// lies on fewer of them (504 blocks, 28 layers 398 and 407 us).
// inv_g: floor((2^32 - 1) / G), so that the upper word of a row times it is row / G or one less.
template <typename T, int D, int NB, bool FLAT>
__global__ void __launch_bounds__(128) combine_kernel(PlanDevice pd, T* __restrict__ out, int n_rows, int n_q_heads, int G, uint32_t inv_g) {
  pdl_launch_dependents();
  // (what all lanes agree on is taken from lane 0, which lets the compiler know: 9 instead of 15 KB of code)
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  int row, pair, g;                                // of all rows; of all (token, KV head) pairs; in the pair's group
  if constexpr (FLAT) {
    row = blockIdx.x * 4 + warp;
    const int r = min(row, n_rows - 1);
    pair = (int)__umulhi((uint32_t)r, inv_g); g = r - pair * G;
    if (g >= G) { ++pair; g -= G; }
  } else {
    const int tok = blockIdx.x, hq = blockIdx.y * 4 + warp, h = hq / G;
    row = tok * n_q_heads + hq; pair = tok * (n_q_heads / G) + h; g = hq - h * G;
  }
  const int p0 = uniform(pd.part_base[pair]), n = uniform(pd.part_base[pair + 1]) - p0;
  pdl_wait();
  if (!FLAT || row < n_rows) combine_row<T, D, NB>(pd.ws_o, pd.ws_ml, p0, n, G, g, lane, out + (size_t)row * D);
}

template <typename T>
__global__ void read_token_kernel(const T* pool, size_t tile, int row, int head_dim, float* out) {
  const int e = threadIdx.x;
  out[e] = to_f32(*reinterpret_cast<const T*>(reinterpret_cast<const char*>(pool) + tile + tile_offset(row, e * sizeof(T), head_dim * sizeof(T))));
}

constexpr int kCombineClaim = 115 * 1024;        // more than half of the 228 KB of an SM
inline int check_launch() { return cudaGetLastError() == cudaSuccess ? ASPD_OK : ASPD_ERR_CUDA; }
inline int status_of(cudaError_t e) { return e == cudaSuccess ? ASPD_OK : ASPD_ERR_CUDA; }

}  // namespace

int launch_append(const aspd_plan* p, const void* k_new, const void* v_new, const int32_t* pos, void* k_pool,
                  void* v_pool, cudaStream_t s) {
  const aspd_shape_t& sh = p->shape;
  const int chunks = sh.head_dim / 2 / (16 / esize_of(sh.dtype));
  const dim3 grid((unsigned)(((long)p->n_new * sh.n_kv_heads * chunks + kAppendThreads - 1) / kAppendThreads)), block(kAppendThreads);
  const float2* cs = pos == p->dev.tok_pos ? p->dev.q_cs : nullptr;
  if (sh.dtype == ASPD_DTYPE_BF16)
    return status_of(launch_pdl(append_kernel<__nv_bfloat16>, grid, block, 0, s, (const __nv_bfloat16*)k_new,
                                (const __nv_bfloat16*)v_new, pos, cs, p->dev.tok_page, p->dev.tok_row, p->dev.inv_freq,
                                (__nv_bfloat16*)k_pool, (__nv_bfloat16*)v_pool, p->n_new, sh.n_kv_heads, sh.head_dim, sh.page_size, p->dev));
  return status_of(launch_pdl(append_kernel<float>, grid, block, 0, s, (const float*)k_new, (const float*)v_new, pos, cs,
                              p->dev.tok_page, p->dev.tok_row, p->dev.inv_freq, (float*)k_pool, (float*)v_pool, p->n_new,
                              sh.n_kv_heads, sh.head_dim, sh.page_size, p->dev));
}

template <typename T, int D, int RPW>
static int launch_generic_rows(const aspd_plan* p, const void* q, const void* k_new, const void* v_new, const void* k_pool, const void* v_pool,
                               cudaStream_t s) {
  static bool configured[64] = {};                 // the attribute belongs to the (function, device) pair
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ASPD_ERR_CUDA;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    if (cudaFuncSetAttribute(attn_generic_kernel<T, D, RPW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GenSmem<T, D>)) != cudaSuccess)
      return ASPD_ERR_CUDA;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const aspd_shape_t& sh = p->shape;
  return status_of(launch_pdl(attn_generic_kernel<T, D, RPW>, dim3(p->n_ctas), dim3(kGenThreads), sizeof(GenSmem<T, D>), s, p->dev,
                              (const T*)q, (const T*)k_new, (const T*)v_new, (T*)k_pool, (T*)v_pool, sh.n_q_heads, sh.n_kv_heads, sh.page_size, sh.sm_scale * kLog2e));
}
template <typename T, int D>
static int launch_generic(const aspd_plan* p, const void* q, const void* k_new, const void* v_new, const void* k_pool, const void* v_pool, cudaStream_t s) {
  const int m = p->max_rows;                       // eight warps
  return m <= 8 ? launch_generic_rows<T, D, 1>(p, q, k_new, v_new, k_pool, v_pool, s) : m <= 16 ? launch_generic_rows<T, D, 2>(p, q, k_new, v_new, k_pool, v_pool, s)
       : m <= 32 ? launch_generic_rows<T, D, 4>(p, q, k_new, v_new, k_pool, v_pool, s) : launch_generic_rows<T, D, 8>(p, q, k_new, v_new, k_pool, v_pool, s);
}

int launch_attn_generic(const aspd_plan* p, const void* q, const void* k_new, const void* v_new, const void* k_pool, const void* v_pool,
                        cudaStream_t s) {
  if (p->n_items == 0) return ASPD_OK;
  const aspd_shape_t& sh = p->shape;
  if (sh.dtype == ASPD_DTYPE_BF16) return sh.head_dim == 128 ? launch_generic<__nv_bfloat16, 128>(p, q, k_new, v_new, k_pool, v_pool, s)
                                                             : launch_generic<__nv_bfloat16, 64>(p, q, k_new, v_new, k_pool, v_pool, s);
  return sh.head_dim == 128 ? launch_generic<float, 128>(p, q, k_new, v_new, k_pool, v_pool, s) : launch_generic<float, 64>(p, q, k_new, v_new, k_pool, v_pool, s);
}

int launch_qcs(const aspd_plan* p, cudaStream_t s) {
  const int half = p->shape.head_dim / 2;
  const long n = (long)p->n_new * half;
  qcs_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p->dev.tok_pos, p->dev.inv_freq, const_cast<float2*>(p->dev.q_cs), p->n_new, half);
  return check_launch();
}

template <typename T, int D, int NB, bool FLAT>
static int launch_combine_rows(const aspd_plan* p, void* out, cudaStream_t s) {
  const aspd_shape_t& sh = p->shape;
  static int sms[64] = {};                         // per device: SMs, known once the kernel has been configured there
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return ASPD_ERR_CUDA;
  int n_sms = dev >= 0 && dev < 64 ? sms[dev] : 0;
  if (n_sms == 0) {
    if (cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(combine_kernel<T, D, NB, FLAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCombineClaim) != cudaSuccess)
      return ASPD_ERR_CUDA;
    if (dev >= 0 && dev < 64) sms[dev] = n_sms;
  }
  // The launch attribute lets the blocks wait on the SMs while the attention pass ends, so that the merge starts
  // without the latency of a launch.  They come to the SMs as those fall free, as many as fit: all 56 of one long
  // request onto the first SM or two, whose memory pipes then do all the work.  So the blocks of a grid that has an
  // SM for each claim, without using it, more than half of an SM's shared memory.  A pass of layers launched from
  // the host, in us, without the attribute / with it / with the claim as well: four branches over 2 k tokens 360 /
  // 330 / 306, one token after another over 1 k 255 / 213 / 213, eight branches over 16 k 517 / 627 / 495, eight
  // requests with heads of 64 410 / 402 / 364.  A grid larger than the chip spreads anyway, and would run in waves
  // (six branches opened with twelve tokens each, 504 blocks: 480 / 438 / 524).
  const int rows = p->n_new * sh.n_q_heads, blocks = (rows + 3) / 4, G = sh.n_q_heads / sh.n_kv_heads;
  const size_t claim = blocks <= n_sms ? kCombineClaim : 0;
  const dim3 grid = FLAT ? dim3(blocks) : dim3(p->n_new, sh.n_q_heads / 4);
  return status_of(launch_pdl(combine_kernel<T, D, NB, FLAT>, grid, dim3(128), claim, s, p->dev, (T*)out, rows, sh.n_q_heads, G, 0xFFFFFFFFu / (uint32_t)G));
}

template <typename T, int D, bool FLAT>
static int launch_combine_of(const aspd_plan* p, void* out, cudaStream_t s) {
  // as many records in flight as the plan's rows have, up to 32: more take registers, and with them blocks from an SM
  // (504 blocks of rows with six records at three: 418 us a pass of 28 layers, at one 395)
  const int nb = (p->max_parts + 7) / 8;
  return nb <= 1 ? launch_combine_rows<T, D, 1, FLAT>(p, out, s) : nb == 2 ? launch_combine_rows<T, D, 2, FLAT>(p, out, s)
       : nb == 3 ? launch_combine_rows<T, D, 3, FLAT>(p, out, s) : launch_combine_rows<T, D, 4, FLAT>(p, out, s);
}

template <typename T, int D>
static int launch_combine_heads(const aspd_plan* p, void* out, cudaStream_t s) {
  return p->shape.n_q_heads % 4 == 0 ? launch_combine_of<T, D, false>(p, out, s) : launch_combine_of<T, D, true>(p, out, s);
}

int launch_combine(const aspd_plan* p, void* out, cudaStream_t s) {
  const aspd_shape_t& sh = p->shape;
  if (sh.dtype == ASPD_DTYPE_BF16) return sh.head_dim == 128 ? launch_combine_heads<__nv_bfloat16, 128>(p, out, s) : launch_combine_heads<__nv_bfloat16, 64>(p, out, s);
  return sh.head_dim == 128 ? launch_combine_heads<float, 128>(p, out, s) : launch_combine_heads<float, 64>(p, out, s);
}

int launch_rerotate(const aspd_shape_t* sh, void* k_pool, const int32_t* pages, const int32_t* rows, const int32_t* delta,
                    int n, cudaStream_t s) {
  const int chunks = sh->head_dim / 2 / (16 / esize_of(sh->dtype));
  const dim3 grid((unsigned)(((long)n * chunks + kRerotateThreads - 1) / kRerotateThreads)), block(kRerotateThreads);
  InvFreq table;
  for (int i = 0; i < sh->head_dim / 2; ++i) table.f[i] = pow((double)sh->rope_theta, -2.0 * i / (double)sh->head_dim);
  if (sh->dtype == ASPD_DTYPE_BF16)
    return status_of(launch_pdl(rerotate_kernel<__nv_bfloat16>, grid, block, 0, s, (__nv_bfloat16*)k_pool, pages, rows,
                                delta, table, n, sh->n_kv_heads, sh->head_dim, sh->page_size));
  return status_of(launch_pdl(rerotate_kernel<float>, grid, block, 0, s, (float*)k_pool, pages, rows, delta,
                              table, n, sh->n_kv_heads, sh->head_dim, sh->page_size));
}

int launch_rerotate_ranges(const aspd_shape_t* sh, void* const* k_pools, int n_layers, const int32_t* page_table,
                           const int32_t* ranges, int n_ranges, cudaStream_t s) {
  const int chunks = sh->head_dim / 2 / (16 / esize_of(sh->dtype)), ps = sh->page_size;
  InvFreq table;
  for (int i = 0; i < sh->head_dim / 2; ++i) table.f[i] = pow((double)sh->rope_theta, -2.0 * i / (double)sh->head_dim);
  for (int r0 = 0; r0 < n_ranges;) {
    RerotateRanges rr;
    rr.n = 0; rr.unit0[0] = 0;
    for (; r0 < n_ranges && rr.n < kMaxRanges; ++r0) {
      const int32_t* g = ranges + 4 * (size_t)r0;
      if (g[2] <= 0) continue;                                   // an empty range moves nothing
      const int pages = (g[1] + g[2] - 1) / ps - g[1] / ps + 1;
      rr.r[rr.n] = make_int4(g[0], g[1], g[2], g[3]);
      rr.unit0[rr.n + 1] = rr.unit0[rr.n] + pages;
      ++rr.n;
    }
    if (rr.n == 0) continue;
    for (int l0 = 0; l0 < n_layers; l0 += kMaxLayerPools) {
      PoolList pools;
      const int nl = std::min(kMaxLayerPools, n_layers - l0);
      for (int l = 0; l < kMaxLayerPools; ++l) pools.p[l] = k_pools[l0 + std::min(l, nl - 1)];
      const dim3 grid((unsigned)rr.unit0[rr.n], (unsigned)nl), block((unsigned)(ps * chunks));
      cudaError_t e;
      if (sh->dtype == ASPD_DTYPE_BF16)
        e = launch_pdl(rerotate_ranges_kernel<__nv_bfloat16>, grid, block, 0, s, pools, page_table, rr, table, sh->n_kv_heads,
                       sh->head_dim, ps);
      else
        e = launch_pdl(rerotate_ranges_kernel<float>, grid, block, 0, s, pools, page_table, rr, table, sh->n_kv_heads,
                       sh->head_dim, ps);
      if (e != cudaSuccess) return ASPD_ERR_CUDA;
    }
  }
  return ASPD_OK;
}

int launch_read_token(const aspd_shape_t* sh, const void* pool, int64_t page, int row, int kv_head, float* out_dev,
                      cudaStream_t s) {
  const int es = esize_of(sh->dtype);
  const size_t tile = ((size_t)page * sh->n_kv_heads + kv_head) * tile_bytes(sh->page_size, sh->head_dim, es);
  if (sh->dtype == ASPD_DTYPE_BF16)
    read_token_kernel<__nv_bfloat16><<<1, sh->head_dim, 0, s>>>((const __nv_bfloat16*)pool, tile, row, sh->head_dim, out_dev);
  else
    read_token_kernel<float><<<1, sh->head_dim, 0, s>>>((const float*)pool, tile, row, sh->head_dim, out_dev);
  return check_launch();
}

}  // namespace aspd

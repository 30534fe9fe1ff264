// Split-K attention on the 5th-generation tensor cores (tcgen05 + TMEM) for the bf16 shapes that aspd_attn_tc.cu
// does not take: head_dim 64, and pages of 8 or 32 tokens at head_dim 64 or 128.
//
// A decoding step has few query rows (tokens x group heads, at most 64 in a row block), so the products are taken
// transposed -- keys and head dimensions fill the rows of the MMAs, the query rows are their N -- and nothing is
// replicated or padded to 128:
//
//     S^T = K . Q^T        tcgen05.mma M = 128 keys, N = rows, K = head_dim    TMEM, two buffers
//     softmax              a thread owns one key of the tile and half of the rows: exponentials against the
//                          rows' references (shared memory, broadcast reads), P^T to shared memory
//     O^T += V^T . P^T     tcgen05.mma M = head_dim, N = rows, K = keys        TMEM
//
// K and V tiles of 128 keys come page by page as linear bulk copies (the cache's tile format is the
// 128-byte-swizzled operand image already; V is the MN-major A operand).
//
// Precision: these shapes ran on the CUDA-core kernel with fp32 queries and weights, and still do: the rotated
// queries and P go into the MMAs as three bf16 pieces each (24 bits, an MMA per piece into the same fp32
// accumulator); K and V are bf16 as stored.
//
// Bound by latency on the steps these shapes have so far: measured on 8 requests of 0.5-4 k tokens (14/2 heads of
// 64, 9.4 MB a layer) 14.8 us a layer from the host, against 1060 us with the CUDA-core kernel, whose warps walked a row's
// keys alone.  One CTA per SM, as many K and V tiles in flight as fit (up to four of either).
//
// Warp roles: 0-7 softmax, query preparation and epilogue (TMEM lane quadrant = warp % 4; warps w and w + 4
// share a quadrant's keys and take half of the rows each), 8 / 9 K / V producers, 10 / 11 issuers of S^T / O^T,
// before that the fused append.  All hand-offs are mbarriers with bounded waits (ASPD_ERR_TIMEOUT on expiry).
#include <stddef.h>

#include <type_traits>

#include "aspd_internal.cuh"
#include "aspd_tc_common.cuh"

namespace aspd {
namespace {

constexpr int kTile = 128;                 // keys per tile
constexpr int kThreads = 384, kSmThreads = 256;
constexpr int W_K = 8, W_V = 9, W_S = 10;     // warp 11: O^T issuer
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRaise = 8.0f;                   // the long way raises a reference only beyond 2^8
constexpr float kLazyLimit = 1099511627776.0f;  // 2^40: a tile's sum of exponentials that sends the tile the long way
constexpr uint32_t COL_S = 0, COL_O = 128, kTmemCols = 256;

constexpr int kPieces = 3;                 // bf16 pieces of a query element and of a weight
constexpr int kMaxSlots = 4;               // K tiles (and V tiles) in flight

enum Bar { K_FULL = 0, K_EMPTY = K_FULL + kMaxSlots, V_FULL = K_EMPTY + kMaxSlots, V_EMPTY = V_FULL + kMaxSlots, S_FULL = V_EMPTY + kMaxSlots,
           S_EMPTY = S_FULL + 2, P_FULL = S_EMPTY + 2, P_EMPTY, O_FULL, Q_FULL, Q_EMPTY, A_DONE, NUM_BARS };

struct DecMisc {
  uint64_t bars[NUM_BARS];
  int nval[2 * kMaxSlots][16];  // page entries of a tile's pages (ring: K runs kMaxSlots tiles ahead of the scores, softmax is two behind)
  int4 vis[2][64];              // visible ranges of the item's query tokens, by item parity
  float nm[64];                 // negated reference of every row (0 while the row has seen no key)
  float ref[64];                // reference of every row in log2 units, -inf while it has seen no key
  float al[64];                 // rescale factors of a long tile; in the epilogue 1 / l
  float wm[4][64];              // per quadrant: row maxima of a long tile; in the epilogue row sums
  int row_out[2][64];           // by item parity: where a row goes (record index, or output row of a whole stream)
  uint32_t tmem_base;
  int abort_flag;
};

struct Ctx {
  PlanDevice pd;
  const __nv_bfloat16* q;
  const __nv_bfloat16* k_new;   // non-null (with v_new): write this step's new rows before reading their pages
  const __nv_bfloat16* v_new;
  const char* k_pool;
  const char* v_pool;
  __nv_bfloat16* out;           // non-null (plans that deal whole streams): the final output; null: records for the combine kernel
  int n_q_heads, n_kv_heads, page_size;
  float scale_log2;
  int early_fetch;              // plan promise: pages without new rows are not written by in-flight work
  int k_shift, v_shift;         // log2 of the K / V tiles in flight
  uint32_t off_v, off_q, off_p, off_misc;
};

// ------------------------------------------------------------------------------------- PTX of this file
// Four k-steps of 16 elements inside one 128-byte span of both K-major operands; lane 0 issues.
__device__ __forceinline__ void tc_mma_k64_lane0(uint32_t d_tmem, uint64_t a0, uint64_t b0, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred e, f, o;\n\t.reg .u32 l;\n\t.reg .b64 a, b;\n\t"
      "mov.u32 l, %%laneid;\n\t"
      "setp.eq.u32 e, l, 0;\n\t"
      "setp.ne.b32 f, %4, 0;\n\t"
      "setp.eq.b32 o, 0, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, f;\n\t"
      "add.s64 a, %1, 2;\n\tadd.s64 b, %2, 2;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, %1, 4;\n\tadd.s64 b, %2, 4;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, %1, 6;\n\tadd.s64 b, %2, 6;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t}"
      ::"r"(d_tmem), "l"(a0), "l"(b0), "r"(idesc), "r"(acc) : "memory");
}
// n (1 to 8) k-steps of 16 keys; the operands' descriptors advance by a_step / b_step (16-byte units) per step.
__device__ __forceinline__ void tc_mma_keys_lane0(uint32_t d_tmem, uint64_t a0, uint64_t b0, uint64_t a_step, uint64_t b_step, uint32_t idesc,
                                                  uint32_t acc, int n) {
  asm volatile(
      "{\n\t.reg .pred e, f, o, q;\n\t.reg .u32 l;\n\t.reg .b64 a, b;\n\t"
      "mov.u32 l, %%laneid;\n\t"
      "setp.eq.u32 e, l, 0;\n\t"
      "setp.ne.b32 f, %4, 0;\n\t"
      "setp.eq.b32 o, 0, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, f;\n\t"
      "add.s64 a, %1, %6;\n\tadd.s64 b, %2, %7;\n\tsetp.gt.and.s32 q, %5, 1, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, a, %6;\n\tadd.s64 b, b, %7;\n\tsetp.gt.and.s32 q, %5, 2, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, a, %6;\n\tadd.s64 b, b, %7;\n\tsetp.gt.and.s32 q, %5, 3, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, a, %6;\n\tadd.s64 b, b, %7;\n\tsetp.gt.and.s32 q, %5, 4, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, a, %6;\n\tadd.s64 b, b, %7;\n\tsetp.gt.and.s32 q, %5, 5, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, a, %6;\n\tadd.s64 b, b, %7;\n\tsetp.gt.and.s32 q, %5, 6, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t"
      "add.s64 a, a, %6;\n\tadd.s64 b, b, %7;\n\tsetp.gt.and.s32 q, %5, 7, e;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, o;\n\t}"
      ::"r"(d_tmem), "l"(a0), "l"(b0), "r"(idesc), "r"(acc), "r"(n), "l"(a_step), "l"(b_step) : "memory");
}
#define ASPD_TMEM_LD8(taddr, v, o)                                                                                \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"                    \
               : "=f"(v[o + 0]), "=f"(v[o + 1]), "=f"(v[o + 2]), "=f"(v[o + 3]), "=f"(v[o + 4]), "=f"(v[o + 5]),   \
                 "=f"(v[o + 6]), "=f"(v[o + 7]) : "r"(taddr) : "memory")
#define ASPD_TMEM_ST8(taddr, v, o)                                                                                \
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"                    \
               ::"f"(v[o + 0]), "f"(v[o + 1]), "f"(v[o + 2]), "f"(v[o + 3]), "f"(v[o + 4]), "f"(v[o + 5]),         \
                 "f"(v[o + 6]), "f"(v[o + 7]), "r"(taddr) : "memory")
// HC consecutive columns of this thread's TMEM lane
template <int HC>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[HC]) {
  if constexpr (HC == 32) ASPD_TMEM_LD32(taddr, v, 0);
  else if constexpr (HC == 16) ASPD_TMEM_LD16(taddr, v, 0);
  else ASPD_TMEM_LD8(taddr, v, 0);
}
// Shared-memory descriptor of the P^T operand (MN-major, NR rows = NR * 2 bytes per key): the swizzle is as
// wide as a key's row, so that one atom spans all rows (8 keys x NR rows).
template <int NR>
__device__ __forceinline__ uint64_t p_desc(uint32_t addr) {
  constexpr uint64_t layout = NR == 64 ? 2 : NR == 32 ? 4 : 6;      // 128-, 64-, 32-byte swizzle
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(NR * 16 >> 4) << 32) | (1ull << 46) | (layout << 61);
}

// The next bf16 pair of (a, b): what is left after `packed`, which is taken off a and b
__device__ __forceinline__ uint32_t pack_next(float& a, float& b, uint32_t packed) {
  a -= __uint_as_float(packed << 16);
  b -= __uint_as_float(packed & 0xffff0000u);
  return pack_bf16(a, b);
}

// N columns reduced over the warp's lanes; lane l ends with column l / (32 / N) (butterfly: N - 1 + log2(32 / N)
// shuffles; redux.sync.max.f32 per column took about 180 cycles each here).
template <int N, typename Op>
__device__ __forceinline__ float lane_reduce(float (&v)[N], int lane, Op op) {
  int n = N;
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    if (n > 1) {
      n >>= 1;
#pragma unroll
      for (int i = 0; i < N / 2; ++i) {
        if (i >= n) break;
        const bool up = (lane & off) != 0;
        const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
        v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, off));
      }
    } else {
      v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], off));
    }
  }
  return v[0];
}

// ------------------------------------------------------------------------------- start of a CTA, start of an item
// New K/V rows of the step in pages that THIS CTA reads (fused step): K rotated at the token's position (cos/sin
// table of the plan), V as is.  CTAs that read the same page write identical bytes.  One unit = one 16-byte
// chunk pair of K (D / 16 per row) or one 16-byte chunk of V (D / 8 per row).
template <int D>
__device__ __forceinline__ void append_rows(const Ctx& c, int tid, int n_threads, int d0, int n_rows) {
  constexpr int UK = D / 16, U = UK + D / 8;
  const uint32_t tb = (uint32_t)c.page_size * D * 2;
  for (int u = tid; u < n_rows * U; u += n_threads) {
    int4 d = c.pd.dirty[d0 + u / U];                              // (page, KV head, token, row | ...)
    d.w &= 255;
    const int sub = u % U;
    if (!bounds_ok(c.pd, d.x, d.w, c.page_size)) continue;
    const size_t src = ((size_t)d.z * c.n_kv_heads + d.y) * D, tile = ((size_t)d.x * c.n_kv_heads + d.y) * tb;
    if (sub < UK) {
      const uint4 a = *reinterpret_cast<const uint4*>(c.k_new + src + sub * 8), b = *reinterpret_cast<const uint4*>(c.k_new + src + D / 2 + sub * 8);
      const float4* cs = reinterpret_cast<const float4*>(c.pd.q_cs + (size_t)d.z * (D / 2) + sub * 8);
      const __nv_bfloat162* a2 = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* b2 = reinterpret_cast<const __nv_bfloat162*>(&b);
      uint32_t lo[4], hi[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 w = cs[i];
        const float2 x0 = __bfloat1622float2(a2[i]), x1 = __bfloat1622float2(b2[i]);
        lo[i] = pack_bf16(x0.x * w.x - x1.x * w.y, x0.y * w.z - x1.y * w.w);
        hi[i] = pack_bf16(x1.x * w.x + x0.x * w.y, x1.y * w.z + x0.y * w.w);
      }
      char* kt = const_cast<char*>(c.k_pool) + tile;
      *reinterpret_cast<uint4*>(kt + tile_offset(d.w, sub * 16, D * 2)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      *reinterpret_cast<uint4*>(kt + tile_offset(d.w, D + sub * 16, D * 2)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    } else {
      const uint4 a = *reinterpret_cast<const uint4*>(c.v_new + src + (sub - UK) * 8);
      *reinterpret_cast<uint4*>(const_cast<char*>(c.v_pool) + tile + tile_offset(d.w, (sub - UK) * 16, D * 2)) = a;
    }
  }
  asm volatile("fence.proxy.async;" ::: "memory");                // before the producers' async-proxy copies
}

// The item's query rows, rotated (RoPE at the token's position), bf16, as the 128-byte-swizzled K-major B
// operand of NR rows (rows beyond the item's are zero).
template <int D, int NR>
__device__ __forceinline__ void prep_q(const Ctx& c, const DeviceItem& it, uint32_t qbuf, int tid) {
  constexpr int UPR = D / 16, UNITS = NR * UPR, PER = (UNITS + kSmThreads - 1) / kSmThreads;
  const int G = c.n_q_heads / c.n_kv_heads, M = it.n_q_tok * G;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int e = tid + u * kSmThreads, r = e / UPR, ch = e % UPR;
    if (UNITS % kSmThreads != 0 && e >= UNITS) break;
    float2 y0[4], y1[4];                                          // the rotated chunk of the first and of the second half
#pragma unroll
    for (int i = 0; i < 4; ++i) y0[i] = y1[i] = make_float2(0.f, 0.f);
    if (r < M) {
      const int tok = it.q_tok0 + r / G, hq = it.kv_head * G + r % G;
      const __nv_bfloat16* qrow = c.q + ((size_t)tok * c.n_q_heads + hq) * D;
      const uint4 a = *reinterpret_cast<const uint4*>(qrow + ch * 8), b = *reinterpret_cast<const uint4*>(qrow + D / 2 + ch * 8);
      const float4* cs = reinterpret_cast<const float4*>(c.pd.q_cs + (size_t)tok * (D / 2) + ch * 8);
      const __nv_bfloat162* a2 = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* b2 = reinterpret_cast<const __nv_bfloat162*>(&b);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 w = cs[i];
        const float2 x0 = __bfloat1622float2(a2[i]), x1 = __bfloat1622float2(b2[i]);
        y0[i] = make_float2(x0.x * w.x - x1.x * w.y, x0.y * w.z - x1.y * w.w);
        y1[i] = make_float2(x1.x * w.x + x0.x * w.y, x1.y * w.z + x0.y * w.w);
      }
    }
    const int ch_hi = ch + D / 16;                                // the chunk D / 2 elements further
    uint32_t a_lo = qbuf + (ch >> 3) * (NR * 128) + r * 128 + (((ch & 7) ^ (r & 7)) << 4);
    uint32_t a_hi = qbuf + (ch_hi >> 3) * (NR * 128) + r * 128 + (((ch_hi & 7) ^ (r & 7)) << 4);
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int pc = 0; pc < kPieces; ++pc, a_lo += NR * D * 2, a_hi += NR * D * 2) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        lo[i] = pc == 0 ? pack_bf16(y0[i].x, y0[i].y) : pack_next(y0[i].x, y0[i].y, lo[i]);
        hi[i] = pc == 0 ? pack_bf16(y1[i].x, y1[i].y) : pack_next(y1[i].x, y1[i].y, hi[i]);
      }
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a_lo), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a_hi), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
    }
  }
  fence_async_smem();
}
// One arrival per warp: what its lanes wrote before is ordered by the warp barrier.
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// ---------------------------------------------------------------------------------------- softmax of an item
// All tiles of one item: scores out of tensor memory, exponentials, P^T.  Leaves the row sums of every quadrant's
// keys in misc->wm.
template <int D, int NR>
__device__ __forceinline__ bool softmax_item(const Ctx& c, const DeviceItem& it, DecMisc* misc, uint32_t bars, uint32_t smem_p, uint32_t tmem,
                                             int par, int& g) {
  constexpr int HC = NR / 2;
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31, q = warp & 3, r0 = (warp >> 2) * HC;
  const int kl = q * 32 + lane;                                  // this thread's key inside a tile
  const int ps = c.page_size, ps_shift = 31 - __clz(ps), ppt = kTile >> ps_shift;
  const int G = c.n_q_heads / c.n_kv_heads, M = it.n_q_tok * G;
  const int n_tiles = (it.n_pages + ppt - 1) / ppt, pe = misc->vis[par][0].x;   // the prefix ends at the same key for all tokens of a block
  volatile int* ab = &misc->abort_flag;
  const uint32_t lane_addr = (uint32_t)(q * 32) << 16, o_addr = tmem + lane_addr + COL_O + r0;
  const float2 sc2 = make_float2(c.scale_log2, c.scale_log2);
  float2 l2[HC / 2];                          // this thread's key's share of the row sums: rows r0 + 2 i, + 1
#pragma unroll
  for (int i = 0; i < HC / 2; ++i) l2[i] = make_float2(0.f, 0.f);
  bool settled = false, dead = false;       // settled: every row of the block has seen a key
  for (int t = 0; t < n_tiles; ++t, ++g) {
    const int sb = g & 1;
    dead |= !mbar_wait(bars + 8 * (S_FULL + sb), (g >> 1) & 1, ab);
    tc_fence_after();
    float s[HC];
    const uint32_t s_addr = tmem + lane_addr + COL_S + sb * 64 + r0;
    tmem_ld<HC>(s_addr, s);
    // Most tiles lie wholly inside what every row may see (the prefix, full pages): one vote.  Elsewhere a bit
    // per row of this thread: the key is a valid row of its page and inside the token's ranges.
    const int ye = misc->nval[g & (2 * kMaxSlots - 1)][kl >> ps_shift], row = kl & (ps - 1), kg = it.key0 + t * kTile + kl;
    const bool valid = row < (ye & 255), full = __all_sync(0xffffffffu, valid && kg < pe) != 0;
    uint32_t bits = 0xffffffffu;
    if (!full) {
      bits = 0;
      const int ofs = (ye >> 13) * ps + row;                      // visible mask of the ablation: the key's offset in its branch
      for (int tl = r0 / G; tl < it.n_q_tok && tl * G < r0 + HC; ++tl) {
        const int4 v = misc->vis[par][tl];
        const int a = max(tl * G - r0, 0), b = min(tl * G + G - r0, HC);
        if (valid && (kg < v.x || (kg >= v.y && kg < v.z) || ofs < v.w)) bits |= (0xffffffffu >> (32 - b)) & ~((1u << a) - 1u);
      }
    }
    tmem_wait_ld();
    // The usual tile is one pass against the references as they are.  An exponent beyond 2^40 shows in the sum
    // and sends the tile the long way (everything is floating point: a reference up to 2^40 below a row's maximum
    // costs no precision), which an item's first tile and tiles while a row has not seen a key take anyway.
    bool redo = !settled;
    for (;;) {
      if (redo) {
        // the long way: row maxima over the tile's keys, references moved, O^T and the sums rescaled
#pragma unroll
        for (int i = 0; i < HC; ++i) s[i] = (bits >> i) & 1u ? s[i] : -INFINITY;
        const float mx = lane_reduce<HC>(s, lane, [](float a, float b) { return fmaxf(a, b); });
        if (lane % (32 / HC) == 0) misc->wm[q][r0 + lane / (32 / HC)] = mx;
        named_sync(1, kSmThreads);
        bool need = false, unset = false;
        if (tid < NR) {
          const float mt = fmaxf(fmaxf(misc->wm[0][tid], misc->wm[1][tid]), fmaxf(misc->wm[2][tid], misc->wm[3][tid])) * c.scale_log2;
          const float old = t > 0 ? misc->ref[tid] : -INFINITY;
          const bool upd = mt > old + kRaise;                     // also true for the first finite maximum (old = -inf)
          const float now = upd ? mt : old;
          misc->ref[tid] = now;
          misc->nm[tid] = now == -INFINITY ? 0.f : -now;
          misc->al[tid] = upd ? ex2(old - mt) : 1.f;
          need = upd && old > -INFINITY;
          unset = tid < M && now == -INFINITY;
        }
        const bool any_need = named_sync_or(1, kSmThreads, need);
        settled = !named_sync_or(1, kSmThreads, unset);
        if (any_need) {
          dead |= !mbar_wait(bars + 8 * P_EMPTY, (g - 1) & 1, ab);   // the O^T of the previous tile is done
          tc_fence_after();
#pragma unroll 1
          for (int c8 = 0; c8 < HC; c8 += 8) {
            float o[8];
            ASPD_TMEM_LD8(o_addr + c8, o, 0);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) o[i] *= misc->al[r0 + c8 + i];
            ASPD_TMEM_ST8(o_addr + c8, o, 0);
          }
          tmem_wait_st();
#pragma unroll
          for (int i = 0; i < HC / 2; ++i) { l2[i].x *= misc->al[r0 + 2 * i]; l2[i].y *= misc->al[r0 + 2 * i + 1]; }
        }
        tmem_ld<HC>(s_addr, s);
        tmem_wait_ld();
      }
      float2 tsum = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < HC; i += 4) {                           // s -> 2^(s * scale - reference)
        const float4 n4 = *reinterpret_cast<const float4*>(&misc->nm[r0 + i]);
        float2 x0 = __ffma2_rn(make_float2(s[i], s[i + 1]), sc2, make_float2(n4.x, n4.y));
        float2 x1 = __ffma2_rn(make_float2(s[i + 2], s[i + 3]), sc2, make_float2(n4.z, n4.w));
        if (!full) {
          x0.x = (bits >> i) & 1u ? x0.x : -INFINITY;       x0.y = (bits >> (i + 1)) & 1u ? x0.y : -INFINITY;
          x1.x = (bits >> (i + 2)) & 1u ? x1.x : -INFINITY; x1.y = (bits >> (i + 3)) & 1u ? x1.y : -INFINITY;
        }
        x0.x = ex2(x0.x); x0.y = ex2(x0.y); x1.x = ex2(x1.x); x1.y = ex2(x1.y);
        s[i] = x0.x; s[i + 1] = x0.y; s[i + 2] = x1.x; s[i + 3] = x1.y;
        tsum = __fadd2_rn(tsum, __fadd2_rn(x0, x1));
      }
      if (redo || !named_sync_or(1, kSmThreads, !(tsum.x + tsum.y <= kLazyLimit))) break;
      redo = true;
      tmem_ld<HC>(s_addr, s);
      tmem_wait_ld();
    }
    tc_fence_before();
    warp_arrive(bars + 8 * (S_EMPTY + sb), lane);                 // the scores are not needed again
#pragma unroll
    for (int i = 0; i < HC / 2; ++i) l2[i] = __fadd2_rn(l2[i], make_float2(s[2 * i], s[2 * i + 1]));
    if (g > 0) dead |= !mbar_wait(bars + 8 * P_EMPTY, (g - 1) & 1, ab);   // the P^T tile is free again
    // key kl's row of P^T: NR bf16, 16-byte chunks swizzled over the atom's width
    const int sw = NR == 64 ? kl & 7 : NR == 32 ? (kl >> 1) & 3 : (kl >> 2) & 1;
#pragma unroll
    for (int c8 = 0; c8 < HC / 8; ++c8) {
      const uint32_t addr = smem_p + kl * (NR * 2) + (((r0 / 8 + c8) ^ sw) << 4);
      uint32_t w[4];
#pragma unroll
      for (int pc = 0; pc < kPieces; ++pc) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float &x = s[c8 * 8 + 2 * i], &y = s[c8 * 8 + 2 * i + 1];
          w[i] = pc == 0 ? pack_bf16(x, y) : pack_next(x, y, w[i]);
        }
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr + pc * (kTile * NR * 2)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                     : "memory");
      }
    }
    fence_async_smem();
    tc_fence_before();
    warp_arrive(bars + 8 * P_FULL, lane);
  }
  float l[HC];
#pragma unroll
  for (int i = 0; i < HC / 2; ++i) { l[2 * i] = l2[i].x; l[2 * i + 1] = l2[i].y; }
  const float sum = lane_reduce<HC>(l, lane, [](float a, float b) { return a + b; });
  constexpr int REP = 32 / HC;
  if (lane % REP == 0) misc->wm[q][r0 + lane / REP] = sum;
  return !dead;
}

// --------------------------------------------------------------------------------------- end of an item
// O^T (tensor memory: lane = element of the head, column = row) and the sums become one record per row for the
// combine kernel, or the final output (plans that deal whole streams).  Returned: something of this thread's is not
// finite (see redo_item).
template <int D, int NR>
__device__ __forceinline__ bool finish_item(const Ctx& c, const DeviceItem& it, DecMisc* misc, uint32_t tmem, int par, bool dead) {
  constexpr int HC = NR / 2;
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31, q = warp & 3, r0 = (warp >> 2) * HC;
  const int M = it.n_q_tok * (c.n_q_heads / c.n_kv_heads);
  const uint32_t o_addr = tmem + ((uint32_t)(q * 32) << 16) + COL_O + r0;
  // head element of this thread's lane: M = 64 MMAs (D = 64) keep 16 rows in lanes 0..15 of each quadrant
  const int d = D == 128 ? q * 32 + lane : q * 16 + lane;
  const bool has_d = (D == 128 || lane < 16) && !dead;
  const bool whole = c.out != nullptr;
  bool bad = false;
  uint32_t top = 0;                                               // largest magnitude, as bits
  if (tid < NR) {
    const float l = (misc->wm[0][tid] + misc->wm[1][tid]) + (misc->wm[2][tid] + misc->wm[3][tid]);
    misc->al[tid] = l > 0.f ? 1.f / l : 0.f;
    bad = tid < M && (!(l < INFINITY) || misc->ref[tid] == INFINITY);
    if (!whole && tid < M && !dead) c.pd.ws_ml[misc->row_out[par][tid]] = make_float2(l > 0.f ? misc->ref[tid] : -INFINITY, l);
  }
  if (whole) named_sync(1, kSmThreads);
#pragma unroll
  for (int c8 = 0; c8 < HC; c8 += 8) {
    float o[8];
    ASPD_TMEM_LD8(o_addr + c8, o, 0);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 8; ++i) top = max(top, __float_as_uint(o[i]) & 0x7fffffffu);   // (a test per stored element: 1.3 us a layer)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = r0 + c8 + i;
      if (!has_d || r >= M) continue;
      const size_t at = (size_t)misc->row_out[par][r] * D + d;
      if (whole) c.out[at] = __float2bfloat16_rn(o[i] * misc->al[r]);
      else c.pd.ws_o[at] = o[i];
    }
  }
  return bad || (has_d && top >= 0x7f800000u);
}

// An item whose result is not finite, once more on the CUDA cores and straight from the pools.  The MMAs multiply every
// V row of a tile by every row's weight, 0 for a key that the row does not see, so that Inf or NaN in one branch's
// values becomes NaN in its sibling branches; and of an Inf that a row does see the pieces of queries and weights
// make NaN.  Here a row takes the keys that it sees, as the CUDA-core kernel does.  A warp per query row, 32
// keys at a time, a key per lane for the scores and D / 32 elements of the head per lane for the sum; nothing is
// tuned, since finite values never come here (a vote that the item's end takes anyway asks for it) and a function
// of its own keeps it out of the loop's code.  What the steps pay for asking, us a layer before and now: 8 requests with
// heads of 64 from the host 14.6 and 14.8, steps with pages of 8 or 32 up to 2 % (inlined: up to 3 %).
template <int D>
__device__ __noinline__ void redo_item(const Ctx& c, const DeviceItem it, DecMisc* misc, float* q_sm, int par) {
  constexpr int EPL = D / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, G = c.n_q_heads / c.n_kv_heads, M = it.n_q_tok * G;
  const int ps = c.page_size, n_keys = it.n_pages * ps;
  const uint32_t tb = (uint32_t)ps * D * 2;
  float* qw = q_sm + warp * D;                                    // the row's query, rotated and scaled
#pragma unroll 1
  for (int r = warp; r < M; r += 8) {
    const int tok = it.q_tok0 + r / G;
    const __nv_bfloat16* qrow = c.q + ((size_t)tok * c.n_q_heads + it.kv_head * G + r % G) * D;
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < D / 2; i += 32) {
      const float2 cs = c.pd.q_cs[(size_t)tok * (D / 2) + i];
      const float x0 = __bfloat162float(qrow[i]), x1 = __bfloat162float(qrow[i + D / 2]);
      qw[i] = (x0 * cs.x - x1 * cs.y) * c.scale_log2;
      qw[i + D / 2] = (x1 * cs.x + x0 * cs.y) * c.scale_log2;
    }
    __syncwarp();
    const int4 vis = misc->vis[par][r / G];
    float m = -INFINITY, l = 0.f, acc[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < n_keys; k0 += 32) {
      const int j = min(k0 + lane, n_keys - 1), row = j & (ps - 1), kg = it.key0 + j;
      const int2 pg = c.pd.visit[it.page0 + j / ps];
      const bool seen = k0 + lane < n_keys && row < (pg.y & 255) && (kg < vis.x || (kg >= vis.y && kg < vis.z) || (pg.y >> 13) * ps + row < vis.w) &&
                        bounds_ok(c.pd, pg.x, row, ps);
      if (!__any_sync(0xffffffffu, seen)) continue;
      float s = -INFINITY;
      if (seen) {
        const char* tile = c.k_pool + ((size_t)pg.x * c.n_kv_heads + it.kv_head) * tb;
        s = 0.f;
#pragma unroll 2
        for (int ch = 0; ch < D / 8; ++ch) {
          const uint4 raw = __ldcg(reinterpret_cast<const uint4*>(tile + tile_offset(row, ch * 16, D * 2)));
          const __nv_bfloat162* k2 = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 x = __bfloat1622float2(k2[i]), w = *reinterpret_cast<const float2*>(qw + ch * 8 + 2 * i);
            s = fmaf(w.x, x.x, s); s = fmaf(w.y, x.y, s);
          }
        }
      }
      float mn = s;
#pragma unroll
      for (int o = 16; o; o >>= 1) mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mn = fmaxf(m, mn);
      const float w = seen ? exp2f(s - mn) : 0.f, alpha = m == -INFINITY ? 0.f : exp2f(m - mn);
      float sum = w;
#pragma unroll
      for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      l = l * alpha + sum;
      m = mn;
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] *= alpha;
#pragma unroll 2
      for (int kk = 0; kk < 32; ++kk) {
        const float wk = __shfl_sync(0xffffffffu, w, kk);
        const int page = __shfl_sync(0xffffffffu, pg.x, kk), vrow = __shfl_sync(0xffffffffu, row, kk);
        if (wk == 0.f) continue;
        const char* vt = c.v_pool + ((size_t)page * c.n_kv_heads + it.kv_head) * tb;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
          const uint32_t bits = __ldcg(reinterpret_cast<const unsigned short*>(vt + tile_offset(vrow, (e * 32 + lane) * 2, D * 2)));
          acc[e] = fmaf(wk, __uint_as_float(bits << 16), acc[e]);
        }
      }
    }
    const size_t at = misc->row_out[par][r];
    if (c.out == nullptr && lane == 0) c.pd.ws_ml[at] = make_float2(m, l);
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      if (c.out != nullptr) c.out[at * D + e * 32 + lane] = __float2bfloat16_rn(acc[e] * (1.f / l));
      else c.pd.ws_o[at * D + e * 32 + lane] = acc[e];
    }
  }
}

// -------------------------------------------------------------------------------------------- the kernel
// NR: rows that the plan's largest row block is padded to; its smaller blocks are padded as far.  (One instance that
// chose per item was 161 KB of code, these are 65 to 99, and a short launch waits for its instructions: 14.5 against
// 14.1 us a layer in a graph on the step above.)
template <int D, int NR>
__global__ void __launch_bounds__(kThreads, 1) attn_dec_kernel(const __grid_constant__ Ctx c) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  DecMisc* misc = reinterpret_cast<DecMisc*>(smem_raw + (base - raw) + c.off_misc);
  const uint32_t bars = base + c.off_misc;          // bars[] is the first member
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  volatile int* ab = &misc->abort_flag;
  constexpr uint32_t kTileBytes = kTile * D * 2;
  if (tid == 0) pdl_launch_dependents();
  const int4 head = c.pd.cta_head[2 * blockIdx.x], head2 = c.pd.cta_head[2 * blockIdx.x + 1];
  const int item_begin = uniform(head.x), item_end = uniform(head.y);
  const int ps = c.page_size, ps_shift = 31 - __clz(ps), ppt = kTile >> ps_shift;
  int2 first_pages = make_int2(0, 0);
  if ((warp == W_K || warp == W_V) && lane < head.w) first_pages = c.pd.visit[head.z + lane];
  if (tid == 0) {
    auto count = [](int i) { return i >= S_EMPTY && i < P_FULL ? 8 : i == P_FULL || i == Q_FULL ? 8 : i == A_DONE ? 2 : 1; };   // one arrival per warp that takes part
    for (int i = 0; i < NUM_BARS; ++i) mbar_init(bars + 8 * i, count(i));
    misc->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == W_S) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&misc->tmem_base)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc->tmem_base;
  // plan data of the first item
  DeviceItem first = {};
  if (warp < 8 && item_begin < item_end) first = uniform_item(c.pd.items[item_begin]);
  // everything above touches only the plan's own tables; inputs written by earlier kernels of the stream are
  // used from here on.  With the plan's stable-cache promise the producers go ahead with pages that hold no
  // new rows; they wait themselves before the first page that does.
  const bool producer = warp == W_K || warp == W_V, runs_ahead = c.early_fetch && producer;
  if (!runs_ahead) pdl_wait();
  bool dead = false;

  if (warp < 8) {
    // ============================ softmax, query preparation, append, epilogue ============================
    const int G = c.n_q_heads / c.n_kv_heads;
    int g = 0, item_no = 0;
    // the item's query tile, its tokens' ranges and where its rows go
    auto start_item = [&](const DeviceItem& it, int par) {
      const int m = it.n_q_tok * G;
      int4 vis = make_int4(0, 0, 0, 0);
      int row_out = 0;
      if (tid < it.n_q_tok) vis = c.pd.tok_vis[it.q_tok0 + tid];
      if (tid < m) {
        const int tok = it.q_tok0 + tid / G;
        row_out = c.out != nullptr ? tok * c.n_q_heads + it.kv_head * G + tid % G
                                   : (c.pd.part_base[tok * c.n_kv_heads + it.kv_head] + it.part_slot) * G + tid % G;
      }
      prep_q<D, NR>(c, it, base + c.off_q, tid);
      if (tid < it.n_q_tok) misc->vis[par][tid] = vis;
      if (tid < m) misc->row_out[par][tid] = row_out;
      warp_arrive(bars + 8 * Q_FULL, lane);
    };
    if (item_begin < item_end) start_item(first, 0);
    for (int idx = item_begin; idx < item_end; ++idx, ++item_no) {
      const DeviceItem it = idx == item_begin ? first : uniform_item(c.pd.items[idx]);
      const int par = item_no & 1;
      named_sync(1, kSmThreads);                                  // the item's ranges are there
      dead |= !softmax_item<D, NR>(c, it, misc, bars, base + c.off_p, tmem, par, g);
      if (idx + 1 < item_end) {                                   // the next query tile as soon as this item's last scores are issued
        dead |= !mbar_wait(bars + 8 * Q_EMPTY, item_no & 1, ab);
        start_item(uniform_item(c.pd.items[idx + 1]), par ^ 1);
      }
      dead |= !mbar_wait(bars + 8 * O_FULL, item_no & 1, ab);
      tc_fence_after();
      named_sync(1, kSmThreads);                                  // the row sums of all quadrants
      const bool bad = finish_item<D, NR>(c, it, misc, tmem, par, dead || *ab);
      tc_fence_before();
      if (named_sync_or(1, kSmThreads, bad || dead || *ab)) {
        if (c.k_new != nullptr) dead |= !mbar_wait(bars + 8 * A_DONE, 0, ab);     // the step's own rows are in the pools
        if (named_sync_or(1, kSmThreads, dead || *ab)) break;
        redo_item<D>(c, it, misc, reinterpret_cast<float*>(smem_raw + (base - raw) + c.off_p), par);
      }
    }
  } else if (producer) {
    // ================================ bulk-copy producers ================================
    // Lane l keeps stream-page entry (batch * 32 + l) of the item in a register; the next batch is requested
    // before the current one is consumed, also across an item boundary.
    const bool is_v = warp == W_V;
    const char* pool = is_v ? c.v_pool : c.k_pool;
    const int shift = is_v ? c.v_shift : c.k_shift;
    const uint32_t page_bytes = (uint32_t)ps * D * 2, dst0 = base + (is_v ? c.off_v : 0u);
    const int tpb = 32 / ppt;                                     // tiles per batch of 32 entries
    int g = 0;
    bool ok = true, appended = false, waited = false;
    int2 nxt = first_pages;
    for (int idx = item_begin; idx < item_end && ok; ++idx) {
      const DeviceItem it = uniform_item(c.pd.items[idx]);
      const int n_tiles = (it.n_pages + ppt - 1) / ppt;
      int2 cur = make_int2(0, 0);
      for (int t = 0; t < n_tiles && ok; ++t, ++g) {
        if (t % tpb == 0) {
          cur = nxt;
          nxt = make_int2(0, 0);
          const int ahead = (t + tpb) * ppt;
          if (ahead < it.n_pages) {
            if (ahead + lane < it.n_pages) nxt = c.pd.visit[it.page0 + ahead + lane];
          } else if (idx + 1 < item_end) {
            const int2 nx = make_int2(c.pd.items[idx + 1].page0, c.pd.items[idx + 1].n_pages);
            if (lane < nx.y) nxt = c.pd.visit[nx.x + lane];
          }
        }
        const int npg = min(ppt, it.n_pages - t * ppt);
        // pages of 8: an odd last page is copied twice, so that the last k-step of 16 keys reads no stale rows
        const int ncopy = ps == 8 ? (npg + 1) & ~1 : npg, sl = g & ((1 << shift) - 1), fill = g >> shift;
        int2 pg;
        const int src_lane = (t % tpb) * ppt + min(lane & (ppt - 1), npg - 1);
        pg.x = __shfl_sync(0xffffffffu, cur.x, src_lane);
        pg.y = __shfl_sync(0xffffffffu, cur.y, src_lane);
        if (lane >= npg) pg.y = 0;                                // no valid rows behind the item's pages
        if (lane < ncopy && !bounds_ok(c.pd, pg.x, 0, ps)) pg.x = 0;     // checking builds: flagged, page 0 read instead
        const bool fresh = __any_sync(0xffffffffu, ((pg.y >> 8) & 31) != 0) != 0;
        if (runs_ahead && !waited && fresh) {
          pdl_wait();                                             // new rows come from the previous kernel (or from this one)
          waited = true;
        }
        if (c.k_new != nullptr && !appended && fresh) {           // fused append: the rows are being written by this CTA
          ok = __all_sync(0xffffffffu, mbar_wait(bars + 8 * A_DONE, 0, ab)) != 0;
          if (!ok) break;
          appended = true;
        }
        const uint32_t full = bars + 8 * ((is_v ? V_FULL : K_FULL) + sl), empty = bars + 8 * ((is_v ? V_EMPTY : K_EMPTY) + sl);
        ok = __all_sync(0xffffffffu, mbar_wait(empty, (fill & 1) ^ 1, ab)) != 0;
        if (!ok) break;
        if (!is_v && lane < 16) misc->nval[g & (2 * kMaxSlots - 1)][lane] = pg.y;   // read by the softmax warps of tile g
        __syncwarp();
        if (lane == 0) mbar_expect_tx(full, (uint32_t)ncopy * page_bytes);
        __syncwarp();
        if (lane < ncopy)
          bulk_copy(dst0 + sl * kTileBytes + lane * page_bytes, pool + ((size_t)pg.x * c.n_kv_heads + it.kv_head) * page_bytes, page_bytes, full);
      }
    }
  } else {
    // ================== MMA issuers (one in-order stream of operations each; all lanes wait, lane 0 issues) ==================
    const uint32_t fm = 0xffffffffu;
    const uint32_t tmem_u = __shfl_sync(fm, tmem, 0), base_u = __shfl_sync(fm, base, 0), bars_u = base_u + c.off_misc;
    const int ib = __shfl_sync(fm, item_begin, 0), ie = __shfl_sync(fm, item_end, 0), G = c.n_q_heads / c.n_kv_heads;
    auto wait_all = [&](uint32_t bar, uint32_t parity) { return __all_sync(fm, mbar_wait(bar, parity, ab)) != 0; };
    constexpr uint32_t kRowGroup = 8 * D * 2;                     // bytes of 8 tokens in a tile
    if (c.k_new != nullptr) {                                     // beside the preparation of the first query tile
      append_rows<D>(c, tid - W_S * 32, 64, head2.x, head2.y);
      warp_arrive(bars + 8 * A_DONE, lane);
    }
    int g = 0, item_no = 0;
    bool ok = true;
    for (int idx = ib; idx < ie && ok; ++idx, ++item_no) {
      const int n_pages = __shfl_sync(fm, c.pd.items[idx].n_pages, 0);
      const int n_tiles = (n_pages + ppt - 1) / ppt;
      for (int t = 0; t < n_tiles && ok; ++t, ++g) {
        if (warp == W_S) {
          const int sb = g & 1, sl = g & ((1 << c.k_shift) - 1), fill = g >> c.k_shift;
          ok = (t > 0 || wait_all(bars_u + 8 * Q_FULL, item_no & 1)) && wait_all(bars_u + 8 * (K_FULL + sl), fill & 1) &&
               wait_all(bars_u + 8 * (S_EMPTY + sb), ((g >> 1) & 1) ^ 1);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a = smem_desc(base_u + sl * kTileBytes, 16, kRowGroup), b = smem_desc(base_u + c.off_q, 16, 1024);
          const uint32_t idesc = instr_desc(NR, 0), d = tmem_u + COL_S + sb * 64;
#pragma unroll
          for (int pc = 0; pc < kPieces; ++pc) {                 // the queries' pieces lie NR * D * 2 bytes apart
            tc_mma_k64_lane0(d, a, b + pc * (NR * D / 8), idesc, pc);
            if constexpr (D == 128) tc_mma_k64_lane0(d, a + 64, b + pc * (NR * D / 8) + NR * 8, idesc, 1);   // second span: 1024 B further in K, NR * 128 B in Q
          }
          tc_commit_lane0(bars_u + 8 * (S_FULL + sb));
          tc_commit_lane0(bars_u + 8 * (K_EMPTY + sl));
          if (t == n_tiles - 1) tc_commit_lane0(bars_u + 8 * Q_EMPTY);
        } else {
          const int sl = g & ((1 << c.v_shift) - 1), fill = g >> c.v_shift;
          const int steps = (min(ppt, n_pages - t * ppt) * ps + 15) >> 4;
          ok = wait_all(bars_u + 8 * (V_FULL + sl), fill & 1) && wait_all(bars_u + 8 * P_FULL, g & 1);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a = smem_desc(base_u + c.off_v + sl * kTileBytes, 1024, kRowGroup);
          const uint64_t b = p_desc<NR>(base_u + c.off_p);
          // both operands MN-major; 16 keys are two groups of 8 in either
          const uint32_t idesc = instr_desc(NR, 1, D) | (1u << 15);
#pragma unroll
          for (int pc = 0; pc < kPieces; ++pc)
            tc_mma_keys_lane0(tmem_u + COL_O, a, b + pc * (kTile * NR / 8), 2 * kRowGroup >> 4, NR * 2, idesc, t > 0 || pc > 0 ? 1u : 0u, steps);
          tc_commit_lane0(bars_u + 8 * P_EMPTY);
          tc_commit_lane0(bars_u + 8 * (V_EMPTY + sl));
          if (t == n_tiles - 1) tc_commit_lane0(bars_u + 8 * O_FULL);
        }
      }
    }
    __syncwarp();
  }

  // ---- on a time-out give outstanding copies and MMAs time to land before the CTA's shared memory and TMEM go away
  if (*ab) {
    if (tid == 0) atomicCAS(c.pd.status, 0, (int)ASPD_ERR_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == W_S) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

inline uint32_t up1k(uint32_t x) { return (x + 1023u) & ~1023u; }

// Shared memory of a plan whose row blocks are padded to nr rows: 1 to 4 K tiles and V tiles, as many as fit.
constexpr uint32_t kSmemMax = 232448;
inline uint32_t smem_layout(int D, int nr, Ctx* c) {
  const uint32_t tile = kTile * D * 2, q = up1k(kPieces * nr * D * 2), p = up1k(kPieces * kTile * nr * 2);
  const uint32_t rest = q + p + (uint32_t)sizeof(DecMisc) + 1024;       // + slack to align the base
  auto fits = [&](int k, int v) { return ((1u << k) + (1u << v)) * tile + rest <= kSmemMax; };
  c->k_shift = fits(2, 2) ? 2 : fits(1, 0) ? 1 : 0;
  c->v_shift = fits(2, 2) ? 2 : fits(1, 1) ? 1 : 0;
  c->off_v = tile << c->k_shift;
  c->off_q = c->off_v + (tile << c->v_shift);
  c->off_p = c->off_q + q;
  c->off_misc = c->off_p + p;
  return c->off_misc + (uint32_t)sizeof(DecMisc) + 1024;
}

template <int D, int NR>
cudaError_t launch(const aspd_plan* p, Ctx& c, cudaStream_t s) {
  static bool configured[64] = {};                 // the attribute belongs to the (function, device) pair
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(attn_dec_kernel<D, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const uint32_t smem = smem_layout(D, NR, &c);
  return launch_pdl(attn_dec_kernel<D, NR>, dim3(p->n_ctas), dim3(kThreads), smem, s, c);
}

}  // namespace

int launch_attn_dec(const aspd_plan* p, const void* q, const void* k_new, const void* v_new, const void* k_pool, const void* v_pool,
                    void* out, cudaStream_t s) {
  if (p->n_items == 0) return ASPD_OK;
  const aspd_shape_t& sh = p->shape;
  Ctx c;
  c.pd = p->dev;
  c.q = (const __nv_bfloat16*)q;
  c.k_new = (const __nv_bfloat16*)k_new; c.v_new = (const __nv_bfloat16*)v_new;
  c.k_pool = (const char*)k_pool; c.v_pool = (const char*)v_pool;
  c.out = p->dealt ? (__nv_bfloat16*)out : nullptr;
  c.n_q_heads = sh.n_q_heads; c.n_kv_heads = sh.n_kv_heads; c.page_size = sh.page_size;
  c.scale_log2 = sh.sm_scale * kLog2e;
  c.early_fetch = p->stable_cache;
  const int nr = padded_rows(p->max_rows);
  const cudaError_t e = sh.head_dim == 64 ? (nr == 16 ? launch<64, 16>(p, c, s) : nr == 32 ? launch<64, 32>(p, c, s) : launch<64, 64>(p, c, s))
                                          : (nr == 16 ? launch<128, 16>(p, c, s) : nr == 32 ? launch<128, 32>(p, c, s) : launch<128, 64>(p, c, s));
  return e == cudaSuccess ? ASPD_OK : ASPD_ERR_CUDA;
}

}  // namespace aspd

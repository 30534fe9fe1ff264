// The two-tile variant of the tensor-core attention kernel (plans that deal whole streams with row
// blocks of up to 256 query rows: masked prefill, teacher forcing).  Included by aspd_attn_tc.cu.
//
// A row block is two query tiles of 128 rows (tile j holds tokens j * (128 / G) ...).  Every K/V
// tile the CTA fetches is scored against both:
//
//     S_j = Q_j . K^T        tcgen05.mma M=128, N=keys, K=128       TMEM columns 128 j
//     softmax group j        four warps, thread r = row r of tile j: the tile's keys in two halves of
//                            64, exponentials against the row's reference maximum (raised only when
//                            an exponent passes 2^40, decided by the thread alone: no exchange), P half
//                            (64 keys, bf16) over the first 32 columns of the half's own scores
//     O_j += P_j . V         tcgen05.mma M=128, N=128, K=64 per half, A operand from tensor memory
//                            TMEM columns 256 + 128 j
//
// so that while one group is in its exponentials the tensor pipe works for the other, and a thread
// owns its row from the query's rotation to the normalised output (it prepares its group's query tile,
// divides by l and stores the row itself; nothing is handed over).  Warp roles: 0-3 group 0, 4-7 group
// 1, 8 / 9 K / V producers, 10 / 11 issuers of the MMAs of group 0 / 1.  Single buffers for S and the
// query tiles; K and V tiles double-buffered.  All waits are bounded as in the other variants.
//
// Bound by the softmax groups' passes (about 1 000-1 200 cycles for 64 scores a row beside the other group's, 512 of
// them the special-function unit's) and, in long runs, by the power cap.  Whole branches of 32 requests, 28 layers:
// 25.2 -> 22.2 ms a pass under the cap (24.9 -> 23.8 on a box that held less clock); of four requests, below the cap,
// 1 605 -> 1 197 us.
// What made the difference to four issuer warps and 512 threads of 128 registers: a group rotates its next query
// tile itself right after its last P of an item, all loads at once (four warps that issued MMAs as well took 16 000
// cycles from an item's last P to the next item's first scores, thirteen times a CTA), and scores run right behind the
// P.V before them without a word in between (see the issuers).  Measured and not taken, same workload: scores of a whole tile in one
// MMA (26.2 ms: nothing for the tensor pipe to do while a group is in its passes), a quarter of the exponentials as a
// polynomial on the FMA pipe (22.9; it takes power, and is less precise), the next half's scores asked for before P
// is stored (24.1).
#pragma once

namespace {      // included inside namespace aspd

constexpr int kThreadsW2 = 384;               // 168 registers a thread; 44 bytes are spilled
constexpr int W2_KPROD = 8, W2_VPROD = 9, W2_ISSUE = 10;
constexpr uint32_t W2_OFF_K = 0, W2_OFF_V = 2 * kTileBytes, W2_OFF_Q = 4 * kTileBytes, W2_OFF_OUT = 6 * kTileBytes,
                   W2_OFF_MISC = 7 * kTileBytes;
constexpr size_t kSmemBytesW2 = 7 * kTileBytes + 2048 + 1024;   // + Misc + slack to align the base to 1024
constexpr int kItemCacheW2 = 8;
constexpr int kPageRingW2 = 8;      // tiles whose page entries are kept: a group may be read up to four tiles late (see softmax_group_w2)
// The reference maximum of a row is raised when an exponent passes 2^40 (everything is floating point,
// bf16 and fp32 alike, so the distance costs no precision; what must not happen is an overflow, and
// 2^40 x 2^13 keys x |v| is far from one).  The one-tile variants raise at 2^8.
constexpr float kRaiseW2 = 40.0f, kRaiseSumW2 = 1099511627776.0f;

// S_FULL / P_FULL: one per (group, half of the tile's keys)
enum BarW2 { WK_FULL = 0, WK_EMPTY = 2, WV_FULL = 4, WV_EMPTY = 6, WS_FULL = 8, WP_FULL = 12, WPV_DONE = 16, WO_FULL = 18, WQ_FULL = 20,
             W2_NUM_BARS = 22 };

struct MiscW2 {
  uint64_t bars[W2_NUM_BARS];
  int nval[kPageRingW2][8];          // page entries of the 8 pages of a tile
  DeviceItem items[kItemCacheW2];
  uint32_t tmem_base;
  int abort_flag;
  int lead;                          // the item group 0's issuer is at (read by group 1's)
};
static_assert(sizeof(MiscW2) <= 2048, "MiscW2 must fit behind the tiles");

__device__ __forceinline__ DeviceItem get_item_w2(const Ctx& c, const MiscW2* misc, int idx, int item_begin) {
  const int rel = idx - item_begin;
  return uniform_item(rel < kItemCacheW2 ? misc->items[rel] : c.pd.items[idx]);
}

// One arrival per warp: what its lanes did before is ordered by the warp barrier.
__device__ __forceinline__ void warp_arrive_w2(uint32_t bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

// The group's query tile of an item: rows rotated (RoPE at the token's position, cos/sin table of the plan), bf16,
// as the 128-byte-swizzled K-major A operand (rows beyond the item's are zero).  A thread takes the 16-byte chunk
// `rank % 8` of both halves of rows rank / 8 + 16 u; all of its query loads are on their way before the first is used.
__device__ __forceinline__ void prep_tile_w2(const Ctx& c, int q_tok0, int n_tok, int kv_head, uint32_t qbuf, int rank) {
  const int G = c.G, M = n_tok * G, ch = rank & 7, row0 = rank >> 3;
  const __nv_bfloat16* q0 = c.q + ((size_t)q_tok0 * c.n_q_heads + kv_head * G) * 128 + ch * 8;
  const float4* cs0 = reinterpret_cast<const float4*>(c.pd.q_cs + (size_t)q_tok0 * 64 + ch * 8);
  uint4 a[8], b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int r = row0 + 16 * u, tl = token_of(c, r);
    a[u] = make_uint4(0, 0, 0, 0); b[u] = make_uint4(0, 0, 0, 0);
    if (r < M) {
      const __nv_bfloat16* p = q0 + (size_t)(tl * (c.n_q_heads - G) + r) * 128;      // (tl * n_q_heads + r - tl * G) rows further
      a[u] = *reinterpret_cast<const uint4*>(p);
      b[u] = *reinterpret_cast<const uint4*>(p + 64);
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int r = row0 + 16 * u, tl = token_of(c, r);
    const float4* cs = cs0 + (size_t)(r < M ? tl : 0) * 32;
    const __nv_bfloat162* a2 = reinterpret_cast<const __nv_bfloat162*>(&a[u]);
    const __nv_bfloat162* b2 = reinterpret_cast<const __nv_bfloat162*>(&b[u]);
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 w = cs[i];
      const float2 x0 = __bfloat1622float2(a2[i]), x1 = __bfloat1622float2(b2[i]);
      lo[i] = pack_bf16(x0.x * w.x - x1.x * w.y, x0.y * w.z - x1.y * w.w);
      hi[i] = pack_bf16(x1.x * w.x + x0.x * w.y, x1.y * w.z + x0.y * w.w);
    }
    const uint32_t addr = qbuf + r * 128 + ((ch ^ (r & 7)) << 4);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr + kHalf), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
  }
  fence_async_smem();
}

// One softmax group over all items of the CTA.  grp = 0 / 1, r = the thread's row in its tile.
__device__ __forceinline__ void softmax_group_w2(const Ctx& c, MiscW2* misc, uint32_t bars, uint32_t base, uint32_t tmem, int item_begin,
                                                 int item_end, int grp, int tpt) {
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31, r = tid & 127;
  const int G = c.G;
  volatile int* ab = &misc->abort_flag;
  const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t s_base = tmem + lane_addr + COL_S + grp * 128, o_base = tmem + lane_addr + COL_O + grp * 128;
  const uint32_t qbuf = base + W2_OFF_Q + grp * kTileBytes, obuf = base + W2_OFF_OUT + warp * 4096;
  const uint32_t bar_sfull = bars + 8 * (WS_FULL + 2 * grp), bar_pfull = bars + 8 * (WP_FULL + 2 * grp),      // + 8 h
                 bar_pvdone = bars + 8 * (WPV_DONE + grp), bar_ofull = bars + 8 * (WO_FULL + grp), bar_qfull = bars + 8 * (WQ_FULL + grp);
  // the first item from `idx` on in which the group has a tile; its query tile is prepared
  auto next_item = [&](int idx) {
    for (; idx < item_end; ++idx) {
      const DeviceItem it = get_item_w2(c, misc, idx, item_begin);
      if (it.n_q_tok > grp * tpt) {
        prep_tile_w2(c, it.q_tok0 + grp * tpt, min(tpt, it.n_q_tok - grp * tpt), it.kv_head, qbuf, r);
        warp_arrive_w2(bar_qfull);
        break;
      }
    }
  };
  next_item(item_begin);
  int g = 0;            // tiles of the CTA so far (both groups count the same)
  int sc[2] = {0, 0}, hc = 0, ic = 0;   // this group's score operations (first / second half), P halves and items so far
  bool dead = false;
  for (int idx = item_begin; idx < item_end; ++idx) {
    const DeviceItem it = get_item_w2(c, misc, idx, item_begin);
    const int n_tiles = (it.n_pages + 7) >> 3;
    const int n_tok = min(tpt, it.n_q_tok - grp * tpt);
    if (n_tok <= 0) { g += n_tiles; continue; }                // the block has no second tile
    const int tl = token_of(c, r), M = n_tok * G, tok = it.q_tok0 + grp * tpt + tl;
    int4 vis = make_int4(0, 0, 0, 0);                          // padding rows see nothing
    if (r < M) vis = c.pd.tok_vis[tok];
    float m_ref = 0.f, l = 0.f;                                 // see the one-tile variant: the reference starts at 0
    bool seen = r >= M;                                         // padding rows never need the tracking pass
    bool warp_seen = false;                                     // all rows of the warp have (kept up in the full path only)
    for (int t = 0; t < n_tiles; ++t, ++g) {
      const int npg = min(8, it.n_pages - t * 8), halves = npg > 4 ? 2 : 1;
      dead |= !mbar_wait(bar_sfull, sc[0] & 1, ab);
      // The tile's page entries.  (The K producer cannot have come to tile g + kPageRingW2 meanwhile: V tile g + 2 waits
      // for this group's P.V of tile g, group 0's scores of tile g + 3 for its own P.V of tile g + 2, and K tile g + 5
      // for those.)
      int ye8[8];
      {
        const int4* yp = reinterpret_cast<const int4*>(&misc->nval[g & (kPageRingW2 - 1)][0]);
        const int4 ya = yp[0], yb = yp[1];
        ye8[0] = ya.x; ye8[1] = ya.y; ye8[2] = ya.z; ye8[3] = ya.w; ye8[4] = yb.x; ye8[5] = yb.y; ye8[6] = yb.z; ye8[7] = yb.w;
      }
      // Most halves lie wholly inside what every row of the warp may see (the prefix, full pages): the
      // warp then takes the pass without any mask arithmetic.  Both halves' verdicts are taken here.
      const int kbt = it.key0 + t * kTile;
      const bool plain0 = r >= M || (kbt + 64 <= vis.x && (ye8[0] & 255) + (ye8[1] & 255) + (ye8[2] & 255) + (ye8[3] & 255) == 64);
      const bool plain1 = r >= M || (kbt + 128 <= vis.x && (ye8[4] & 255) + (ye8[5] & 255) + (ye8[6] & 255) + (ye8[7] & 255) == 64);
      const bool masked0 = __any_sync(0xffffffffu, !plain0), masked1 = __any_sync(0xffffffffu, !plain1);
      for (int h = 0; h < halves; ++h, ++hc) {
        if (h > 0) dead |= !mbar_wait(bar_sfull + 8, sc[1] & 1, ab);    // h = 0: waited for above
        ++sc[h];
        tc_fence_after();
        if (tid == 0) ASPD_STAMP(c, g, 4 * h);
        uint32_t pk[32];
        float tile_sum, tmax;
        // p = 2^(s * scale - ref) for the thread's 64 scores of this half.  The common pass does not
        // track the largest exponent: packed fp32 pairs (one FFMA and one FADD per two scores), the
        // exponentials, the bf16 pairs.  An exponent beyond 2^40 shows in the sum; the tracking pass
        // then (and for rows that have not seen a key yet) finds the maximum.
        const int kb0 = kbt + h * 64;
        const bool masked = h ? masked1 : masked0;
        auto pass_impl = [&](float ref, auto track_tag, auto masked_tag) {
          constexpr bool TRACK = decltype(track_tag)::value, MASKED = decltype(masked_tag)::value;
          float mx0 = -INFINITY, mx1 = -INFINITY;
          float2 sum0 = make_float2(0.f, 0.f), sum1 = sum0, sum2 = sum0, sum3 = sum0;
          const float2 sc2 = make_float2(c.scale_log2, c.scale_log2), nb2 = make_float2(-ref, -ref);
          float s0[32], s1[32];
          ASPD_TMEM_LD32(s_base + h * 64, s0, 0);
          tmem_wait_ld32(s0);
          ASPD_TMEM_LD32(s_base + h * 64 + 32, s1, 0);        // on its way beside the arithmetic of the first 32
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            if (ch == 1) tmem_wait_ld32(s1);
            const float (&s)[32] = ch ? s1 : s0;
#pragma unroll
            for (int pg = 0; pg < 2; ++pg) {
              const int nv = (h ? ye8[4 + ch * 2 + pg] : ye8[ch * 2 + pg]) & 255;
              const int kb = kb0 + ch * 32 + pg * 16;
              uint32_t mask = 0xFFFFu;
              if constexpr (MASKED) mask = bits_between(0, min(nv, vis.x - kb)) | bits_between(vis.y - kb, min(nv, vis.z - kb));
#pragma unroll
              for (int i = 0; i < 16; i += 4) {
                float2 x0 = __ffma2_rn(make_float2(s[pg * 16 + i], s[pg * 16 + i + 1]), sc2, nb2);
                float2 x1 = __ffma2_rn(make_float2(s[pg * 16 + i + 2], s[pg * 16 + i + 3]), sc2, nb2);
                if (MASKED && mask != 0xFFFFu) {
                  x0.x = (mask >> i) & 1u ? x0.x : -INFINITY;
                  x0.y = (mask >> (i + 1)) & 1u ? x0.y : -INFINITY;
                  x1.x = (mask >> (i + 2)) & 1u ? x1.x : -INFINITY;
                  x1.y = (mask >> (i + 3)) & 1u ? x1.y : -INFINITY;
                }
                if constexpr (TRACK) { mx0 = fmaxf(mx0, fmaxf(x0.x, x0.y)); mx1 = fmaxf(mx1, fmaxf(x1.x, x1.y)); }
                x0.x = ex2(x0.x); x0.y = ex2(x0.y); x1.x = ex2(x1.x); x1.y = ex2(x1.y);
                if (i & 4) { sum2 = __fadd2_rn(sum2, x0); sum3 = __fadd2_rn(sum3, x1); }
                else       { sum0 = __fadd2_rn(sum0, x0); sum1 = __fadd2_rn(sum1, x1); }
                pk[ch * 16 + pg * 8 + (i >> 1)] = pack_bf16(x0.x, x0.y);
                pk[ch * 16 + pg * 8 + (i >> 1) + 1] = pack_bf16(x1.x, x1.y);
              }
            }
          }
          const float2 st = __fadd2_rn(__fadd2_rn(sum0, sum1), __fadd2_rn(sum2, sum3));
          tile_sum = st.x + st.y;
          tmax = fmaxf(mx0, mx1);
        };
        auto pass = [&](float ref, auto track_tag) {
          if (masked) pass_impl(ref, track_tag, std::true_type());
          else pass_impl(ref, track_tag, std::false_type());
        };
        // The common case -- every row of the warp has seen a key and no exponent passed 2^40 -- is
        // the plain pass and one vote; everything else goes the full way.
        bool settled = false;
        if (warp_seen) {
          pass(m_ref, std::false_type());
          // an exponent beyond 2^40 makes the sum exceed it (the converse is harmless: one more pass)
          settled = !__any_sync(0xffffffffu, !(tile_sum <= kRaiseSumW2));
        }
        if (!settled) {
          pass(m_ref, std::true_type());
          // move the reference: up when an exponent passed 2^40; down only while the row has not seen a
          // key yet (l and its row of O are still exactly 0 then, so nothing is rescaled)
          const bool raise = tmax > kRaiseW2, lower = !seen && tmax < -kLower && tmax > -INFINITY;
          const bool upd = raise || lower;
          seen |= tmax > -INFINITY;
          warp_seen = !__any_sync(0xffffffffu, !seen);
          float alpha = 1.f;
          if (raise) alpha = ex2(-tmax);
          if (upd) m_ref += tmax;
          l *= alpha;
          if (__any_sync(0xffffffffu, upd)) {
            if (t > 0 || h > 0) {                     // the rows' O so far is rescaled in TMEM (the warp together)
              dead |= !mbar_wait(bar_pvdone, (hc - 1) & 1, ab);      // the P.V of the previous half is done
              tc_fence_after();
#pragma unroll 1
              for (int q4 = 0; q4 < 4; ++q4) {
                float o[32];
                ASPD_TMEM_LD32(o_base + q4 * 32, o, 0);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] *= alpha;
                ASPD_TMEM_ST32(o_base + q4 * 32, o, 0);
              }
              tmem_wait_st();
            }
            pass(m_ref, std::false_type());           // the whole warp again (TMEM loads are warp-wide)
          }
        }
        l += tile_sum;
        if (tid == 0) ASPD_STAMP(c, g, 4 * h + 1);
        // the half's P (64 bf16 = 32 columns) over its own scores, which nobody needs any more: the next
        // scores go there behind the P.V that reads it, from the same issuer
        ASPD_TMEM_ST32U(s_base + h * 64, pk, 0);
        tmem_wait_st();
        tc_fence_before();
        warp_arrive_w2(bar_pfull + 8 * h);
        if (tid == 0) ASPD_STAMP(c, g, 4 * h + 2);
      }
    }
    // ---- the next query tile, so that its scores are made beside the rest of this item (the old one is free: all of
    // the group's scores are there)
    next_item(idx + 1);
    // ---- the row is complete: normalise and store it.  A warp's 32 rows go through shared memory by half rows, so
    // that eight lanes write 128 consecutive bytes.
    dead |= !mbar_wait(bar_ofull, ic & 1, ab);
    tc_fence_after();
    ++ic;
    {
      const float inv_l = l > 0.f ? 1.f / l : 0.f;
      const int rw0 = (warp & 3) * 32, ch = lane & 7;
      __nv_bfloat16* out0 = c.out + ((size_t)(it.q_tok0 + grp * tpt) * c.n_q_heads + it.kv_head * G) * 128 + ch * 8;
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int q2 = 0; q2 < 2; ++q2) {
          float o[32];
          ASPD_TMEM_LD32(o_base + half * 64 + q2 * 32, o, 0);
          tmem_wait_ld32(o);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(obuf + lane * 128 + (((q2 * 4 + i) ^ (lane & 7)) << 4)),
                         "r"(pack_bf16(o[8 * i] * inv_l, o[8 * i + 1] * inv_l)), "r"(pack_bf16(o[8 * i + 2] * inv_l, o[8 * i + 3] * inv_l)),
                         "r"(pack_bf16(o[8 * i + 4] * inv_l, o[8 * i + 5] * inv_l)), "r"(pack_bf16(o[8 * i + 6] * inv_l, o[8 * i + 7] * inv_l))
                         : "memory");
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int rl = k * 4 + (lane >> 3), ro = rw0 + rl;
          uint4 x;
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                       : "r"(obuf + rl * 128 + ((ch ^ (rl & 7)) << 4)) : "memory");
          if (ro < M && !dead) *reinterpret_cast<uint4*>(out0 + (size_t)(token_of(c, ro) * (c.n_q_heads - G) + ro) * 128 + half * 64) = x;
        }
        __syncwarp();
      }
      tc_fence_before();
    }
    if (named_sync_or(1 + grp, 128, dead || *ab)) break;
  }
}


__global__ void __launch_bounds__(kThreadsW2, 1) attn_tc_w2_kernel(Ctx c) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  MiscW2* misc = reinterpret_cast<MiscW2*>(smem + W2_OFF_MISC);
  const uint32_t bars = base + W2_OFF_MISC;       // bars[] is the first member
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  volatile int* ab = &misc->abort_flag;
  if (tid == 0) ASPD_CTA_STAMP(c, 0);
  if (tid == 0) pdl_launch_dependents();
  const int4 head = c.pd.cta_head[2 * blockIdx.x];
  const int item_begin = uniform(head.x), item_end = uniform(head.y);
  int2 first_pages = make_int2(0, 0);
  if ((warp == W2_KPROD || warp == W2_VPROD) && lane < head.w) first_pages = c.pd.visit[head.z + lane];
  {
    const int n_cached = min(item_end - item_begin, kItemCacheW2);
    for (int e = tid; e < n_cached * (int)(sizeof(DeviceItem) / 4); e += kThreadsW2)
      reinterpret_cast<int*>(misc->items)[e] = reinterpret_cast<const int*>(c.pd.items + item_begin)[e];
  }
  if (tid == 0) {
    //                               K_FULL K_EMPTY V_FULL V_EMPTY S_FULL(4)    P_FULL(4)   PV_DONE O_FULL Q_FULL
    const int counts[W2_NUM_BARS] = {1, 1,  2, 2,   1, 1,  2, 2,   1, 1, 1, 1,  4, 4, 4, 4, 1, 1,   1, 1,  4, 4};
    for (int i = 0; i < W2_NUM_BARS; ++i) mbar_init(bars + 8 * i, counts[i]);
    misc->abort_flag = 0;
    misc->lead = item_begin;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&misc->tmem_base)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc->tmem_base;
  const int G = c.G, tpt = 128 / G;      // tokens per query tile
  // inputs written by earlier kernels of the stream are used from here on; with the plan's
  // stable-cache promise the producers go ahead (such plans never carry new rows in their pages'
  // entries only when the step was appended by an earlier kernel: they wait before the first such page)
  const bool producer_runs_ahead = c.early_fetch && (warp == W2_KPROD || warp == W2_VPROD);
  if (!producer_runs_ahead) pdl_wait();
  if (tid == 0) ASPD_CTA_STAMP(c, 1);

  if (warp < 8) {
    softmax_group_w2(c, misc, bars, base, tmem, item_begin, item_end, warp >> 2, tpt);
  } else if (warp == W2_KPROD || warp == W2_VPROD) {
    // ================================ bulk-copy producers (as in the other variants) ================================
    const int kv = warp == W2_KPROD ? 0 : 1;
    const char* pool = kv ? c.v_pool : c.k_pool;
    int g = 0;
    bool ok = true, waited = false;
    int2 nxt = first_pages;
    for (int idx = item_begin; idx < item_end && ok; ++idx) {
      const DeviceItem it = get_item_w2(c, misc, idx, item_begin);
      const int n_tiles = (it.n_pages + 7) >> 3;
      int2 cur = make_int2(0, 0);
      for (int t = 0; t < n_tiles && ok; ++t, ++g) {
        if ((t & 3) == 0) {
          cur = nxt;
          nxt = make_int2(0, 0);
          const int ahead = (t + 4) * 8 + lane;
          if ((t + 4) * 8 < it.n_pages) {
            if (ahead < it.n_pages) nxt = c.pd.visit[it.page0 + ahead];
          } else if (idx + 1 < item_end) {          // first batch of the next item
            const DeviceItem nx = get_item_w2(c, misc, idx + 1, item_begin);
            if (lane < nx.n_pages) nxt = c.pd.visit[nx.page0 + lane];
          }
        }
        const int npg = min(8, it.n_pages - t * 8), sl = g & 1;
        int2 pg;
        pg.x = __shfl_sync(0xffffffffu, cur.x, (t & 3) * 8 + (lane & 7));
        pg.y = __shfl_sync(0xffffffffu, cur.y, (t & 3) * 8 + (lane & 7));
        if (lane >= npg) pg = make_int2(0, 0);
        if (lane < npg && !bounds_ok(c.pd, pg.x, 0, 16)) pg.x = 0;
        if (producer_runs_ahead && !waited && __any_sync(0xffffffffu, ((pg.y >> 8) & 31) != 0)) {
          pdl_wait();                                  // new rows come from the previous kernel
          waited = true;
        }
        const uint32_t full = bars + 8 * ((kv ? WV_FULL : WK_FULL) + sl), empty = bars + 8 * ((kv ? WV_EMPTY : WK_EMPTY) + sl);
        int good = 1;
        if (lane == 0) good = mbar_wait(empty, ((g >> 1) & 1) ^ 1, ab) ? 1 : 0;
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) { ok = false; break; }
        if (lane == 0) ASPD_STAMP(c, g, 13 + kv);
        if (kv == 0 && lane < 8) misc->nval[g & (kPageRingW2 - 1)][lane] = pg.y;   // read by the softmax groups of tile g
        __syncwarp();
        if (lane == 0) mbar_expect_tx(full, (uint32_t)npg * 4096u);
        __syncwarp();
        if (lane < npg)
          bulk_copy(base + (kv ? W2_OFF_V : W2_OFF_K) + sl * kTileBytes + lane * 4096,
                    pool + ((size_t)pg.x * c.n_kv_heads + it.kv_head) * 4096, 4096, full);
      }
    }
  } else {
    // ================================ MMA issuers (warp 10: group 0, warp 11: group 1) ================================
    // One warp per group, one cursor, operations in the order the operands come: the P.V of a half as soon as its P
    // is there, the next scores right behind the P.V that frees their columns.  Scores that overwrite P have no word that
    // the P.V has read it: they rest on the tensor pipe's taking the MMAs of one thread in the order that it issues them.
    // PTX names that order for MMAs of one shape into one accumulator; for these two, which differ in both, it is how the
    // pipe works, and what attention kernels with P over its scores commonly rest on.  (A wait for the P.V there: 24.6
    // instead of 22.4 ms a pass.)  All lanes wait
    // (suspending), lane 0 issues: a warp that diverges around a wait, or polls, spends more cycles on asking
    // than the operations take.
    const int grp = warp - W2_ISSUE;
    const uint32_t fm = 0xffffffffu;
    const uint32_t tmem_u = __shfl_sync(fm, tmem, 0), base_u = __shfl_sync(fm, base, 0), bars_u = base_u + W2_OFF_MISC;
    const int ib = item_begin, ie = item_end;
    auto wait_all = [&](uint32_t bar, uint32_t parity) { return __all_sync(fm, mbar_wait(bar, parity, ab)) != 0; };
    // A parity only tells the two latest phases of a barrier apart.  Group 1 is absent from items with
    // a single query tile, so its cursor may come to an item that group 0 has not reached yet and
    // would then take an older phase of a K or V barrier for its own: it holds until group 0's cursor
    // has reached the item (group 0's warp publishes how far it is).
    volatile int* lead = &misc->lead;
    const uint32_t idesc_pv = instr_desc(128, 1);
    const uint32_t s_tmem = tmem_u + COL_S + grp * 128, o_tmem = tmem_u + COL_O + grp * 128;
    const uint64_t adesc_q = smem_desc(base_u + W2_OFF_Q + grp * kTileBytes, 16, 1024);
    const uint32_t bar_sfull = bars_u + 8 * (WS_FULL + 2 * grp), bar_pfull = bars_u + 8 * (WP_FULL + 2 * grp), bar_pvdone = bars_u + 8 * (WPV_DONE + grp);
    int gbase = 0, ic = 0, cnt_p[2] = {0, 0};        // tiles so far; the group's items and P halves (first / second) so far
    bool ok = true;
    for (int idx = ib; idx < ie && ok; ++idx) {
      const DeviceItem it = get_item_w2(c, misc, idx, ib);
      const int n_pages = it.n_pages, n_q_tok = it.n_q_tok, n_tiles = (n_pages + 7) >> 3;
      if (n_q_tok > grp * tpt) {
        const bool both = n_q_tok > tpt;
        // a K or V tile is free when both groups are through with it; a group that is absent has its share done here
        auto release = [&](uint32_t bar) {
          tc_commit_lane0(bar);
          if (!both && lane == 0) mbar_arrive(bar);
        };
        auto k_there = [&](int t) { return wait_all(bars_u + 8 * (WK_FULL + ((gbase + t) & 1)), ((gbase + t) >> 1) & 1); };
        auto issue_s = [&](int t, int h) {             // scores of keys [64 h, 64 h + 64) of tile t
          const int g = gbase + t, sb = g & 1, npg = min(8, n_pages - t * 8);
          const uint32_t idesc_s = instr_desc((uint32_t)min(4, npg - 4 * h) * 16u, 0);
          if (lane == 0 && grp == 0) ASPD_STAMP(c, g, 8 + h);
          tc_mma_ss_k128_lane0<kHalf, 1024>(s_tmem + h * 64, adesc_q, smem_desc(base_u + W2_OFF_K + sb * kTileBytes + h * 16384, 16, 2048), idesc_s);
          tc_commit_lane0(bar_sfull + 8 * h);
          if (h == 1 || npg <= 4) release(bars_u + 8 * (WK_EMPTY + sb));
        };
        if (grp == 1) {
          const long long t0 = clock64();
          while (ok && __shfl_sync(fm, *lead, 0) < idx) {
            __nanosleep(100);
            if (__shfl_sync(fm, (*ab || clock64() - t0 > kWaitCycles) ? 1 : 0, 0)) { *ab = 1; ok = false; }
          }
        }
        ok = ok && wait_all(bars_u + 8 * (WQ_FULL + grp), ic & 1);
        ++ic;
        ok = ok && k_there(0);
        if (!ok) break;
        tc_fence_after();
        issue_s(0, 0);
        if (n_pages > 4) issue_s(0, 1);
        for (int t = 0; t < n_tiles && ok; ++t) {
          const int g = gbase + t, npg = min(8, n_pages - t * 8), halves = npg > 4 ? 2 : 1;
          const uint32_t vbuf = base_u + W2_OFF_V + (g & 1) * kTileBytes;
          const int npg1 = min(8, n_pages - t * 8 - 8);          // pages of the next tile
          // what is usually there is waited for first, so that a half's P is all that its operations still need
          ok = wait_all(bars_u + 8 * (WV_FULL + (g & 1)), (g >> 1) & 1) && (npg1 <= 0 || k_there(t + 1));
          for (int h = 0; h < halves && ok; ++h) {
            ok = wait_all(bar_pfull + 8 * h, cnt_p[h] & 1);
            ++cnt_p[h];
            if (!ok) break;
            tc_fence_after();
            if (lane == 0 && grp == 0) ASPD_STAMP(c, g, 10 + h);
            // 16 keys = one page per k-step
            tc_mma_ts_pv_lane0(o_tmem, s_tmem + h * 64, smem_desc(vbuf + 4 * h * 4096, 1024, 2048), idesc_pv, (t > 0 || h > 0) ? 1u : 0u, min(4, npg - 4 * h));
            // (Asked for only when a row's reference moves.  Before the word of the scores behind it, which send the group
            // two halves on, and before O's: a group that waits for half hc - 1 then knows that half hc - 2 is through,
            // and the parity tells the two apart.)
            tc_commit_lane0(bar_pvdone);
            if (npg1 > 4 * h) issue_s(t + 1, h);
            if (h == halves - 1) {
              if (t == n_tiles - 1) tc_commit_lane0(bars_u + 8 * (WO_FULL + grp));
              release(bars_u + 8 * (WV_EMPTY + (g & 1)));
            }
          }
        }
        if (grp == 0 && lane == 0) *lead = idx + 1;
      } else if (grp == 0 && lane == 0) *lead = idx + 1;
      gbase += n_tiles;
    }
    if (grp == 0 && lane == 0) *lead = ie;
    __syncwarp();
  }

  // ---- drain: on a time-out give outstanding copies and MMAs time to land before the CTA's
  // shared memory and TMEM go away
  if (*ab) {
    if (tid == 0) atomicCAS(c.pd.status, 0, (int)ASPD_ERR_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0) ASPD_CTA_STAMP(c, 3);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

}  // namespace

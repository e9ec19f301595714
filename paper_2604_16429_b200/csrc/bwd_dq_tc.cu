// dQ of the block-sparse attention backward on Blackwell tensor cores (tcgen05 + TMEM + TMA).
//
// Paper, appendix "Block-sparse attention implementation", paragraph "Kernel Design": the backward
// recomputes the probabilities from the saved log-sum-exp instead of storing the attention matrix, and
// the query gradient is query-block stationary with the same traversal as the forward.
//   P = exp(scale * Q K^T - LSE),  dP = dO V^T,  dS = P o (dP - D),  dQ = scale * dS K,
// D = rowsum(dO o O) from the preprocessing kernel; the selection is a constant of the backward.
//
// Same work decomposition as the forward kernel: a persistent CTA per SM draws 256-row items (two
// 128-row tiles, four 64-row halves) from a queue; a planner warp merges the key lists of the item's
// query blocks; a producer warp streams 64-token K and V chunks through a ring; one warp per tile issues
// the tensor-core work; two groups of four warps (thread = query row = TMEM lane) turn S and dP into dS.
// Per product and tile: S = Q K^T and dP = dO V^T (eight MMAs into two 64-column TMEM buffers); the row
// threads pull both into registers and hand the buffers back at once, so the next product's S and dP are
// computed while they form dS (bf16, two buffers of 32 TMEM columns in turn); then dQ += dS K (dS is the TMEM A operand,
// the K chunk in shared memory is read as the MN-major B operand), issued one product behind.
// BR, the three-branch form: a list entry carries a mask of the halves that attend it locally and one of those that selected
// it; the row threads take the matching statistics, gate and dO share, so one launch serves both branches, and the epilogue adds the
// block level's share (with two launches, their sum in a third: 254 + 20 us at 8 units of 28800 tokens, now 188).
// Bound by the row threads' queue of MUFU, shared-memory and TMEM instructions, in which a wait on a completed barrier takes
// 150 to 250 cycles: a second dS buffer, which saves one, and cheaper polls took 64 units of 28800 tokens from 1401 to 1151 us.
// With 64-token blocks the producer counts too: with its whole warp at work 8 units of 28800 tokens take 174 us instead of 178.
// Every mbarrier wait is bounded; on expiry the CTA records MOSAIC_E_DEVICE_TIMEOUT and drains.
#include "tc_common.cuh"

namespace mosaic {

namespace {

constexpr int kStages = 6;       // key/value ring depth (K + V chunk per stage)
constexpr int kThreads = 384;
constexpr uint32_t kTmemCols = 512;
// dQ of tile t at 64 t; S of tile t at 128 + 128 t, dP right after it; dS buffer b (bf16) of tile t at 384 + 64 t + 32 b
constexpr uint32_t kColDQ = 0, kColS = 128, kColDS = 384;

struct Smem {
  unsigned char q[2][2 * kTile];           // [tile][128 rows x 128 B]
  unsigned char d_o[2][2 * kTile];         // [tile][128 rows x 128 B]
  unsigned char kv[kStages][2][kTile];     // [stage][K, V]
  unsigned long long kv_full[kFullBars], kv_empty[kStages];
  unsigned long long q_full[2], q_empty[2], s_full[2], sdp_free[2];  // [tile]
  unsigned long long p_full[2][2], pv_done[2][2];  // [tile][dS buffer]
  unsigned long long mma_drain_bar[2];  // abort path: completion of each issuer's outstanding products
  unsigned long long list_full[kLists], list_empty[kLists];
  uint32_t tmem_base;
  int abort;
  RowItem info[kLists];
  alignas(16) int ids[kLists][kMaxUnion];
  unsigned char mask[kLists][kMaxUnion];
  unsigned short steps[kLists][2][kMaxUnion];  // [list][tile]
  alignas(16) int tmp_ids[kMaxUnion];            // planner scratch: merged list before reordering
  unsigned char tmp_mask[kMaxUnion];
};

static_assert(kFullBars >= kMaxUnion + kStages && (kFullBars & (kFullBars - 1)) == 0, "a list's chunks land on barriers of their own");

}  // namespace

// BR: backward of the three-branch form.  The local and the selected blocks have a softmax of their own, so a row has two
// sets of statistics and its dO is scaled by the branch's gate: dS = P (gate dP - gate <dO, O>); the block's share from
// the compression branch (dqm) is added at the end.
template <bool F16, bool BR>
__global__ void __launch_bounds__(kThreads, 1)
    dq_tc_kernel(const Geo g, const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_do,
                 const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                 const int32_t* __restrict__ block_idx, const RowStats st, __nv_bfloat16* __restrict__ dq, int* status,
                 int* work_counter, int ipu, const Queue queue) {
  extern __shared__ unsigned char smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(s32(&sm.kv_empty[s]), 2);
    for (int t = 0; t < 2; ++t) {
      mbar_init(s32(&sm.q_full[t]), 1);
      mbar_init(s32(&sm.q_empty[t]), 1);
      mbar_init(s32(&sm.mma_drain_bar[t]), 1);
      mbar_init(s32(&sm.s_full[t]), 1);
      mbar_init(s32(&sm.sdp_free[t]), 128);
      mbar_init(s32(&sm.p_full[t][0]), 128);
      mbar_init(s32(&sm.p_full[t][1]), 128);
      mbar_init(s32(&sm.pv_done[t][0]), 1);
      mbar_init(s32(&sm.pv_done[t][1]), 1);
    }
    for (int i = 0; i < kLists; ++i) {
      mbar_init(s32(&sm.list_full[i]), 1);
      mbar_init(s32(&sm.list_empty[i]), 11);  // 8 row-thread warps + 2 MMA warps + TMA producer
    }
    sm.abort = 0;
  }
  for (int s = tid; s < kFullBars; s += kThreads) mbar_init(s32(&sm.kv_full[s]), 1);
  cta_publish_barriers();
  block_idx += await_stream();  // before the TMEM is taken: a kernel ahead may still need it
  const uint32_t tmem = cta_tmem_alloc(warp == 9, &sm.tmem_base, kTmemCols);
  volatile int* abort = &sm.abort;

  if (warp == 11) {
    planner_loop<BR ? kPlanTagged : kPlanUnion>(sm, g, block_idx, work_counter, ipu, queue, lane, abort, status);
  } else if (warp == 8) {
    // ------------------------------------------------------------- TMA producer
    uint32_t step = 0;   // key/value chunks issued so far (ring position)
    int q_armed[2] = {-1, -1};  // phase parity of the last load into each tile's Q / dO buffer
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int buf = it % kLists;
      ok = warp_wait(s32(&sm.list_full[buf]), (it / kLists) & 1, abort, status);
      if (!ok) break;
      const RowItem& inf = sm.info[buf];
      const int n = inf.n, u = inf.unit;
      if (n < 0) break;
      // Q and dO tiles: free once the tile's last S / dP products of the previous item have completed
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (ok) ok = warp_wait(s32(&sm.q_empty[t]), (it & 1) ^ 1, abort, status);
        if (!ok) break;
        q_armed[t] = it & 1;
        if (elect_one()) {
          mbar_expect_tx(s32(&sm.q_full[t]), 4 * kTile);
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const int x = inf.hx[2 * t + hh], y = inf.hy[2 * t + hh];
            tma_load_4d(s32(sm.q[t] + hh * kTile), &map_q, s32(&sm.q_full[t]), 0, x, y, u);
            tma_load_4d(s32(sm.d_o[t] + hh * kTile), &map_do, s32(&sm.q_full[t]), 0, x, y, u);
          }
        }
        __syncwarp();
      }
      // (key/value head of this query head's group)
      if (ok) ok = produce_chunks<kStages>(sm, g, &map_k, &map_v, buf, n, kv_unit(g, u), step, lane, abort, status);
      if (ok && elect_one()) mbar_arrive(s32(&sm.list_empty[buf]));
    }
    if (lane == 0) {
      if (*abort) {  // copies this warp issued must land before the CTA's memory is released
        const uint32_t first = step > kStages ? step - kStages : 0;
        for (uint32_t s = first; s < step; ++s) mbar_drain(s32(&sm.kv_full[s % kFullBars]), (s / kFullBars) & 1);
        for (int t = 0; t < 2; ++t)
          if (q_armed[t] >= 0) mbar_drain(s32(&sm.q_full[t]), (uint32_t)q_armed[t]);
      } else {       // drain: the last uses of every ring stage have been released by both tiles
        const uint32_t first = step > kStages ? step - kStages : 0;
        for (uint32_t s = first; s < step; ++s)
          if (!mbar_wait(s32(&sm.kv_empty[s % kStages]), (s / kStages) & 1, abort, status)) break;
      }
    }
  } else if (warp == 9 || warp == 10) {
    // ------------------------------------------------------------- MMA issuer of tile t
    // The whole warp walks the loop; one elected lane issues the tensor-core instructions.
    const int t = warp - 9;
    constexpr uint32_t idesc_nt = make_idesc(false, 64u, F16), idesc_nn = make_idesc(true, 64u, F16);
    const uint64_t qdesc = smem_desc(s32(sm.q[t])), dodesc = smem_desc(s32(sm.d_o[t]));
    const uint32_t tcol_dq = tmem + kColDQ + 64 * t, tcol_s = tmem + kColS + 128 * t, tcol_dp = tcol_s + 64;
    const uint32_t tcol_ds = tmem + kColDS + 64 * t;
    uint32_t base = 0;    // ring position of the item's first chunk
    uint32_t nt = 0;      // products started by this tile so far (phase of the per-product barriers)
    bool ok = true;
    // dQ += dS K of the product whose K chunk sits in ring stage `pst` (the previous product of this tile)
    auto issue_dq = [&](int pst, bool pfirst) {
      ok = warp_wait(s32(&sm.p_full[t][(nt - 1) & 1]), ((nt - 1) >> 1) & 1, abort, status);
      if (!ok) return;
      tc_fence_after();
      const uint64_t kmn = smem_desc(s32(sm.kv[pst][0]));
      const uint32_t dscol = tcol_ds + 32 * ((nt - 1) & 1);
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_ts(tcol_dq, dscol + 8 * kk, kmn + (uint64_t)((2048 * kk) >> 4), idesc_nn, (!pfirst || kk > 0));
        tc_commit(s32(&sm.kv_empty[pst]));
        tc_commit(s32(&sm.pv_done[t][(nt - 1) & 1]));
      }
      __syncwarp();
    };
    for (int it = 0; ok; ++it) {
      const int buf = it % kLists;
      ok = warp_wait(s32(&sm.list_full[buf]), (it / kLists) & 1, abort, status);
      if (!ok) break;
      const int n = sm.info[buf].n;
      if (n < 0) break;
      const int cnt = sm.info[buf].nsteps[t];
      // the tiles are loaded for every item; they must have landed before their buffers are handed back
      ok = warp_wait(s32(&sm.q_full[t]), it & 1, abort, status);
      if (!ok) break;
      if (cnt == 0 && elect_one()) mbar_arrive(s32(&sm.q_empty[t]));
      bool first = true, pend = false, pend_first = false;
      int pend_st = 0;
      uint32_t pend_step = 0;
      for (int i = 0; i < cnt && ok; ++i) {
        uint32_t step = base + (sm.steps[buf][t][i] >> 8) * (uint32_t)g.cpb;
        for (int c = 0; c < g.cpb && ok; ++c, ++step) {
          const uint32_t st = step % kStages;
          // across a long gap in the tile's entries the chunk only lands once the pending product frees its stage
          if (pend && step - pend_step >= (uint32_t)kStages) {
            issue_dq(pend_st, pend_first);
            pend = false;
            if (!ok) break;
          }
          ok = warp_wait(s32(&sm.kv_full[step % kFullBars]), (step / kFullBars) & 1u, abort, status);
          if (!ok) break;
          // S and dP may be overwritten once the row threads hold the previous product's values in registers
          if (nt > 0) {
            ok = warp_wait(s32(&sm.sdp_free[t]), (nt - 1) & 1, abort, status);
            if (!ok) break;
          }
          tc_fence_after();
          const uint64_t kdesc = smem_desc(s32(sm.kv[st][0])), vdesc = smem_desc(s32(sm.kv[st][1]));
          const bool release_q = i == cnt - 1 && c == g.cpb - 1;
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma_ss(tcol_s, qdesc + 2 * kk, kdesc + 2 * kk, idesc_nt, kk > 0);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma_ss(tcol_dp, dodesc + 2 * kk, vdesc + 2 * kk, idesc_nt, kk > 0);
            tc_commit(s32(&sm.s_full[t]));
            if (release_q) tc_commit(s32(&sm.q_empty[t]));
          }
          __syncwarp();
          if (pend) issue_dq(pend_st, pend_first);  // previous product: its dS is ready or about to be
          if (!ok) break;
          pend = true; pend_st = (int)st; pend_step = step; pend_first = first;
          first = false;
          ++nt;
        }
      }
      base += (uint32_t)(n * g.cpb);
      if (ok && pend) issue_dq(pend_st, pend_first);  // the item's last product
      if (ok && elect_one()) mbar_arrive(s32(&sm.list_empty[buf]));
    }
    if (*abort) {  // products already issued must finish before TMEM and shared memory are released
      if (elect_one()) mma_drain(s32(&sm.mma_drain_bar[t]));
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------- row threads of tile t: S, dP -> dS; then epilogue
    const int t = warp >> 2;        // tile
    const int hh = (warp >> 1) & 1; // 64-row half of the tile this warp's rows belong to
    const int h = 2 * t + hh;
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t ts = tmem + lane_off + kColS + 128 * t, tdp = ts + 64, tdq = tmem + lane_off + kColDQ + 64 * t;
    const uint32_t tds = tmem + lane_off + kColDS + 64 * t;
    const uint64_t scale2 = pack2(g.scale_log2, g.scale_log2);
    const int row_y = (tid & 63) / g.bw, row_x = (tid & 63) - row_y * g.bw;  // the row's place in its chunk
    uint32_t nt = 0;
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int buf = it % kLists;
      ok = warp_wait(s32(&sm.list_full[buf]), (it / kLists) & 1, abort, status);
      if (!ok) break;
      const int n = sm.info[buf].n;
      if (n < 0) break;
      const bool valid = (sm.info[buf].hvalid >> h) & 1;
      const long long tok =
          (long long)sm.info[buf].unit * g.N + (long long)(sm.info[buf].hy[h] + row_y) * g.nlon + sm.info[buf].hx[h] + row_x;
      // negated log-sum-exp (in base-2 units), negated D and gate of this thread's query row, per branch
      float nl[2], nd[2], gt[2];
#pragma unroll
      for (int x = 0; x < (BR ? 2 : 1); ++x) {
        const long long at = (x ? (long long)g.U * g.N : 0) + tok;
        nl[x] = valid ? __ldg(st.neg_lse2 + at) : 0.f;
        nd[x] = valid ? __ldg(st.neg_d + at) : 0.f;
        gt[x] = BR && valid ? __ldg(st.gate + at) : 0.f;
      }
      uint64_t neg_lse2 = pack2(nl[0], nl[0]), neg_d2 = pack2(nd[0], nd[0]), gate2 = pack2(gt[0], gt[0]);
      const int cnt = sm.info[buf].nsteps[t];
      const unsigned short* steps = sm.steps[buf][t];
      for (int i0 = 0; i0 < cnt && ok; ++i0) {
        const uint32_t code = steps[i0];
        const bool attends = (code >> hh) & 1u;
        if (BR) {
          const bool sel = (code >> (2 + hh)) & 1u;
          const float a = sel ? nl[1] : nl[0], b = sel ? nd[1] : nd[0], c = sel ? gt[1] : gt[0];
          neg_lse2 = pack2(a, a);
          neg_d2 = pack2(b, b);
          gate2 = pack2(c, c);
        }
        for (int c = 0; c < g.cpb; ++c) {
          ok = warp_wait(s32(&sm.s_full[t]), nt & 1, abort, status);
          if (!ok) break;
          tc_fence_after();
          uint32_t pk[32];
          if (attends) {
            // all 64 + 64 values into registers, then S and dP are handed back to the tensor core at once
            uint32_t sv[64], dp[64];
            tmem_ld32(ts, *reinterpret_cast<uint32_t(*)[32]>(&sv[0]));
            tmem_ld32(ts + 32, *reinterpret_cast<uint32_t(*)[32]>(&sv[32]));
            tmem_ld32(tdp, *reinterpret_cast<uint32_t(*)[32]>(&dp[0]));
            tmem_ld32(tdp + 32, *reinterpret_cast<uint32_t(*)[32]>(&dp[32]));
            tmem_wait_ld();
            tc_fence_before();
            mbar_arrive(s32(&sm.sdp_free[t]));
#pragma unroll
            for (int i = 0; i < 64; i += 2) {
              float x0, x1, d0, d1;
              unpack2(fma2(pack2(__uint_as_float(sv[i]), __uint_as_float(sv[i + 1])), scale2, neg_lse2), x0, x1);
              const uint64_t dp2 = pack2(__uint_as_float(dp[i]), __uint_as_float(dp[i + 1]));
              const uint64_t dmd = BR ? fma2(dp2, gate2, neg_d2) : add2(dp2, neg_d2);
              unpack2(mul2(pack2(ex2(x0), ex2(x1)), dmd), d0, d1);
              pk[i >> 1] = pack2<F16>(d0, d1);
            }
          } else {
            tc_fence_before();
            mbar_arrive(s32(&sm.sdp_free[t]));
#pragma unroll
            for (int i = 0; i < 32; ++i) pk[i] = 0u;
          }
          // dS buffer nt & 1 was read by dQ += dS K of product nt - 2, issued before this product's S by the same warp, whose
          // commit for S therefore covers it: no wait
          tmem_st32(tds + 32 * (nt & 1), pk);
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive(s32(&sm.p_full[t][nt & 1]));
          ++nt;
        }
      }
      if (!ok) break;
      if (cnt > 0) {
        ok = warp_wait(s32(&sm.pv_done[t][(nt - 1) & 1]), ((nt - 1) >> 1) & 1, abort, status);
        if (!ok) break;
        tc_fence_after();
        if (valid) {
          uint4* dst = reinterpret_cast<uint4*>(dq + tok * kD);
#pragma unroll
          for (int part = 0; part < 2; ++part) {
            uint32_t ov[32];
            tmem_ld32(tdq + 32 * part, ov);
            tmem_wait_ld();
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(ov[i]) * g.scale;
            if (BR) {
              const float4* add = reinterpret_cast<const float4*>(
                  st.dqm + ((long long)sm.info[buf].unit * g.m + sm.info[buf].hb[h]) * kD + 32 * part);
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 x = __ldg(add + i);
                v[4 * i] += x.x; v[4 * i + 1] += x.y; v[4 * i + 2] += x.z; v[4 * i + 3] += x.w;
              }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
              dst[part * 4 + i] = make_uint4(pack2<F16>(v[8 * i], v[8 * i + 1]), pack2<F16>(v[8 * i + 2], v[8 * i + 3]),
                                             pack2<F16>(v[8 * i + 4], v[8 * i + 5]), pack2<F16>(v[8 * i + 6], v[8 * i + 7]));
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(s32(&sm.list_empty[buf]));
    }
  }
  cta_tmem_free(warp == 9, tmem, kTmemCols);
}

// `work_counter` must be zero when the kernel starts (a word of the workspace status block).
template <bool F16, bool BR>
static int launch_dq_tc_t(const HostCtx& c, const void* q, const void* k, const void* v, const void* d_o,
                          const RowStats& st, const int32_t* block_idx, void* dq, int* work_counter) {
  const Geo& g = c.g;
  CUtensorMap mq, mdo, mk, mv;
  if (!make_map(&mq, q, g, g.U) || !make_map(&mdo, d_o, g, g.U) || !make_map(&mk, k, g, g.Ukv) || !make_map(&mv, v, g, g.Ukv))
    return MOSAIC_E_CUDA;
  const size_t smem = sizeof(Smem) + 1024;
  static unsigned long long configured = 0;  // devices on which the kernel's shared-memory opt-in is set
  int sms = 0;
  if (const int rc = launch_setup(reinterpret_cast<const void*>(dq_tc_kernel<F16, BR>), smem, &configured, &sms)) return rc;
  const int ipu = items_per_unit(g);
  const long long total = (long long)g.U * ipu;
  if (total > 0x7fffff00ll) return MOSAIC_E_UNSUPPORTED;
  const Queue queue = make_queue(total, sms);
  const int grid = queue.positions < sms ? queue.positions : sms;
  return launch_kernel(dq_tc_kernel<F16, BR>, dim3((unsigned)grid), kThreads, smem, c.stream, true, 0, g, mq, mdo, mk, mv, block_idx,
                       st, (__nv_bfloat16*)dq, c.status, work_counter, ipu, queue);
}

int launch_dq_tc(const HostCtx& c, const void* q, const void* k, const void* v, const void* d_o, const RowStats& st,
                 const int32_t* block_idx, void* dq, int* work_counter) {
  if (st.gate)
    return c.g.f16 ? launch_dq_tc_t<true, true>(c, q, k, v, d_o, st, block_idx, dq, work_counter)
                   : launch_dq_tc_t<false, true>(c, q, k, v, d_o, st, block_idx, dq, work_counter);
  return c.g.f16 ? launch_dq_tc_t<true, false>(c, q, k, v, d_o, st, block_idx, dq, work_counter)
                 : launch_dq_tc_t<false, false>(c, q, k, v, d_o, st, block_idx, dq, work_counter);
}

}  // namespace mosaic

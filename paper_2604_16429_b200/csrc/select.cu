// Selection: block-level scores on the pooled sums, per-query-block top-k.
//
// Paper, section "Block-Sparse Attention": paragraph "Compression" defines the pooled block
// representations (phi = mean pooling) and the block-level score; paragraph "Selection" takes the
// top-n key blocks per query block.  The mean's 1/b, the 1/sqrt(d_k) and the row softmax are
// strictly increasing, so ranking the raw dot product of block SUMS gives the same blocks.
//
// Arithmetic is fixed so that the chosen ids are unique and reproducible bit for bit:
//   pooled sum  = fp64 accumulation over the block's tokens in row-major order, one rounding to fp32
//   score       = fp64 accumulation over channels 0..d-1 of the exact products of two fp32 values
//   order       = (score descending, block id ascending); +0 == -0; a NaN ranks last
#include "common.cuh"

namespace mosaic {

// ------------------------------------------------------------------------------------------
// topk_kernel<TI, CAP>: ranking of the key blocks of TI query blocks of one unit by a CTA of eight warps.
//
// The ids must be those of the exact fp64 scores, but almost all of the m scores of a row are irrelevant,
// so the kernel screens with tensor cores and scores exactly only what survives:
//   1. screening score  s~: the fp32 vectors are split into two bf16 parts each (a = ah + al + ea, |al| <= 2^-9 |a|,
//      |ea| <= 2^-18 |a| per channel) and s~ = ah.bh + ah.bl + al.bh by mma.sync with fp32 accumulation.  What is left
//      out (al.bl and the ea, eb terms) is at most 3 * 2^-18 (1 + 2^-8) |a||b| by Cauchy-Schwarz; twelve accumulation steps of
//      sixteen exact products, each step off by at most 17 * 2^-23 |a||b| even if it truncates, add 2^-15.3 |a||b|.
//      The kernel uses eps = 2^-14 * na * nb + 1e-37 with the norm bounds of the pooling kernel, 1.7 times the sum.  A
//      non-finite s~, and vectors so short that their parts may be subnormal, make the candidate's interval (-inf, +inf).
//   2. first pass: every lane keeps the largest lower bounds s~ - eps of its share of a row's keys; the k-th largest of
//      the row's 64 kept values is a lower bound thr of the row's k-th best exact score (they belong to k distinct
//      candidates).
//   3. second pass, the same products again: a candidate with s~ + eps < thr is worse than k others whatever the ties;
//      the rest (about 1.2 k of them) collect in shared memory.  A row whose survivors overflow (massive ties) falls back
//      to scoring every key exactly.
//   4. exact phase: the fp64 chain of the selection's definition for every survivor of the warp's rows (lanes take
//      survivors, two chains in flight each), then each row ranks its survivors by (score descending, id ascending) by
//      counting, and ranks 0..k-1 are written.
// Screening twice costs less than keeping a threshold current during one pass did: with FMAs on the CUDA cores, their
// operand loads (6 words per 8 FMAs) and the running thresholds a warp spent 1770 instructions on 4 rows x 64 keys; now
// about 200 per pass on 16 rows x 16 keys.
// What bounds it now is the split of the keys into parts and, for few rows, the chain of phases.  us, before -> after: 8 units
// of 450 blocks 38.7 -> 26.2, 192 units 528 -> 384, 8 units of 4050 blocks 1382 -> 798, 24 units of 384 blocks with top-k 24
// 136 -> 62.
// ------------------------------------------------------------------------------------------

// Total-order key: larger key = better score.  0 = not a candidate, 1 = NaN.
__device__ __forceinline__ unsigned long long score_key(double s) {
  if (s != s) return 1ull;
  s += 0.0;  // -0 -> +0
  unsigned long long b = (unsigned long long)__double_as_longlong(s);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// does (ka, ia) rank before (kb, ib)?
__device__ __forceinline__ bool ranks_before(unsigned long long ka, int ia, unsigned long long kb, int ib) {
  return ka > kb || (ka == kb && ia < ib);
}

// order-preserving map of non-NaN floats to unsigned integers
__device__ __forceinline__ unsigned ordered_bits(float f) {
  const unsigned b = __float_as_uint(f);
  return (b >> 31) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(unsigned o) {
  return __uint_as_float((o >> 31) ? (o & 0x7fffffffu) : ~o);
}

constexpr int kKStr = kD + 4;   // padded row of the staged vectors (floats): 16-byte reads of one row per lane hit every bank once

constexpr int kTW = 8;           // warps of a ranking CTA
constexpr int kTJ = 64;          // keys of a chunk
constexpr int kHStr = kD + 8;    // padded row of the split keys (16-bit elements): ldmatrix reads hit every bank once
constexpr int kTracked = 64;     // lower bounds kept per row

template <int TI, int CAP>
struct TopkSmem {
  union {
    struct {
      __nv_bfloat16 kh[2][2][kTJ][kHStr];  // [buffer][high part, low part][key][channel]
      float nk[2][kTJ];                    // norm bounds of the keys times 2^-14
    } scr;
    float tracked[TI][kTracked];           // between the passes
    unsigned long long ekey[TI][CAP];      // exact phase: score keys of the rows' survivors (rows that did not overflow)
  };
  float qs[TI][kKStr];   // pooled queries of this CTA
  float nq[TI], thr[TI];
  int cnt[TI];
  int surv[TI][CAP];     // surviving key ids per row
};

// a = high + low + rest: two floats into packed bf16 high parts and packed low parts
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The warp's sorted list of the best candidates so far holds one entry per lane (lane r = rank r).  Offers this
// lane's candidate (key 0 = none) together with those of the other lanes; every candidate that belongs to the k
// best is inserted.
__device__ __forceinline__ void insert_batch(unsigned long long key, int id, unsigned long long& lkey, int& lid, int k,
                                             int lane) {
  while (true) {
    // warp-wide best remaining candidate: maximum of the key's high word, then of the low word among the lanes
    // that hold that high word, then the lowest id among the lanes that hold the key
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const unsigned long long bk = ((unsigned long long)mh << 32) | ml;
    if (bk == 0ull) return;
    const int bj = (int)__reduce_min_sync(0xffffffffu, key == bk ? (unsigned)id : 0x7fffffffu);
    const unsigned long long tk = __shfl_sync(0xffffffffu, lkey, k - 1);
    const int ti = __shfl_sync(0xffffffffu, lid, k - 1);
    if (!(tk == 0ull || ranks_before(bk, bj, tk, ti))) return;  // the batch's best does not enter: nothing does
    const bool before = lkey != 0ull && ranks_before(lkey, lid, bk, bj);
    const int p = __popc(__ballot_sync(0xffffffffu, before));
    const unsigned long long uk = __shfl_up_sync(0xffffffffu, lkey, 1);
    const int ui = __shfl_up_sync(0xffffffffu, lid, 1);
    if (lane == p) { lkey = bk; lid = bj; }
    else if (lane > p) { lkey = uk; lid = ui; }
    if (key == bk && id == bj) key = 0ull;  // taken
  }
}

// exact score of (pooled query row in shared memory, pooled key row j in global memory) as a sortable key
__device__ __forceinline__ unsigned long long exact_key(const float* qrow, const float* __restrict__ pk_u, int j) {
  const float4* krow = reinterpret_cast<const float4*>(pk_u + (long long)j * kD);
  double s = 0.0;
#pragma unroll
  for (int half = 0; half < 2; ++half) {  // eight 16-byte loads in flight, then their 32 sequential FMAs
    float4 kv[kD / 8];
#pragma unroll
    for (int c4 = 0; c4 < kD / 8; ++c4) kv[c4] = __ldg(krow + half * (kD / 8) + c4);
#pragma unroll
    for (int c4 = 0; c4 < kD / 8; ++c4) {
      const float4 qv = *reinterpret_cast<const float4*>(qrow + 4 * (half * (kD / 8) + c4));
      s = fma((double)qv.x, (double)kv[c4].x, s);
      s = fma((double)qv.y, (double)kv[c4].y, s);
      s = fma((double)qv.z, (double)kv[c4].z, s);
      s = fma((double)qv.w, (double)kv[c4].w, s);
    }
  }
  return score_key(s);
}

template <int TI, int CAP>
__global__ void __launch_bounds__(kTW * 32, 2) topk_kernel(Geo g, const float* __restrict__ pq, const float* __restrict__ pk,
                                                           const float* __restrict__ nq, const float* __restrict__ nk,
                                                           int32_t* __restrict__ block_idx) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using SM = TopkSmem<TI, CAP>;
  SM& sm = *reinterpret_cast<SM*>(smem_raw);
  constexpr int RT = TI / 16;              // 16-row tiles of the products
  constexpr int NT8 = RT;                  // 8-key tiles per warp and chunk: the eight warps share RT x 8 of them
  constexpr int kDepth = kTracked * RT / 32;  // lower bounds a lane keeps per row (32 / RT lanes share a row)
  constexpr int RI = TI / kTW;             // rows per warp in the exact phase
  constexpr int NT = kTW * 32;
  const float kInf = __int_as_float(0x7f800000);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tiles = (g.m + TI - 1) / TI;
  const int cta = (int)blockIdx.x + await_stream();
  const int u = cta / tiles, i0 = (cta - u * tiles) * TI;
  const float* pq_u = pq + (long long)u * g.m * kD;
  const float* pk_u = pk + (long long)kv_unit(g, u) * g.m * kD;   // grouped-query attention: the group's key head
  const float* nk_u = nk + (long long)kv_unit(g, u) * g.m;
  const int nchunks = (g.m + kTJ - 1) / kTJ;

  // a chunk's keys: four threads per key, sixteen channels each, fetched into registers one chunk ahead
  float4 stage[4];
  float stage_n = 0.f;
  const int sj = tid >> 2, sc = 16 * (tid & 3);
  auto fetch = [&](int ch) {
    const int j = ch * kTJ + sj;
#pragma unroll
    for (int x = 0; x < 4; ++x)
      stage[x] = j < g.m ? __ldg(reinterpret_cast<const float4*>(pk_u + (long long)j * kD + sc) + x) : make_float4(0.f, 0.f, 0.f, 0.f);
    stage_n = j < g.m ? __ldg(nk_u + j) : 0.f;
  };
  auto deposit = [&](int buf) {
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      split2(stage[x].x, stage[x].y, hi[2 * x], lo[2 * x]);
      split2(stage[x].z, stage[x].w, hi[2 * x + 1], lo[2 * x + 1]);
    }
    uint4* h = reinterpret_cast<uint4*>(&sm.scr.kh[buf][0][sj][sc]);
    uint4* l = reinterpret_cast<uint4*>(&sm.scr.kh[buf][1][sj][sc]);
    h[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    h[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
    l[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    l[1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
    // a vector too short to be split safely (its parts may be subnormal) gets an infinite bound
    if ((tid & 3) == 0) sm.scr.nk[buf][sj] = stage_n < 1e-30f ? kInf : stage_n * 6.103515625e-5f;
  };
  fetch(0);
  for (int e = tid; e < TI * (kD / 4); e += NT) {
    const int r = e / (kD / 4), c4 = e - r * (kD / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 + r < g.m) v = __ldg(reinterpret_cast<const float4*>(pq_u + (long long)(i0 + r) * kD + 4 * c4));
    *reinterpret_cast<float4*>(&sm.qs[r][4 * c4]) = v;
  }
  if (tid < TI) {
    const float n = i0 + tid < g.m ? __ldg(nq + (long long)u * g.m + i0 + tid) : 1.f;
    sm.nq[tid] = n < 1e-30f ? kInf : n;
    sm.cnt[tid] = 0;
  }
  deposit(0);
  __syncthreads();

  // this warp's part of the products: rows of one 16-row tile, NT8 groups of eight keys
  const int rt = warp % RT, n0 = (warp / RT) * NT8;
  const int rr[2] = {16 * rt + (lane >> 2), 16 * rt + (lane >> 2) + 8};  // the lane's two rows
  uint32_t ah[4][4], al[4][4];
#pragma unroll
  for (int ks = 0; ks < 4; ++ks)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const float2 v = *reinterpret_cast<const float2*>(&sm.qs[rr[x & 1]][16 * ks + 8 * (x >> 1) + 2 * (lane & 3)]);
      split2(v.x, v.y, ah[ks][x], al[ks][x]);
    }
  const float nqv[2] = {sm.nq[rr[0]], sm.nq[rr[1]]};
  // block coordinates of the rows (group mode: of their groups)
  const float inv_nbw = 1.0f / (float)g.nbw, inv_rlat = 1.0f / (float)max(g.rlat, 1), inv_rlon = 1.0f / (float)max(g.rlon, 1);
  int iy[2], ix[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int i = min(i0 + rr[a], g.m - 1);
    iy[a] = i / g.nbw;
    ix[a] = i - iy[a] * g.nbw;
    if (g.local_groups) { iy[a] /= g.rlat; ix[a] /= g.rlon; }
  }
  // block rows (group mode: group rows) that hold keys local to a row of the 16-row tile
  int iy_lo = (i0 + 16 * rt) / g.nbw, iy_hi = (i0 + 16 * rt + 15) / g.nbw;
  if (g.local_groups) { iy_lo /= g.rlat; iy_hi /= g.rlat; }
  else { iy_lo -= g.rlat; iy_hi += g.rlat; }
  float best[2][kDepth], thr[2] = {0.f, 0.f};
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int d = 0; d < kDepth; ++d) best[a][d] = -kInf;

  int buf = 0;
  for (int pass = 0; pass < 2; ++pass) {
    for (int ch = 0; ch < nchunks; ++ch) {
      const bool more = ch + 1 < nchunks || pass == 0;
      if (more) fetch(ch + 1 < nchunks ? ch + 1 : 0);  // the next chunk streams in while this one is screened
      const int j0 = ch * kTJ;
      float c[NT8][4];
#pragma unroll
      for (int n = 0; n < NT8; ++n) {
#pragma unroll
        for (int x = 0; x < 4; ++x) c[n][x] = 0.f;
        // eight keys: per part two loads of four 8 x 8 matrices (channels 0-31, 32-63)
        uint32_t bh[2][4], bl[2][4];
        const int key = 8 * (n0 + n) + (lane & 7), col = 8 * (lane >> 3);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          ldmatrix4(bh[x], &sm.scr.kh[buf][0][key][32 * x + col]);
          ldmatrix4(bl[x], &sm.scr.kh[buf][1][key][32 * x + col]);
        }
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          mma_bf16(c[n], al[ks], bh[ks >> 1][2 * (ks & 1)], bh[ks >> 1][2 * (ks & 1) + 1]);
          mma_bf16(c[n], ah[ks], bl[ks >> 1][2 * (ks & 1)], bl[ks >> 1][2 * (ks & 1) + 1]);
        }
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
          mma_bf16(c[n], ah[ks], bh[ks >> 1][2 * (ks & 1)], bh[ks >> 1][2 * (ks & 1) + 1]);
      }
      // Plain chunk for this warp (the common case): wholly inside the grid, every row of the tile exists, and no key of
      // the chunk can be local to any of the rows, so every (row, key) pair is a candidate.
      bool plain = j0 + kTJ <= g.m && i0 + 16 * rt + 15 < g.m;
      if (plain) {
        int jy_lo = quick_div(j0, g.nbw, inv_nbw), jy_hi = quick_div(j0 + kTJ - 1, g.nbw, inv_nbw);
        if (g.local_groups) {
          jy_lo = quick_div(jy_lo, g.rlat, inv_rlat);
          jy_hi = quick_div(jy_hi, g.rlat, inv_rlat);
        }
        plain = jy_lo > iy_hi || jy_hi < iy_lo;
      }
#pragma unroll
      for (int n = 0; n < NT8; ++n) {
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const int jj = 8 * (n0 + n) + 2 * (lane & 3) + y, j = j0 + jj;
          const float nkc = sm.scr.nk[buf][jj];
          bool cand[2] = {true, true};
          if (!plain) {
            int jy = quick_div(j, g.nbw, inv_nbw), jx = j - jy * g.nbw;
            if (g.local_groups) {
              jy = quick_div(jy, g.rlat, inv_rlat);
              jx = quick_div(jx, g.rlon, inv_rlon);
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
              int dx = jx - ix[a];
              dx += dx < 0 ? g.nbw : 0;  // (jx - ix) mod nbw
              const bool local = g.local_groups ? (jy == iy[a] && jx == ix[a])
                                                : (abs(jy - iy[a]) <= g.rlat && (dx <= g.rlon || g.nbw - dx <= g.rlon));
              cand[a] = j < g.m && !local && i0 + rr[a] < g.m;
            }
          }
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            const float s = c[n][2 * a + y], eps = fmaf(nqv[a], nkc, 1e-37f);
            const bool fin = fabsf(s) <= 1e38f;  // (an infinite eps gives the bounds -inf and +inf by itself)
            if (pass == 0) {
              float x = fin && cand[a] ? s - eps : -kInf;
#pragma unroll
              for (int d = 0; d < kDepth; ++d) {  // insertion into the lane's sorted list
                const float top = fmaxf(best[a][d], x);
                x = fminf(best[a][d], x);
                best[a][d] = top;
              }
            } else if (cand[a] && !(fin && s + eps < thr[a])) {
              const int at = atomicAdd(&sm.cnt[rr[a]], 1);
              if (at < CAP) sm.surv[rr[a]][at] = j;
            }
          }
        }
      }
      if (ch + 1 < nchunks) {
        deposit(buf ^ 1);
        buf ^= 1;
        __syncthreads();
      }
    }
    if (pass == 0) {
      // thr <- k-th largest of a row's kept lower bounds, two per lane; the rows of a warp in lockstep so that the
      // latencies of the warp-wide steps overlap.  A pop takes the largest out of its lane's pair.
      __syncthreads();
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int d = 0; d < kDepth; ++d) sm.tracked[rr[a]][((warp / RT) * 4 + (lane & 3)) * kDepth + d] = best[a][d];
      __syncthreads();
      float t1[RI], t2[RI];
#pragma unroll
      for (int a = 0; a < RI; ++a) {
        const float x = sm.tracked[warp * RI + a][lane], y = sm.tracked[warp * RI + a][lane + 32];
        t1[a] = fmaxf(x, y);
        t2[a] = fminf(x, y);
      }
      for (int r = 0; r + 1 < g.topk; ++r) {
#pragma unroll
        for (int a = 0; a < RI; ++a) {
          const unsigned o = ordered_bits(t1[a]);
          const unsigned top = __reduce_max_sync(0xffffffffu, o);
          const unsigned who = __ballot_sync(0xffffffffu, o == top);
          if (lane == __ffs(who) - 1) { t1[a] = t2[a]; t2[a] = -kInf; }
        }
      }
#pragma unroll
      for (int a = 0; a < RI; ++a) {
        const float t = from_ordered_bits(__reduce_max_sync(0xffffffffu, ordered_bits(t1[a])));
        if (lane == 0) sm.thr[warp * RI + a] = t;
      }
      __syncthreads();  // the kept values are consumed: the first chunk may land in their place
      buf = 0;
      deposit(0);
      __syncthreads();
      thr[0] = sm.thr[rr[0]];
      thr[1] = sm.thr[rr[1]];
    }
  }
  __syncthreads();  // the survivors are complete, the staging buffers are free
  int cnt[RI];
#pragma unroll
  for (int a = 0; a < RI; ++a) cnt[a] = sm.cnt[warp * RI + a];

  // ---- exact phase (the staging buffers are free now and hold the survivors' score keys)
  // rows whose survivors fit the counting rank: flatten (row, entry) pairs over the lanes, two chains in flight
  int base_of[RI + 1];
  base_of[0] = 0;
  unsigned slow = 0;  // rows that take the insertion path (their survivors overflowed)
#pragma unroll
  for (int a = 0; a < RI; ++a) {
    const bool row_ok = i0 + warp * RI + a < g.m;
    const bool fast = row_ok && cnt[a] <= CAP;
    if (row_ok && !fast) slow |= 1u << a;
    base_of[a + 1] = base_of[a] + (fast ? cnt[a] : 0);
  }
  __syncwarp();
  const int total = base_of[RI];
  for (int p0 = 0; p0 < total; p0 += 64) {
    int pa[2], pe[2], pj[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int p = p0 + 32 * t + lane;
      pa[t] = -1; pe[t] = 0; pj[t] = 0;
      if (p < total) {
#pragma unroll
        for (int a = 0; a < RI; ++a)
          if (p >= base_of[a] && p < base_of[a + 1]) { pa[t] = a; pe[t] = p - base_of[a]; }
        pj[t] = sm.surv[warp * RI + pa[t]][pe[t]];
      }
    }
    // both chains in one instruction stream (inlined twice; the loads of the second overlap the first's arithmetic)
    unsigned long long k0 = 0ull, k1 = 0ull;
    if (pa[0] >= 0) k0 = exact_key(sm.qs[warp * RI + pa[0]], pk_u, pj[0]);
    if (pa[1] >= 0) k1 = exact_key(sm.qs[warp * RI + pa[1]], pk_u, pj[1]);
    if (pa[0] >= 0) sm.ekey[warp * RI + pa[0]][pe[0]] = k0;
    if (pa[1] >= 0) sm.ekey[warp * RI + pa[1]][pe[1]] = k1;
  }
  __syncwarp();
#pragma unroll
  for (int a = 0; a < RI; ++a) {
    const int row = warp * RI + a, i = i0 + row;
    if (i >= g.m) break;  // warp-uniform
    int32_t* out = block_idx + ((long long)u * g.m + i) * g.topk;
    if (!((slow >> a) & 1u)) {
      const int n = cnt[a];
      for (int e = lane; e < n; e += 32) {  // rank by counting the survivors that come first
        const unsigned long long key = sm.ekey[row][e];
        const int id = sm.surv[row][e];
        int rank = 0;
        for (int f = 0; f < n; ++f) rank += ranks_before(sm.ekey[row][f], sm.surv[row][f], key, id) ? 1 : 0;
        if (rank < g.topk) out[rank] = id;
      }
      if (lane >= n && lane < g.topk) out[lane] = -1;
    } else {
      unsigned long long lkey = 0ull;
      int lid = -1;
      // too many survivors to hold: score every key of the unit
      for (int jb = 0; jb < g.m; jb += 32) {
        const int j = jb + lane;
        bool cand = j < g.m;
        if (cand) {
          cand = !is_local(g, i, j);
        }
        insert_batch(cand ? exact_key(sm.qs[row], pk_u, j) : 0ull, j, lkey, lid, g.topk, lane);
      }
      if (lane < g.topk) out[lane] = lkey != 0ull ? lid : -1;
    }
  }
}

template <int TI, int CAP>
int launch_topk(const HostCtx& c, const float* pooled_q, const float* pooled_k, const float* norm_q, const float* norm_k,
                int32_t* block_idx) {
  const Geo& g = c.g;
  const size_t smem = sizeof(TopkSmem<TI, CAP>);
  static unsigned long long configured = 0;  // devices on which the kernel's shared-memory opt-in is set
  int sms = 0;
  if (const int rc = launch_setup(reinterpret_cast<const void*>(topk_kernel<TI, CAP>), smem, &configured, &sms)) return rc;
  const long long ctas = (long long)g.U * ((g.m + TI - 1) / TI);
  if (ctas > 0x7fffffffll) return MOSAIC_E_UNSUPPORTED;
  return launch_kernel(topk_kernel<TI, CAP>, dim3((unsigned)ctas), kTW * 32, smem, c.stream, ctas <= sms, 0, g, pooled_q, pooled_k, norm_q,
                       norm_k, block_idx);
}

int launch_select(const HostCtx& c, const void* q, const void* k, int32_t* block_idx, float* pooled_q,
                  float* pooled_k, float* norm_q, float* norm_k) {
  const Geo& g = c.g;
  PoolArgs a = {};
  a.n = 2;
  a.job[0] = {q, pooled_q, norm_q, nullptr, g.U};
  a.job[1] = {k, pooled_k, norm_k, nullptr, g.Ukv};
  if (const int rc = launch_pool(c, a)) return rc;
  if (g.topk > 0) {
    // 32 query blocks per CTA where that still gives every SM about two CTAs, 16 below (192 units of 450 blocks 390 us with 32,
    // 455 with 16; 8 units 47 with 32, 26 with 16).  The survivors of a row grow with
    // top-k (the threshold is the k-th best of 64 kept bounds), and a row whose survivors overflow scores every key
    // exactly: beyond top-k 16 there is room for 192 of them.
    const bool wide = (long long)g.U * ((g.m + 31) / 32) >= 296;
    const int rc = g.topk > 16 ? (wide ? launch_topk<32, 192>(c, pooled_q, pooled_k, norm_q, norm_k, block_idx)
                                       : launch_topk<16, 192>(c, pooled_q, pooled_k, norm_q, norm_k, block_idx))
                               : (wide ? launch_topk<32, 96>(c, pooled_q, pooled_k, norm_q, norm_k, block_idx)
                                       : launch_topk<16, 96>(c, pooled_q, pooled_k, norm_q, norm_k, block_idx));
    if (rc) return rc;
  }
  return MOSAIC_OK;
}

}  // namespace mosaic

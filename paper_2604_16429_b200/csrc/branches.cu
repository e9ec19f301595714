// Compression branch of the three-branch form of the operator, forward and backward, on the block level.
//
// Paper: Eq. of the aggregated output (section "Native Sparse Attention") and the "Compression" paragraph of the
// section "Block-Sparse Attention": block-level softmax attention abar_ij over ALL m blocks on the mean-pooled
// queries and keys, obar_i = sum_j abar_ij vbar_j, the same vector for every token of query block i; then
//   o_l = g_CG(l) obar_i + g_FG(l) oFG_l + g_L(l) oL_l .
// The selection and local branch outputs oFG, oL and the gated sum come from the attention kernel.  With dO the gradient
// of o, the backward of this branch is, with dobar_i = sum_{l in block i} g_CG(l) dO_l (from the pooling kernel),
// delta_i = <dobar_i, obar_i>, dp_ij = <dobar_i, vbar_j>, ds_ij = abar_ij (dp_ij - delta_i):
//   dvbar_j = sum_i abar_ij dobar_i,  dqbar_i = scale sum_j ds_ij kbar_j,  dkbar_j = scale sum_i ds_ij qbar_i ;
// a mean spreads its gradient evenly: every token of a block receives 1/b of the block's.  This is the only path by
// which gradient reaches the block-level (routing) scores.
//
// Everything here is fp32 on the CUDA cores (4 to 8 m^2 d FLOP per unit; the inputs are fp32 sums).  A CTA of 256 threads
// owns 64 stationary blocks of one unit and streams the other side in chunks of 64; a thread computes a 4 x 4 tile of a
// 64 x 64 product from shared memory.  The chunks of a tile are split over a cluster of up to 4 CTAs, which add their partial sums over
// distributed shared memory in rank order, so results do not depend on timing.
// Bound by shared-memory operand loads (2 reads of 4 words per 16 FMAs) and, for few tiles, by the length of a stream.  us,
// before -> after: forward of 8 units of 450 blocks twice 77 -> 47, backward of both sides 110 -> 72; backward of 12 units of
// 384 blocks 212 -> 92; of 20 units of 24 blocks 27 -> 16.
#include <cooperative_groups.h>

#include "common.cuh"

namespace mosaic {

namespace {

namespace cgs = cooperative_groups;

constexpr int kT = 64;          // blocks of a tile and of a chunk
constexpr int kRows = 4;        // rows of a thread's tile
constexpr int kThr = 256;       // threads: 16 row groups (4 rows each) x 16 columns (4 of them 16 apart)
constexpr int kStr = kD + 4;    // padded row (floats)
typedef float Tile[kT][kStr];

// 64 pooled vectors (rows r0 .. r0 + 63 of a unit) into shared memory, zeros past the end
__device__ __forceinline__ void load_tile(Tile& t, const float* __restrict__ src, int r0, int m) {
#pragma unroll
  for (int k = 0; k < kT * kD / 4 / kThr; ++k) {
    const int e = threadIdx.x + k * kThr, r = e >> 4, c4 = e & 15;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r0 + r < m) v = __ldg(reinterpret_cast<const float4*>(src + (long long)(r0 + r) * kD) + c4);
    *reinterpret_cast<float4*>(&t[r][4 * c4]) = v;
  }
}
// s[a][b] = <A row 4 ty + a, B row tx + 16 b>
__device__ __forceinline__ void tile_nt(float (&s)[kRows][4], const Tile& A, const Tile& B, int ty, int tx) {
#pragma unroll
  for (int a = 0; a < kRows; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) s[a][b] = 0.f;
#pragma unroll 4
  for (int c4 = 0; c4 < kD / 4; ++c4) {
    float4 bv[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) bv[b] = *reinterpret_cast<const float4*>(&B[tx + 16 * b][4 * c4]);
#pragma unroll
    for (int a = 0; a < kRows; ++a) {
      const float4 x = *reinterpret_cast<const float4*>(&A[kRows * ty + a][4 * c4]);
#pragma unroll
      for (int b = 0; b < 4; ++b)
        s[a][b] = fmaf(x.x, bv[b].x, fmaf(x.y, bv[b].y, fmaf(x.z, bv[b].z, fmaf(x.w, bv[b].w, s[a][b]))));
    }
  }
}
// acc[a][c] += sum_j W[4 ty + a][j] B[j][4 tx + c]
__device__ __forceinline__ void tile_nn(float (&acc)[kRows][4], const Tile& W, const Tile& B, int ty, int tx) {
#pragma unroll 4
  for (int j4 = 0; j4 < kT / 4; ++j4) {
    float4 bv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(&B[4 * j4 + j][4 * tx]);
#pragma unroll
    for (int a = 0; a < kRows; ++a) {
      const float4 w = *reinterpret_cast<const float4*>(&W[kRows * ty + a][4 * j4]);
      acc[a][0] = fmaf(w.x, bv[0].x, fmaf(w.y, bv[1].x, fmaf(w.z, bv[2].x, fmaf(w.w, bv[3].x, acc[a][0]))));
      acc[a][1] = fmaf(w.x, bv[0].y, fmaf(w.y, bv[1].y, fmaf(w.z, bv[2].y, fmaf(w.w, bv[3].y, acc[a][1]))));
      acc[a][2] = fmaf(w.x, bv[0].z, fmaf(w.y, bv[1].z, fmaf(w.z, bv[2].z, fmaf(w.w, bv[3].z, acc[a][2]))));
      acc[a][3] = fmaf(w.x, bv[0].w, fmaf(w.y, bv[1].w, fmaf(w.z, bv[2].w, fmaf(w.w, bv[3].w, acc[a][3]))));
    }
  }
}

struct FwdSmem {
  Tile q, k, v, w;
  float mx[kT], z[kT];
};

// ------------------------------------------------------------------------------------------
// compress_kernel: streaming softmax attention on the pooled vectors.  Pooled sums are block SUMS: the means' 1/b
// enters as scale / b^2 on the logits and 1/b on the output.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThr) compress_kernel(Geo g, const float* __restrict__ pq, const float* __restrict__ pk,
                                                        const float* __restrict__ pv, float* __restrict__ ocg,
                                                        float* __restrict__ lse2) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FwdSmem& sm = *reinterpret_cast<FwdSmem*>(smem_raw);
  const cgs::cluster_group cluster = cgs::this_cluster();
  const int ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int tiles = (g.m + kT - 1) / kT, tile = (int)blockIdx.x / ranks + await_stream();
  const int u = tile / tiles, i0 = (tile - u * tiles) * kT;
  const float* pk_u = pk + (long long)kv_unit(g, u) * g.m * kD;   // grouped-query attention: the group's key/value head
  const float* pv_u = pv + (long long)kv_unit(g, u) * g.m * kD;
  const float inv_b = 1.0f / (float)g.b;
  const float sl2 = g.scale_log2 * inv_b * inv_b;  // logits in base-2 units
  load_tile(sm.q, pq + (long long)u * g.m * kD, i0, g.m);
  float mx[kRows], z[kRows], acc[kRows][4];
#pragma unroll
  for (int a = 0; a < kRows; ++a) { mx[a] = -INFINITY; z[a] = 0.f; acc[a][0] = acc[a][1] = acc[a][2] = acc[a][3] = 0.f; }
  for (int ch = rank; ch < tiles; ch += ranks) {
    const int j0 = ch * kT;
    __syncthreads();  // the previous chunk is consumed
    load_tile(sm.k, pk_u, j0, g.m);
    load_tile(sm.v, pv_u, j0, g.m);
    __syncthreads();
    float s[kRows][4];
    tile_nt(s, sm.q, sm.k, ty, tx);
#pragma unroll
    for (int a = 0; a < kRows; ++a) {
      float cm = -INFINITY;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        s[a][b] = j0 + tx + 16 * b < g.m ? s[a][b] * sl2 : -INFINITY;
        cm = fmaxf(cm, s[a][b]);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, o));  // the row's 16 threads
      const float nm = fmaxf(mx[a], cm);  // finite: every chunk holds at least one block
      const float alpha = exp2f(mx[a] - nm);
      mx[a] = nm;
      z[a] *= alpha;                      // this thread's share of the normaliser
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float w = exp2f(s[a][b] - nm);
        z[a] += w;
        acc[a][b] *= alpha;
        sm.w[kRows * ty + a][tx + 16 * b] = w;
      }
    }
    __syncwarp();  // a row's weights are written and read by the same half-warp
    tile_nn(acc, sm.w, sm.v, ty, tx);
  }
#pragma unroll
  for (int a = 0; a < kRows; ++a)
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) z[a] += __shfl_xor_sync(0xffffffffu, z[a], o);
  // every rank's partial result in its own shared memory; each rank finishes its share of the rows, adding in rank order
  __syncwarp();
#pragma unroll
  for (int a = 0; a < kRows; ++a) {
    *reinterpret_cast<float4*>(&sm.w[kRows * ty + a][4 * tx]) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
    if (tx == 0) { sm.mx[kRows * ty + a] = mx[a]; sm.z[kRows * ty + a] = z[a]; }
  }
  cluster.sync();
  const int per = kT / ranks;
  for (int e = tid; e < per * (kD / 4); e += kThr) {
    const int r = rank * per + (e >> 4), c = 4 * (e & 15);
    if (i0 + r >= g.m) continue;
    float top = -INFINITY;
    for (int p = 0; p < ranks; ++p) top = fmaxf(top, cluster.map_shared_rank(&sm.mx[0], p)[r]);
    float zz = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p = 0; p < ranks; ++p) {
      const float f = exp2f(cluster.map_shared_rank(&sm.mx[0], p)[r] - top);
      const float4 x = *reinterpret_cast<const float4*>(cluster.map_shared_rank(&sm.w[0][0], p) + r * kStr + c);
      zz += f * cluster.map_shared_rank(&sm.z[0], p)[r];
      o.x += f * x.x; o.y += f * x.y; o.z += f * x.z; o.w += f * x.w;
    }
    const float f = inv_b / zz;
    *reinterpret_cast<float4*>(ocg + ((long long)u * g.m + i0 + r) * kD + c) = make_float4(o.x * f, o.y * f, o.z * f, o.w * f);
    // base-2 log-sum-exp of the row's block-level logits, for the backward (which recomputes abar from it)
    if (lse2 && c == 0) lse2[(long long)u * g.m + i0 + r] = top + log2f(zz);
  }
  cluster.sync();  // no rank leaves while another reads its shared memory
}

struct BwdSmem {
  Tile a1, a2;   // stationary side: pooled query sums and dobar (query side) / pooled key and value sums (key side)
  Tile b1, b2;   // streamed side:   pooled key and value sums            / pooled query sums and dobar
  Tile wd, wa;   // ds and (key side) abar of the chunk
  float lse[kT], delta[kT];  // of the tile's rows (query side) / of the chunk's query blocks (key side)
};

// log-sum-exp and delta_i = <dobar_i, obar_i> of 64 query blocks whose dobar is in `dob`: four threads per block
__device__ __forceinline__ void row_stats(BwdSmem& sm, const Tile& dob, const float* __restrict__ ocg_u,
                                          const float* __restrict__ lse_u, int r0, int m) {
  const int r = threadIdx.x >> 2, part = threadIdx.x & 3;
  float d = 0.f;
  if (r0 + r < m) {
    const float4* o = reinterpret_cast<const float4*>(ocg_u + (long long)(r0 + r) * kD + 16 * part);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 x = __ldg(o + c), y = *reinterpret_cast<const float4*>(&dob[r][16 * part + 4 * c]);
      d = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, d))));
    }
  }
  d += __shfl_xor_sync(0xffffffffu, d, 1);
  d += __shfl_xor_sync(0xffffffffu, d, 2);
  if (part == 0) {
    sm.delta[r] = d;
    sm.lse[r] = r0 + r < m ? __ldg(lse_u + r0 + r) : 0.f;
  }
}

// ------------------------------------------------------------------------------------------
// compress_bwd_tile<KEY_SIDE>: the block-level softmax backward of one tile, recomputing abar from the saved base-2
// log-sum-exp.
//   query side: rows i; dqm_i = scale / b^2 * sum_j ds_ij ksum_j
//   key side:   rows j of a key/value unit, summed over the query heads of its group;
//               dkm_j = scale / b^2 * sum_i ds_ij qsum_i and dvm_j = 1/b * sum_i abar_ij dobar_i
// (sums are block SUMS; dqm, dkm, dvm are what every token of the block receives).
// ------------------------------------------------------------------------------------------
template <bool KEY_SIDE>
__device__ __forceinline__ void compress_bwd_tile(const Geo& g, BwdSmem& sm, int tile, const CompressBwd& a) {
  const cgs::cluster_group cluster = cgs::this_cluster();
  const int ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int tiles = (g.m + kT - 1) / kT;
  const int u = tile / tiles, r0 = (tile - u * tiles) * kT;  // u: query unit / key-value unit
  const float inv_b = 1.0f / (float)g.b;
  const float sl2 = g.scale_log2 * inv_b * inv_b;
  const int ratio = g.H / g.Hkv;
  const long long md = (long long)g.m * kD;
  load_tile(sm.a1, (KEY_SIDE ? a.pk : a.pq) + u * md, r0, g.m);
  load_tile(sm.a2, (KEY_SIDE ? a.pv : a.dob) + u * md, r0, g.m);
  __syncthreads();
  if (!KEY_SIDE) row_stats(sm, sm.a2, a.ocg + u * md, a.lse2 + (long long)u * g.m, r0, g.m);
  float acc1[kRows][4], acc2[KEY_SIDE ? kRows : 1][4];
#pragma unroll
  for (int x = 0; x < kRows; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) { acc1[x][y] = 0.f; if (KEY_SIDE) acc2[x][y] = 0.f; }
  // chunks of the streamed side: the group's keys (query side) / the chunks of each query head of the group (key side)
  const int chunks = KEY_SIDE ? ratio * tiles : tiles;
  for (int ch = rank; ch < chunks; ch += ranks) {
    const int pass = ch / tiles, j0 = (ch - pass * tiles) * kT;
    const int us = KEY_SIDE ? (u / g.Hkv) * g.H + (u - (u / g.Hkv) * g.Hkv) * ratio + pass : kv_unit(g, u);
    __syncthreads();  // the previous chunk is consumed
    load_tile(sm.b1, (KEY_SIDE ? a.pq : a.pk) + us * md, j0, g.m);
    load_tile(sm.b2, (KEY_SIDE ? a.dob : a.pv) + us * md, j0, g.m);
    __syncthreads();
    if (KEY_SIDE) {
      row_stats(sm, sm.b2, a.ocg + us * md, a.lse2 + (long long)us * g.m, j0, g.m);
      __syncthreads();
    }
    float s[kRows][4], dp[kRows][4];
    tile_nt(s, sm.a1, sm.b1, ty, tx);
    tile_nt(dp, sm.a2, sm.b2, ty, tx);
#pragma unroll
    for (int x = 0; x < kRows; ++x) {
      const int r = kRows * ty + x;
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int j = tx + 16 * y;
        const bool in = r0 + r < g.m && j0 + j < g.m;
        const float ab = in ? exp2f(s[x][y] * sl2 - sm.lse[KEY_SIDE ? j : r]) : 0.f;
        sm.wd[r][j] = ab * (dp[x][y] * inv_b - sm.delta[KEY_SIDE ? j : r]);
        if (KEY_SIDE) sm.wa[r][j] = ab;
      }
    }
    __syncwarp();  // a row's weights are written and read by the same half-warp
    tile_nn(acc1, sm.wd, sm.b1, ty, tx);
    if (KEY_SIDE) tile_nn(reinterpret_cast<float(&)[kRows][4]>(acc2), sm.wa, sm.b2, ty, tx);
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < kRows; ++x) {
    *reinterpret_cast<float4*>(&sm.wd[kRows * ty + x][4 * tx]) = make_float4(acc1[x][0], acc1[x][1], acc1[x][2], acc1[x][3]);
    if (KEY_SIDE)
      *reinterpret_cast<float4*>(&sm.wa[kRows * ty + x][4 * tx]) = make_float4(acc2[x][0], acc2[x][1], acc2[x][2], acc2[x][3]);
  }
  cluster.sync();
  const float f1 = g.scale * inv_b * inv_b;
  const int per = kT / ranks;
  for (int e = tid; e < per * (kD / 4); e += kThr) {
    const int r = rank * per + (e >> 4), c = 4 * (e & 15);
    if (r0 + r >= g.m) continue;
#pragma unroll
    for (int which = 0; which < (KEY_SIDE ? 2 : 1); ++which) {
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int p = 0; p < ranks; ++p) {
        const float4 x = *reinterpret_cast<const float4*>(
            cluster.map_shared_rank(which ? &sm.wa[0][0] : &sm.wd[0][0], p) + r * kStr + c);
        o.x += x.x; o.y += x.y; o.z += x.z; o.w += x.w;
      }
      const float f = which ? inv_b : f1;
      float* out = (which ? a.dvm : KEY_SIDE ? a.dkm : a.dqm) + u * md + (long long)(r0 + r) * kD + c;
      *reinterpret_cast<float4*>(out) = make_float4(o.x * f, o.y * f, o.z * f, o.w * f);
    }
  }
  cluster.sync();  // no rank leaves while another reads its shared memory
}

// one launch for both sides: the first `query_ctas` CTAs take the query side
__global__ void __launch_bounds__(kThr) compress_bwd_kernel(Geo g, const CompressBwd a, int query_ctas) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdSmem& sm = *reinterpret_cast<BwdSmem*>(smem_raw);
  const int ranks = (int)cgs::this_cluster().num_blocks();
  const int cta = (int)blockIdx.x + await_stream();
  if (cta < query_ctas) compress_bwd_tile<false>(g, sm, cta / ranks, a);
  else compress_bwd_tile<true>(g, sm, (cta - query_ctas) / ranks, a);
}

// CTAs per tile: at most four, at most one per chunk.  Not by how many units there are, because the sums are formed per CTA:
// a unit's bits must not depend on the others.  us of a pass over units of 450 blocks with a cluster of two, four, eight: training
// 1 unit 314, 274, 260, 4 units 614, 586, 586, 8 units 999, 1001, 1021, 16 units 1850, 1875, 1914, 64 units 6831, 6883, 7034,
// inference of 192 units 4843, 4881, 4993.
int cluster_size(int chunks) {
  int s = 1;
  while (s < 4 && 2 * s <= chunks) s *= 2;
  return s;
}

template <class Kernel, class... Args>
int launch_clustered(const HostCtx& c, Kernel kernel, size_t smem, unsigned long long* configured, long long ctas, int cluster,
                     Args... args) {
  int sms = 0;
  if (const int rc = launch_setup(reinterpret_cast<const void*>(kernel), smem, configured, &sms)) return rc;
  if (ctas > 0x7fffffffll) return MOSAIC_E_UNSUPPORTED;
  return launch_kernel(kernel, dim3((unsigned)ctas), kThr, smem, c.stream, false, cluster, args...);
}

}  // namespace

int launch_compress(const HostCtx& c, const float* pooled_q, const float* pooled_k, const float* pooled_v, float* ocg,
                    float* lse2) {
  static unsigned long long configured = 0;  // devices on which the kernel's shared-memory opt-in is set
  const int tiles = (c.g.m + kT - 1) / kT, s = cluster_size(tiles);
  if ((long long)c.g.U * tiles * s > 0x7fffffffll) return MOSAIC_E_UNSUPPORTED;
  return launch_clustered(c, compress_kernel, sizeof(FwdSmem), &configured, (long long)c.g.U * tiles * s, s, c.g, pooled_q,
                          pooled_k, pooled_v, ocg, lse2);
}

int launch_compress_bwd(const HostCtx& c, const CompressBwd& a) {
  static unsigned long long configured = 0;  // devices on which the kernel's shared-memory opt-in is set
  const int tiles = (c.g.m + kT - 1) / kT;
  const long long q_tiles = (long long)c.g.U * tiles, kv_tiles = (long long)c.g.Ukv * tiles;
  const int s = cluster_size(tiles * (c.g.H / c.g.Hkv));  // the key side has the longer streams
  if (q_tiles * s > 0x7fffffffll) return MOSAIC_E_UNSUPPORTED;
  return launch_clustered(c, compress_bwd_kernel, sizeof(BwdSmem), &configured, (q_tiles + kv_tiles) * s, s, c.g, a,
                          (int)(q_tiles * s));
}

}  // namespace mosaic

// Block sums of Q, K, V and of the gated dO (block representations of the "Compression" paragraph, phi = mean: the
// mean's 1/b is applied where a sum is used).
//
// pooled sum = fp64 accumulation over the block's tokens in row-major order, one rounding to fp32: the selection's ids
// depend on it bit for bit, so a channel is one sequential chain and the work is split over units, blocks and channels only.
//
// HBM-bound on large inputs (2.12 GB in 0.32 ms, the copy rate), latency-bound on small ones, where one launch for all
// tensors of an op pays: backward of the three-branch form over 3072 tokens 9 launches 145 us -> 3 launches 24 us, over 49152
// tokens 206 -> 100 us.
#include "common.cuh"

namespace mosaic {

namespace {

template <int CH>
struct LaneWords { using type = uint4; };
template <>
struct LaneWords<4> { using type = uint2; };
template <>
struct LaneWords<2> { using type = uint32_t; };
__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
__device__ __forceinline__ uint32_t word_of(const uint2& v, int i) { return i == 0 ? v.x : v.y; }
__device__ __forceinline__ uint32_t word_of(const uint32_t& v, int) { return v; }

// One block's share of a lane: CH channels, RU block rows in flight.  GATED: every token weighted by its compression gate.
template <int BW, int CH, int RU, bool GATED>
__device__ __forceinline__ void pool_block(const Geo& g, const typename LaneWords<CH>::type* src, const float* gate,
                                           double (&acc)[CH]) {
  using W = typename LaneWords<CH>::type;
  constexpr int kPer = kD / CH;  // lanes (and vectors) per token
  for (int r0 = 0; r0 < g.bh; r0 += RU) {
    W v[RU][BW];
    float w[GATED ? RU : 1][GATED ? BW : 1];
#pragma unroll
    for (int k = 0; k < RU; ++k) {
      if (r0 + k >= g.bh) break;
      const long long row = (long long)(r0 + k) * g.nlon;
#pragma unroll
      for (int c = 0; c < BW; ++c) {
        v[k][c] = __ldg(src + (row + c) * kPer);
        if (GATED) w[k][c] = __ldg(gate + 3 * (row + c));
      }
    }
#pragma unroll
    for (int k = 0; k < RU; ++k) {
      if (r0 + k >= g.bh) break;
#pragma unroll
      for (int c = 0; c < BW; ++c) {
#pragma unroll
        for (int e = 0; e < CH / 2; ++e) {
          float lo, hi;
          unpack16x2(word_of(v[k][c], e), g.f16 != 0, lo, hi);
          if (GATED) {
            acc[2 * e] = fma((double)w[k][c], (double)lo, acc[2 * e]);
            acc[2 * e + 1] = fma((double)w[k][c], (double)hi, acc[2 * e + 1]);
          } else {
            acc[2 * e] += (double)lo;
            acc[2 * e + 1] += (double)hi;
          }
        }
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// pool_kernel<BW, CH>: kD / CH lanes per (tensor, unit, block), a lane adds its CH consecutive channels token by token.
// HBM-bound where the problem fills the GPU (CH = 8, 16-byte loads: 2.12 GB in 0.32 ms = the copy rate); smaller problems
// are bound by the latency of a block's loads and its chain of additions, and take fewer channels per lane and more block
// rows in flight.  Beside the sums it writes an upper bound of each pooled vector's Euclidean norm (for the ranking
// kernel's screening pass), and it resets the workspace's status block: it is its op's first kernel.
// ------------------------------------------------------------------------------------------
template <int BW, int CH>
__global__ void __launch_bounds__(256) pool_kernel(Geo g, const PoolArgs a) {
  using W = typename LaneWords<CH>::type;
  constexpr int kPer = kD / CH, RU = CH == 8 ? 1 : 128 / (BW * CH);  // up to 64 words of loads in flight per lane
  const int tid = (int)threadIdx.x + await_stream();
  if (blockIdx.x == 0 && tid < kStatusBytes / 4) a.status[tid] = 0;
  const int sub = tid % kPer;
  const long long grp = ((long long)blockIdx.x * blockDim.x + tid) / kPer;
  PoolJob job = a.job[0];
  long long first = 0, at = (long long)job.units * g.m;  // jobs follow one another
#pragma unroll
  for (int i = 1; i < kPoolJobs; ++i) {
    if (i < a.n && grp >= at) {
      job = a.job[i];
      first = at;
    }
    if (i < a.n) at += (long long)a.job[i].units * g.m;
  }
  const bool live = grp < at;  // the last warp may be partly idle; it still takes part in the shuffles
  const long long w = live ? grp - first : 0;
  const int u = (int)(w / g.m), j = (int)(w - (long long)u * g.m);
  const int by = j / g.nbw, bx = j - by * g.nbw;
  const long long tok = (long long)u * g.N + (long long)by * g.bh * g.nlon + bx * BW;
  const W* src = static_cast<const W*>(job.src) + tok * kPer + sub;
  double acc[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) acc[c] = 0.0;
  if (live) {
    if (job.gates) pool_block<BW, CH, (RU > 1 ? RU / 2 : 1), true>(g, src, job.gates + 3 * tok, acc);
    else pool_block<BW, CH, RU, false>(g, src, nullptr, acc);
  }
  float p[CH];
  double ss = 0.0;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    p[c] = (float)acc[c];
    ss += (double)p[c] * (double)p[c];
  }
#pragma unroll
  for (int o = 1; o < kPer; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (!live) return;
  float2* dst = reinterpret_cast<float2*>(job.dst + ((long long)u * g.m + j) * kD + CH * sub);
#pragma unroll
  for (int c = 0; c < CH / 2; ++c) dst[c] = make_float2(p[2 * c], p[2 * c + 1]);
  // rounded up twice, so that it is never below the norm of the fp32 vector (NaN and inf pass through)
  if (sub == 0 && job.norm) job.norm[(long long)u * g.m + j] = __fmul_ru(__double2float_ru(sqrt(ss)), 1.000001f);
}

template <int BW>
int launch_pool_bw(const HostCtx& c, const PoolArgs& a) {
  long long groups = 0;
  for (int i = 0; i < a.n; ++i) groups += (long long)a.job[i].units * c.g.m;
  // 16-byte loads once they make about a quarter of the threads the GPU holds (148 SMs x 2048); below that narrower lanes
  // (channels per lane 8, 4, 2: 192 units of 450 blocks 221, 246, 288 us; 20 units of 24 blocks, the whole op 111, 81, 36)
  const int ch = groups * 8 >= 75000 ? 8 : groups * 16 >= 75000 ? 4 : 2;
  const long long blocks = (groups * (kD / ch) + 255) / 256;
  int sms = 0;
  if (const int rc = launch_setup(nullptr, 0, nullptr, &sms)) return rc;
  if (blocks > 0x7fffffffll) return MOSAIC_E_UNSUPPORTED;
  return launch_kernel(ch == 8 ? pool_kernel<BW, 8> : ch == 4 ? pool_kernel<BW, 4> : pool_kernel<BW, 2>, dim3((unsigned)blocks),
                       256, 0, c.stream, blocks <= sms, 0, c.g, a);
}

}  // namespace

int launch_pool(const HostCtx& c, PoolArgs a) {
  a.status = c.status;
  return c.g.bw == 8 ? launch_pool_bw<8>(c, a) : launch_pool_bw<16>(c, a);
}

}  // namespace mosaic

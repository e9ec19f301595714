// Two-dimensional rotary position embedding of Q and K.
//
// Paper, "Overall architecture" paragraph: RoPE on queries and keys encodes longitude and latitude; the head
// dimension is split equally between the two coordinates and each half receives a standard RoPE of its angle in
// radians (architecture table of the appendix: theta = 10000).  Channels [0, d/2) belong to the longitude,
// [d/2, d) to the latitude; inside a half of width D = d/2 the pair (2i, 2i+1) turns by pos * theta^(-2i/D).
//
// HBM-bound: every element of Q and K is read and written once.  Eight lanes per token, a lane owns eight channels
// (four pairs, 16 bytes) and walks its share of the units of both tensors with the same four (cos, sin), which it computes
// once in fp64; the rotation is fp64 too, rounded to fp32 and then to the storage type.  The conversions set the pace if
// they are left to the conversion unit (16 a clock and SM; two an element took 94 us for 377 MB): the 16-bit patterns are
// moved into the exponent and mantissa of a double instead, which leaves a power of two that the (cos, sin) carry.
#include <cuda_bf16.h>

#include "common.cuh"

namespace mosaic {

namespace {

// Value of a 16-bit pattern times 2^-896 (bf16) or 2^-1008 (binary16), exactly: sign, exponent and mantissa at their places
// in a double.  Infinities and NaNs (all exponent bits set) come out finite and are the caller's to catch.
template <bool F16>
__device__ __forceinline__ double scaled_lo(uint32_t x) {
  const uint32_t s = x << 16;
  return __hiloint2double((int)((s & 0x80000000u) | ((s >> (F16 ? 6 : 3)) & (F16 ? 0x01ffffffu : 0x0fffffffu))), 0);
}
template <bool F16>
__device__ __forceinline__ double scaled_hi(uint32_t x) {
  const uint32_t s = x & 0xffff0000u;
  return __hiloint2double((int)((s & 0x80000000u) | ((s >> (F16 ? 6 : 3)) & (F16 ? 0x01ffffffu : 0x0fffffffu))), 0);
}

template <bool F16>
__device__ __forceinline__ uint4 rotate8(const uint4& v, const double (&c)[4], const double (&s)[4]) {
  constexpr uint32_t kExp = F16 ? 0x7c007c00u : 0x7f807f80u, kOne = F16 ? 0x04000400u : 0x00800080u;
  constexpr double kUnscale = F16 ? 0x1p-1008 : 0x1p-896;
  const uint32_t x[4] = {v.x, v.y, v.z, v.w};
  uint32_t r[4];
  if ((((x[0] & kExp) + kOne) | ((x[1] & kExp) + kOne) | ((x[2] & kExp) + kOne) | ((x[3] & kExp) + kOne)) & 0x80008000u) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // an infinity or a NaN among them
      float lo, hi;
      unpack16x2(x[i], F16, lo, hi);
      const double cc = c[i] * kUnscale, ss = s[i] * kUnscale;
      r[i] = pack16x2(__double2float_rn((double)lo * cc - (double)hi * ss), __double2float_rn((double)lo * ss + (double)hi * cc), F16);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double x0 = scaled_lo<F16>(x[i]), x1 = scaled_hi<F16>(x[i]);
      r[i] = pack16x2(__double2float_rn(x0 * c[i] - x1 * s[i]), __double2float_rn(x0 * s[i] + x1 * c[i]), F16);
    }
  }
  return make_uint4(r[0], r[1], r[2], r[3]);
}

// Units u0 .. u1 of one tensor, this lane's 16 bytes of each: four at a time, the next four fetched before these are turned.
template <bool F16>
__device__ __forceinline__ void turn_units(const uint4* __restrict__ src, uint4* __restrict__ dst, int u0, int u1,
                                           long long step, const double (&c)[4], const double (&s)[4]) {
  src += u0 * step;
  dst += u0 * step;
  uint4 v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (u0 + i < u1) v[i] = __ldg(src + i * step);
  for (int u = u0; u < u1; u += 4) {
    src += 4 * step;
    uint4 n[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (u + 4 + i < u1) n[i] = __ldg(src + i * step);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (u + i < u1) dst[i * step] = rotate8<F16>(v[i], c, s);
      v[i] = n[i];
    }
    dst += 4 * step;
  }
}

constexpr int kFreqs = kD / 4;  // frequencies of a half

template <bool F16>
__global__ void __launch_bounds__(256, 4) rope_kernel(Geo g, const uint4* __restrict__ q, const uint4* __restrict__ k,
                                                   const float* __restrict__ pos, double theta,
                                                   uint4* __restrict__ q_out, uint4* __restrict__ k_out) {
  __shared__ double freq[kFreqs];
  if (threadIdx.x < kFreqs) freq[threadIdx.x] = pow(theta, -2.0 * threadIdx.x / (kD / 2));
  __syncthreads();
  const long long x = ((long long)blockIdx.x * blockDim.x + threadIdx.x + await_stream()) >> 3;  // token of the grid
  const int part = threadIdx.x & 7;
  if (x >= g.N) return;
  const double p = (double)__ldg(pos + 2 * x + (part >> 2));  // longitude for channels 0..31, latitude for 32..63
  double c[4], s[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    sincos(p * freq[4 * (part & 3) + j], &s[j], &c[j]);  // pair 4 (part & 3) + j inside the half
    s[j] *= F16 ? 0x1p1008 : 0x1p896;
    c[j] *= F16 ? 0x1p1008 : 0x1p896;
  }
  // this block's share of the units (Q's, then K's)
  const int total = g.U + g.Ukv, per = (total + (int)gridDim.y - 1) / (int)gridDim.y;
  const int u0 = (int)blockIdx.y * per, u1 = min(total, u0 + per);
  const long long row = x * 8 + part, step = g.N * 8;
  turn_units<F16>(q + row, q_out + row, u0, min(u1, g.U), step, c, s);
  turn_units<F16>(k + row, k_out + row, max(u0, g.U) - g.U, u1 - g.U, step, c, s);
}

}  // namespace

int launch_rope(const HostCtx& c, const void* q, const void* k, const float* pos, double theta, void* q_out, void* k_out) {
  const Geo& g = c.g;
  const long long blocks = (g.N * 8 + 255) / 256;
  if (blocks > 0x7fffffffll) return MOSAIC_E_UNSUPPORTED;
  // short sequences (3072 tokens, 25 units: 20.3 us unsplit, 16.2 split; 49152 tokens 63 us, split to the end 79): the units are split too, until the GPU is full (148 SMs x 8 CTAs) or a share is down to four units
  int split = 1;
  while (blocks * split < 1184 && split * 8 <= g.U + g.Ukv) split *= 2;
  const dim3 grid((unsigned)blocks, (unsigned)split);
  return launch_kernel(g.f16 ? rope_kernel<true> : rope_kernel<false>, grid, 256, 0, c.stream, true, 0, g, (const uint4*)q,
                       (const uint4*)k, pos, theta, (uint4*)q_out, (uint4*)k_out);
}

}  // namespace mosaic

// Shared device/host definitions of the MOSAIC block-sparse attention kernels (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mosaic_bsa.h"

namespace mosaic {

constexpr int kD = 64;            // head dimension
constexpr int kChunk = 64;        // tokens per staged key/value chunk (and per mma.sync query tile)
constexpr int kMaxList = 64;      // most blocks one query block attends (local + top-k)
constexpr int kMaxTopk = 32;
constexpr int kStatusBytes = 256; // status block at the start of every workspace

// Geometry of one call, passed by value to the kernels.
struct Geo {
  int U;            // B*H independent units
  int H, Hkv;       // query heads, key/value heads (grouped-query attention: H / Hkv query heads share a key/value head)
  int Ukv;          // B*Hkv key/value units
  int nlat, nlon;   // grid
  int bh, bw;       // block shape
  int nbh, nbw, m;  // blocks per column / row / unit
  int b;            // tokens per block
  int cpb;          // 64-token chunks per block (b / 64)
  int crows;        // grid rows per chunk (64 / bw)
  int rlat, rlon, topk;
  int local_groups; // 1: the local set is the aligned group of rlat x rlon blocks that holds the block
  int f16;          // 1: the 16-bit tensors are IEEE binary16, 0: bf16
  float scale;      // softmax scale
  float scale_log2; // scale * log2(e)
  long long N;      // tokens per unit
};

// key/value unit read by query unit u
__host__ __device__ __forceinline__ int kv_unit(const Geo& g, int u) {
  const int b = u / g.H;
  return b * g.Hkv + (u - b * g.H) / (g.H / g.Hkv);
}

// Two 16-bit elements of the problem's storage type (bf16 or binary16) packed in a word <-> two floats.
__device__ __forceinline__ void unpack16x2(uint32_t x, bool f16, float& lo, float& hi) {
  if (f16) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&x));
    lo = v.x;
    hi = v.y;
  } else {
    lo = __uint_as_float(x << 16);
    hi = __uint_as_float(x & 0xffff0000u);
  }
}
__device__ __forceinline__ uint32_t pack16x2(float lo, float hi, bool f16) {
  if (f16) {
    const __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// Record the first device-side fault in the workspace status word (never traps).
__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

// Is key block j inside the local set of query block i (window: rows clamp(by+dy), columns (bx+dx) mod nbw;
// group mode: the same aligned group of rlat x rlon blocks)?
__device__ __forceinline__ bool is_local(const Geo& g, int i, int j) {
  int by = i / g.nbw, bx = i - by * g.nbw;
  int jy = j / g.nbw, jx = j - jy * g.nbw;
  if (g.local_groups) return by / g.rlat == jy / g.rlat && bx / g.rlon == jx / g.rlon;
  // clamping only folds an out-of-range row onto a row already in the window
  bool row_ok = abs(jy - by) <= g.rlat;
  int dx = jx - bx;
  dx += dx < 0 ? g.nbw : 0;                       // (jx - bx) mod nbw in [0, nbw)
  bool col_ok = dx <= g.rlon || g.nbw - dx <= g.rlon;
  return row_ok && col_ok;
}

// a / b for 0 <= a < 2^24 and inv = 1.0f / b: the rounded quotient is off by at most one
__device__ __forceinline__ int quick_div(int a, int b, float inv) {
  int q = __float2int_rz((float)a * inv);
  const int r = a - q * b;
  q += r >= b ? 1 : r < 0 ? -1 : 0;
  return q;
}

// First token (row-major grid index inside the unit) of row `r` of chunk `c` of block j.
__device__ __forceinline__ long long chunk_row_token(const Geo& g, int j, int c, int r) {
  int by = j / g.nbw, bx = j - by * g.nbw;
  return (long long)(by * g.bh + c * g.crows + r) * g.nlon + bx * g.bw;
}

// Token of element e (0..63, row-major inside the chunk) of chunk c of block j.
__device__ __forceinline__ long long chunk_token(const Geo& g, int j, int c, int e) {
  int r = e / g.bw;
  return chunk_row_token(g, j, c, r) + (e - r * g.bw);
}

// Work items of 256 rows (four 64-row halves) per unit, as the tensor-core kernels cut a unit's blocks.
__host__ __device__ inline int items_per_unit(const Geo& g) {
  if (g.cpb == 1) return (g.nbh >> 1) * ((g.nbw + 1) >> 1) + (g.nbh & 1) * ((g.nbw + 3) >> 2);
  if (g.cpb == 2) return g.nbw > 1 ? g.nbh * ((g.nbw + 1) >> 1) : (g.nbh + 1) >> 1;
  return g.m * ((g.cpb + 3) >> 2);
}

// A kernel may be launched before the one ahead of it in the stream has finished (launch_kernel below says which are): every
// kernel sets up what touches no global memory, then calls this.  It returns when everything ahead is complete and visible,
// and lets the next kernel's CTAs in as SMs run empty (not earlier: the chain of waits makes "the kernel before me is
// complete" mean "all before it are").  The result is zero, opaque to the compiler: an address that it takes part in cannot
// be read earlier.
__device__ __forceinline__ int await_stream() {
  int zero;
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;\n\tmov.u32 %0, 0;" : "=r"(zero) : : "memory");
  return zero;
}

// ---- host side ---------------------------------------------------------------------------
// Launches a kernel that calls await_stream; with `overlap` its launch and set-up overlap the kernel ahead of it.  A pass
// of ten kernels over 3072 tokens takes 434 us without any overlap and 411 with it.  Not for kernels whose CTAs share SMs
// and are few (pooling and ranking beyond one CTA per SM, the block level): they land where the kernel ahead runs empty
// first and not evenly (pass over 8 units of 450 blocks: pooling 202.0 against 197.4 us, ranking 208.7 against 206.8; its
// three-branch training: block level 1088 against 1082).
template <class... P, class... A>
inline int launch_kernel(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, bool overlap,
                         int cluster, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...) == cudaSuccess ? MOSAIC_OK : MOSAIC_E_CUDA;
}

struct HostCtx {
  Geo g;
  cudaStream_t stream;
  int* status;  // device pointer to the workspace status word
};

int validate(const mosaic_bsa_params* p, Geo* g);
// Current device, its SM count (cached), and the opt-in to `smem` bytes of dynamic shared memory for `func`
// (set once per device; `done` is the caller's per-kernel bit set of devices already configured).
int launch_setup(const void* func, size_t smem, unsigned long long* done, int* sms);
size_t align256(size_t x);

// kernel launchers (one per translation unit)
// Layout of the selection's scratch behind the status block: pooled sums of Q and of K ([U, m, d] fp32 each),
// then the norm bounds of the pooled vectors ([U, m] fp32 each).
struct SelectWs { size_t pq, pk, nq, nk, total; };
SelectWs select_layout(const Geo& g);
int launch_select(const HostCtx& c, const void* q, const void* k, int32_t* block_idx, float* pooled_q,
                  float* pooled_k, float* norm_q, float* norm_k);
// What the attention kernel computes: kFwdUnion one softmax over local and selected blocks (o, lse); kFwdBranches the
// gated sum of the three branches (o, lse of the selection branch, lse_l of the local one; reads gates and the block-level
// output ocg); kFwdStats only what the three-branch backward needs of the forward: the gate gradients and, in two planes
// of [U, N] (local, selected), the negated base-2 log-sum-exp, -gate * <dO, O>, the gate and gate * dO.
enum { kFwdUnion = 0, kFwdBranches = 1, kFwdStats = 2 };
struct FwdOut {
  __nv_bfloat16* o;
  float *lse, *lse_l;
  const float *gates, *ocg;
  const __nv_bfloat16* d_o;
  float *dgates, *neg_lse2, *neg_d, *gate;
  void* gated_do;
};
int launch_fwd_tc(const HostCtx& c, int mode, const void* q, const void* k, const void* v, const int32_t* block_idx,
                  const FwdOut& out, int* work_counter);
// Layout of the three-branch forward's scratch behind the status block
struct BranchWs { size_t pq, pk, pv, ocg, total; };
BranchWs branch_layout(const Geo& g);
// Block sums (pool.cu).  A job is one tensor of `units` units, with or without norm bounds; with gates ([units, N, 3] fp32)
// every token is weighted by its first gate.  The launch also resets the status block.
constexpr int kPoolJobs = 4;
struct PoolJob {
  const void* src;
  float *dst, *norm;
  const float* gates;
  int units;
};
struct PoolArgs {
  PoolJob job[kPoolJobs];
  int n;
  int* status;
};
int launch_pool(const HostCtx& c, PoolArgs a);
// `lse2` (may be null): base-2 log-sum-exp of every query block's block-level logits, [U, m]
int launch_compress(const HostCtx& c, const float* pooled_q, const float* pooled_k, const float* pooled_v, float* ocg,
                    float* lse2);
// backward of the compression branch: pooled sums, dobar, obar and its log-sum-exp in; what every token of a block receives
// out (dqm [U, m, d], dkm, dvm [Ukv, m, d])
struct CompressBwd {
  const float *pq, *pk, *pv, *dob, *ocg, *lse2;
  float *dqm, *dkm, *dvm;
};
int launch_compress_bwd(const HostCtx& c, const CompressBwd& a);
int launch_rope(const HostCtx& c, const void* q, const void* k, const float* pos, double theta, void* q_out, void* k_out);
// What the attention backward reads per query row, [U, N] fp32: the negated base-2 log-sum-exp and -<dO, O>.  Three-branch
// form (gate set): two planes of each (local blocks, selected blocks), the second of them scaled by the gate, the gates
// themselves, dO scaled by each gate ([U, N, d] 16-bit, two planes), and what the compression branch gives every token of a block: dqm [U, m, d], dkm, dvm [Ukv, m, d].
struct RowStats {
  const float *neg_lse2, *neg_d, *gate, *dqm, *dkm, *dvm;
  const void* gated_do;
};
int launch_rowdot(const HostCtx& c, const void* o, const void* d_o, const float* lse, float* neg_d, float* neg_lse2);
int launch_dq_tc(const HostCtx& c, const void* q, const void* k, const void* v, const void* d_o, const RowStats& st,
                 const int32_t* block_idx, void* dq, int* work_counter);
int launch_dkdv_tc(const HostCtx& c, const void* q, const void* k, const void* v, const void* d_o, const RowStats& st,
                   const int32_t* csr_off, const int32_t* csr_q, void* dk, void* dv, int* work_counter, int32_t* order);
int launch_bwd(const HostCtx& c, const void* q, const void* k, const void* v, const RowStats& st, const void* d_o,
               const int32_t* block_idx, void* dq, void* dk, void* dv, int32_t* csr_off, int32_t* csr_q, int32_t* order,
               int* counters);

}  // namespace mosaic

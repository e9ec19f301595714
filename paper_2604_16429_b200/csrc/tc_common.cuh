// Device and host helpers shared by the tensor-core kernels (tcgen05 + TMEM + TMA): mbarrier waits with a
// bound, TMA loads, MMA issue, TMEM loads and stores, packed fp32 arithmetic, operand descriptors, and the
// planner routines that turn a 256-row work item into its merged, interleaved key list.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"

namespace mosaic {

namespace {

constexpr int kTile = 8192;                      // bytes of one 64 x 64 bf16 chunk
constexpr int kMaxUnion = 4 * kMaxList;          // most entries of an item's merged key list
constexpr int kLists = 4;                        // key lists in flight (the planner runs this far ahead)
// Barriers on which the key/value chunks of the row-stationary kernels land: one per ring position modulo kFullBars, many more
// than stages of data.  A tile's issuer looks only at the chunks its tile attends (the producer releases the others on its
// behalf), and a wait on a phase's parity is exact only if the barrier's previous phase has completed: with one barrier per
// stage the phase two rounds back, of an older chunk, passed for the awaited one.  What the issuer knows when it looks at a
// chunk: every earlier list is armed (the list's query tile was loaded after them), and in this list everything up to its
// last chunk.  An armed chunk means that the chunks a ring's length before it have landed, so the barrier's previous phase
// has completed if kFullBars is at least the longest list plus the stages.
constexpr int kFullBars = 512;
#ifdef MOSAIC_TEST_SPIN_CYCLES                   // test build only: a short bound, so that a wait that nothing ends runs out quickly
constexpr long long kSpinCycles = MOSAIC_TEST_SPIN_CYCLES;
#else
constexpr long long kSpinCycles = 4000000000ll;  // bound of a single wait (~2 s)
#endif

// A work item of the row-stationary kernels (forward, dQ) with the list that goes with it.  Its size is a power of two so that an
// index into the array is a shift (with 72 bytes the three-branch dQ takes 156 registers instead of 154).
struct alignas(128) RowItem {
  int n;        // entries of the merged list; -1 = no more work
  int unit;     // (batch, head) unit
  int hvalid;   // bit h: half h exists
  int branch;   // split lists: 0 = the selected blocks, 1 = the local ones
  int nsteps[2]; // entries that tile 0 and tile 1 attend
  int hb[4];    // query block of half h
  int hx[4], hy[4];  // column and row of the half's first token in the grid
};

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One poll.  The hardware parks the thread (for about 8000 cycles at most; it wakes as soon as the phase completes), so
// warps that wait do not take issue slots from warps that work.  No time hint: with one the wake-up takes 120 cycles
// after the arrival instead of 90.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false after the limit (status recorded) or once another thread aborted.
// The clock and the abort flag are looked at only every 64 polls to keep the poll loop light.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort, int* status) {
  const long long t0 = clock64();
#pragma unroll 1
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 0u) {
      if (*abort) return false;
      if (clock64() - t0 > kSpinCycles) {
        set_status(status, MOSAIC_E_DEVICE_TIMEOUT);
        *abort = 1;
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort, int* status) {
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, abort, status);
}

// A bounded wait of a converged warp whose lanes all wait for the same phase: the outcome is the same in every lane, and the
// usual case is one poll and one vote.
__device__ __noinline__ bool warp_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort, int* status) {
  return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, abort, status));
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort, int* status) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  return warp_wait_slow(bar, parity, abort, status);
}

// Abort path only: a bounded wait for phase `parity` of `bar` that records nothing.  After a failed wait the roles
// leave their loops with copies and tensor-core work possibly still in flight; the producer waits on the barriers it
// armed and each MMA issuer commits and waits once more, so that shared memory and TMEM are released only after
// everything that was issued has landed or run out of this (second, shorter) bound.
constexpr long long kDrainCycles = 4000000;  // about 2 ms per barrier
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > kDrainCycles) return false;
  return true;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, "
      "%6}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// One thread's tensor-core work issued so far has completed (or the bound ran out): commit to a barrier of its
// own (count 1, never used before) and wait for it.
__device__ __forceinline__ void mma_drain(uint32_t bar) {
  tc_commit(bar);
  mbar_drain(bar, 0);
}
// CTA prologue and epilogue that the tensor-core kernels share.  After the barriers are initialised (by one thread,
// followed by `cta_publish_barriers`), `alloc_warp` takes the whole of the SM's tensor memory and every thread
// reads its base address; at the end the same warp gives it back once every role has left its loop.
__device__ __forceinline__ void cta_publish_barriers() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ uint32_t cta_tmem_alloc(bool alloc_warp, uint32_t* slot, uint32_t cols) {
  __syncthreads();  // barrier initialisation is visible to every thread
  if (alloc_warp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(slot)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return *slot;
}
__device__ __forceinline__ void cta_tmem_free(bool alloc_warp, uint32_t tmem, uint32_t cols) {
  tc_fence_before();
  __syncthreads();
  if (alloc_warp) {
    tc_fence_after();
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
  }
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void umma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::
          "r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void umma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::
          "r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

#define MOSAIC_R16(r, o)                                                                                          \
  "=r"(r[o + 0]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]),  \
      "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]), "=r"(r[o + 11]), "=r"(r[o + 12]),           \
      "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15])
#define MOSAIC_W16(r, o)                                                                                     \
  "r"(r[o + 0]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), "r"(r[o + 6]),    \
      "r"(r[o + 7]), "r"(r[o + 8]), "r"(r[o + 9]), "r"(r[o + 10]), "r"(r[o + 11]), "r"(r[o + 12]),            \
      "r"(r[o + 13]), "r"(r[o + 14]), "r"(r[o + 15])

// 32 consecutive 32-bit TMEM columns of this thread's lane -> registers r[0..31]
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : MOSAIC_R16(r, 0), MOSAIC_R16(r, 16)
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : MOSAIC_R16(r, 0)
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      MOSAIC_W16(r, 0), MOSAIC_W16(r, 16)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};" ::"r"(taddr),
      MOSAIC_W16(r, 0)
      : "memory");
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// two fp32 lanes in one 64-bit register (packed fp32 arithmetic of this architecture)
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// two floats -> two 16-bit operands in one word (bf16, or binary16 when F16)
template <bool F16>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  uint32_t r;
  if (F16) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// 2^x for two values on the FMA pipe instead of the MUFU pipe (which caps the softmax at d = 64):
// x = n + f with n = round(x), |f| <= 1/2 (adding 1.5 * 2^23 leaves n in the low mantissa bits),
// 2^f by a cubic fitted to a maximum relative error of 1.0e-4 (P is rounded to bf16, 2^-9, afterwards),
// and 2^n by adding n to the exponent field.  Inputs are clamped at -125 so the exponent stays normal.
__device__ __forceinline__ void ex2_poly2(uint64_t x2, float& p0, float& p1) {
  float x0, x1;
  unpack2(x2, x0, x1);
  const uint64_t xc = pack2(fmaxf(x0, -125.f), fmaxf(x1, -125.f));
  const uint64_t t = add2(xc, pack2(12582912.f, 12582912.f));
  const uint64_t n = add2(t, pack2(-12582912.f, -12582912.f));
  const uint64_t f = fma2(n, pack2(-1.f, -1.f), xc);
  uint64_t p = fma2(f, pack2(0.05500893f, 0.05500893f), pack2(0.24221095f, 0.24221095f));
  p = fma2(p, f, pack2(0.6932829f, 0.6932829f));
  p = fma2(p, f, pack2(1.f, 1.f));
  float t0, t1, q0, q1;
  unpack2(t, t0, t1);
  unpack2(p, q0, q1);
  p0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
  p1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}

// Shared-memory operand descriptor: 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;               // leading byte offset (not used by these shapes)
  d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;               // descriptor version of this architecture
  d |= (uint64_t)2 << 61;               // SWIZZLE_128B
  return d;
}
// Instruction descriptor: 16-bit x 16-bit -> fp32 (both operands bf16, or both binary16 when f16), M = 128,
// N = 64 unless given.
__host__ __device__ constexpr uint32_t make_idesc(bool b_mn_major, uint32_t n = 64u, bool f16 = false) {
  return (1u << 4) | ((f16 ? 0u : 1u) << 7) | ((f16 ? 0u : 1u) << 10) | ((b_mn_major ? 1u : 0u) << 16) |
         ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// The four halves of work item `it` (index inside the unit).  Missing halves repeat half 0 (their rows
// are computed with every key masked and never stored).  Returns the bit set of existing halves.
__device__ __forceinline__ int item_halves(const Geo& g, int it, int (&hb)[4], int (&hc)[4]) {
  int valid = 0;
  if (g.cpb == 1) {
    const int ntx = (g.nbw + 1) >> 1, n_main = (g.nbh >> 1) * ntx;
    if (it < n_main) {  // 2 x 2 group
      const int gy = it / ntx, tx = it - gy * ntx;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int by = 2 * gy + (h >> 1), bx = 2 * tx + (h & 1);
        hb[h] = by * g.nbw + bx;
        hc[h] = 0;
        valid |= (bx < g.nbw) << h;
      }
    } else {            // odd last block row: 1 x 4 group
      const int bx0 = 4 * (it - n_main);
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        hb[h] = (g.nbh - 1) * g.nbw + bx0 + h;
        hc[h] = 0;
        valid |= (bx0 + h < g.nbw) << h;
      }
    }
  } else if (g.cpb == 2) {  // two neighbouring 128-token blocks: side by side, or one above the other in a one-column grid
    if (g.nbw > 1) {
      const int ntx = (g.nbw + 1) >> 1, by = it / ntx, tx = it - by * ntx;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int bx = 2 * tx + (h >> 1);
        hb[h] = by * g.nbw + bx;
        hc[h] = h & 1;
        valid |= (bx < g.nbw) << h;
      }
    } else {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int by = 2 * it + (h >> 1);
        hb[h] = by;
        hc[h] = h & 1;
        valid |= (by < g.nbh) << h;
      }
    }
  } else {                  // four chunks of one block
    const int ipb = (g.cpb + 3) >> 2, blk = it / ipb, c0 = 4 * (it - blk * ipb);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      hb[h] = blk;
      hc[h] = c0 + h;
      valid |= (c0 + h < g.cpb) << h;
    }
  }
#pragma unroll
  for (int h = 1; h < 4; ++h)
    if (!((valid >> h) & 1)) { hb[h] = hb[0]; hc[h] = hc[0]; }
  return valid;
}

// Work queue of the row-stationary kernels: `full` items of 256 rows, then the remaining items cut into `pieces` (1, 2 or 4)
// parts of 128 or 64 rows.
struct Queue {
  int full, pieces, positions;
};
// The item of queue position `pos`: its unit and index inside the unit in u and it; the position covers the item's halves
// first .. first + width - 1.
__device__ __forceinline__ void queue_item(const Queue& q, int pos, int ipu, int& u, int& it, int& first, int& width) {
  const int cut = max(pos - q.full, 0), item = min(pos, q.full) + cut / q.pieces;
  u = item / ipu;
  it = item - u * ipu;
  width = pos >= q.full ? 4 / q.pieces : 4;
  first = cut % q.pieces * width;
}
// Mask of an entry in the list of the halves first .. first + width - 1 (which come first there)
__device__ __forceinline__ unsigned part_mask(unsigned m, int first, int width) {
  const unsigned keep = (1u << width) - 1u;
  return ((m & 15u) >> first & keep) | ((m >> 4 >> first & keep) << 4);
}
// Drops the entries that none of the halves first .. first + width - 1 attends; returns the number of entries left.
__device__ __forceinline__ int keep_part(int* ids, unsigned char* mask, int n, int first, int width, int lane) {
  int kept = 0;
  for (int e0 = 0; e0 < n; e0 += 32) {
    const int e = e0 + lane, id = e < n ? ids[e] : 0;
    const unsigned m = e < n ? part_mask(mask[e], first, width) : 0u, act = __ballot_sync(0xffffffffu, m != 0u);
    __syncwarp();
    if (m) {
      const int at = kept + __popc(act & ((1u << lane) - 1u));
      ids[at] = id;
      mask[at] = (unsigned char)m;
    }
    kept += __popc(act);
    __syncwarp();
  }
  return kept;
}

// What a planner's lane needs of the geometry for every block it lists: its place in the local set (row and column offset; in
// group mode inside the group) and reciprocals for quick_div.  A CTA's first list (64-token blocks) takes the planner 11000 to
// 12700 cycles, 6000 of them the merge; a later one, beside busy row threads, 16000 (merge 9700), about as long as a short item:
// with integer divisions a selection and forward of 8 units of 28800 tokens took 188.3 us instead of 185.8.
struct Window {
  int dy, dx;
  bool in;  // the lane holds a place of the local set (columns that come round again in a narrow grid excluded)
  float inv_nbw, inv_rlat, inv_rlon;
};
__device__ __forceinline__ Window make_window(const Geo& g, int lane) {
  Window w;
  const int wide = g.local_groups ? g.rlon : 2 * g.rlon + 1, high = g.local_groups ? g.rlat : 2 * g.rlat + 1;
  w.dy = lane / wide;
  w.dx = lane - w.dy * wide;
  w.in = lane < high * wide && w.dx < g.nbw;
  if (!g.local_groups) { w.dy -= g.rlat; w.dx -= g.rlon; }
  w.inv_nbw = 1.0f / (float)g.nbw;
  w.inv_rlat = 1.0f / (float)max(g.rlat, 1);
  w.inv_rlon = 1.0f / (float)max(g.rlon, 1);
  return w;
}

// This lane's block of query block i's local set (-1: none); the lanes hold the set in list order.  In group mode the set is
// the aligned group of rlat x rlon blocks that holds block i (ragged at the grid's edge), else the window, whose rows beyond the
// grid fold onto rows that it holds anyway.
__device__ __forceinline__ int local_id(const Geo& g, const Window& w, int i) {
  const int by = quick_div(i, g.nbw, w.inv_nbw), bx = i - by * g.nbw;
  const int y = (g.local_groups ? quick_div(by, g.rlat, w.inv_rlat) * g.rlat : by) + w.dy;
  int x = (g.local_groups ? quick_div(bx, g.rlon, w.inv_rlon) * g.rlon : bx) + w.dx;
  const bool keep = w.in && y >= 0 && y < g.nbh && !(g.local_groups && x >= g.nbw);
#pragma unroll
  for (int k = 0; k < 2; ++k) {  // longitude is periodic (offsets of at most two, a grid may be one column wide)
    x += x < 0 ? g.nbw : 0;
    x -= x >= g.nbw ? g.nbw : 0;
  }
  return keep ? y * g.nbw + x : -1;
}
// This lane's entry j of query block i's row of block_idx, -1 if it is none or one that is skipped and reported: an id outside
// [-1, m), inside the local set (attended already) or repeated in the row.
__device__ __forceinline__ int selected_id(const Geo& g, const Window& w, int i, int j, int lane, int* status) {
  const unsigned twins = __match_any_sync(0xffffffffu, j);
  if (j == -1) return -1;
  bool bad = j < 0 || j >= g.m || (__ffs(twins) - 1) != lane;
  if (!bad) {
    const int by = quick_div(i, g.nbw, w.inv_nbw), bx = i - by * g.nbw, jy = quick_div(j, g.nbw, w.inv_nbw), jx = j - jy * g.nbw;
    if (g.local_groups) {
      bad = quick_div(jy, g.rlat, w.inv_rlat) == quick_div(by, g.rlat, w.inv_rlat) &&
            quick_div(jx, g.rlon, w.inv_rlon) == quick_div(bx, g.rlon, w.inv_rlon);
    } else {
      int dx = jx - bx;
      dx += dx < 0 ? g.nbw : 0;  // (jx - bx) mod nbw in [0, nbw)
      bad = abs(jy - by) <= g.rlat && (dx <= g.rlon || g.nbw - dx <= g.rlon);
    }
  }
  if (bad) set_status(status, MOSAIC_E_DEVICE_BAD_INDEX);
  return bad ? -1 : j;
}

// Merges the list of a query block into the item's list (ids/mask, n entries so far): the blocks id0 of all lanes, then the
// blocks id1 (-1: none; no block twice).  Entries already present get the bits OR-ed into their mask, new ones are appended.
// Returns the new n.
__device__ __forceinline__ int merge_list(int id0, unsigned bits0, int id1, unsigned bits1, int* ids, unsigned char* mask, int n,
                                          int lane) {
  const int n0 = n;
  int pos0 = -1, pos1 = -1;
#pragma unroll 4
  for (int a = 0; a < n0; a += 4) {
    const int4 v = *reinterpret_cast<const int4*>(ids + a);
    const int id[4] = {v.x, a + 1 < n0 ? v.y : -2, a + 2 < n0 ? v.z : -2, a + 3 < n0 ? v.w : -2};
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      pos0 = id[x] == id0 ? a + x : pos0;
      pos1 = id[x] == id1 ? a + x : pos1;
    }
  }
  __syncwarp();
  const bool new0 = id0 >= 0 && pos0 < 0, new1 = id1 >= 0 && pos1 < 0;
  const unsigned m0 = __ballot_sync(0xffffffffu, new0), m1 = __ballot_sync(0xffffffffu, new1), lower = (1u << lane) - 1u;
  if (id0 >= 0) {
    const int at = new0 ? n + __popc(m0 & lower) : pos0;
    mask[at] = (unsigned char)(new0 ? bits0 : mask[at] | bits0);
    if (new0) ids[at] = id0;
  }
  n += __popc(m0);
  if (id1 >= 0) {
    const int at = new1 ? n + __popc(m1 & lower) : pos1;
    mask[at] = (unsigned char)(new1 ? bits1 : mask[at] | bits1);
    if (new1) ids[at] = id1;
  }
  __syncwarp();
  return n + __popc(m1);
}

// One lane of a converged warp (the same lane every time).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}

// Reorder a merged key list so that both tiles, and both 64-row halves of a tile, find work all along it.
// Entries fall into seven classes by who attends them: tile 0 only (upper half, lower half, both halves), both
// tiles, tile 1 only (upper, lower, both).  The k-th entry of a class of n gets the fractional position
// (8k + class) / (8n), so every class is spread evenly; in particular products that only the upper half of a
// tile attends alternate with products only its lower half attends, and since S is double-buffered the idle
// half's warps run ahead into the next product.  The order of a softmax sum does not matter to the result
// beyond rounding; the order is a function of the list alone.
// An entry's mask: bit h = half h attends it; in tagged lists bit 4 + h = half h attends it as a selected block, bit h as
// a local one.
__device__ __forceinline__ unsigned who_attends(unsigned m) { return (m | (m >> 4)) & 15u; }
__device__ __forceinline__ int list_class(unsigned m) {
  const unsigned t0 = m & 3u, t1 = (m >> 2) & 3u;
  return t1 == 0u ? (int)t0 - 1 : t0 == 0u ? 3 + (int)t1 : 3;
}
__device__ __forceinline__ void interleave_tiles(const int* sid, const unsigned char* smask, int n, int* did,
                                                 unsigned char* dmask, int lane) {
  constexpr int NC = 7;
  int cnt[NC];
#pragma unroll
  for (int y = 0; y < NC; ++y) cnt[y] = 0;
  for (int e0 = 0; e0 < n; e0 += 32) {
    const int e = e0 + lane;
    const int cls = e < n ? list_class(who_attends(smask[e])) : -1;
#pragma unroll
    for (int y = 0; y < NC; ++y) cnt[y] += __popc(__ballot_sync(0xffffffffu, cls == y));
  }
  int base[NC];
#pragma unroll
  for (int y = 0; y < NC; ++y) base[y] = 0;
  for (int e0 = 0; e0 < n; e0 += 32) {
    const int e = e0 + lane;
    const unsigned m = e < n ? smask[e] : 0u;
    const int cls = e < n ? list_class(who_attends(m)) : -1;
    const unsigned lower = (1u << lane) - 1u;
    int k = 0, nx = 1;
#pragma unroll
    for (int y = 0; y < NC; ++y) {
      const unsigned by = __ballot_sync(0xffffffffu, cls == y);
      if (cls == y) { k = base[y] + __popc(by & lower); nx = cnt[y]; }
      base[y] += __popc(by);
    }
    if (e < n) {
      int pos = k;
      const int step = 8 * nx;
      const float inv = 1.0f / (float)step;
#pragma unroll
      for (int y = 0; y < NC; ++y) {
        const int ny = cnt[y];
        // entries j of class y that come first: (8j + y) nx < (8k + cls) ny, ties to the lower class: one more than the
        // quotient, if there is one (all below 2^20, where the rounded quotient is off by at most one; 191.3 us with divisions, 188.9
        // without, in the pass named at Window)
        const int R = (8 * k + cls) * ny - y * nx - (y > cls ? 1 : 0);
        int q = __float2int_rz((float)R * inv);
        const int r = R - q * step;
        q += r >= step ? 1 : r < 0 ? -1 : 0;
        if (y != cls && R >= 0) pos += min(q + 1, ny);
      }
      did[pos] = sid[e];
      dmask[pos] = (unsigned char)m;
    }
  }
  __syncwarp();
}

// The entries of an item's list that each tile attends: per entry the tile's halves (bits 0, 1), whether they attend it as
// a selected block (bits 2, 3, tagged lists) and, from bit 8, the entry's place in the list.
__device__ __forceinline__ void tile_steps(const unsigned char* mask, int n, unsigned short (*steps)[kMaxUnion], int* nsteps,
                                           int lane) {
  int cnt[2] = {0, 0};
  for (int e0 = 0; e0 < n; e0 += 32) {
    const int e = e0 + lane;
    const unsigned m = e < n ? mask[e] : 0u;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const unsigned code = (who_attends(m) >> (2 * t)) & 3u;
      const unsigned act = __ballot_sync(0xffffffffu, code != 0u);
      if (code)
        steps[t][cnt[t] + __popc(act & ((1u << lane) - 1u))] =
            (unsigned short)(code | (((m >> (4 + 2 * t)) & 3u) << 2) | ((unsigned)e << 8));
      cnt[t] += __popc(act);
    }
  }
  if (lane == 0) { nsteps[0] = cnt[0]; nsteps[1] = cnt[1]; }
}

// Planner warp: draws work items from the queue (the first item of a CTA is its own index) and builds each
// item's merged, interleaved key list one or more items ahead of the warps that consume it.  `SM` is the
// kernel's shared-memory struct (info, ids, mask, steps, tmp_ids, tmp_mask, list_full, list_empty).
//   kPlanUnion:  one list, the union of the local and the selected blocks
//   kPlanSplit:  two lists per item, the selected blocks (info.branch 0), then the local ones (1)
//   kPlanTagged: one list like kPlanUnion's whose masks tell the two kinds apart
enum { kPlanUnion = 0, kPlanSplit = 1, kPlanTagged = 2 };
template <int PLAN, class SM>
__device__ __forceinline__ void planner_loop(SM& sm, const Geo& g, const int32_t* __restrict__ block_idx,
                                             int* work_counter, int ipu, const Queue& queue, int lane,
                                             volatile int* abort, int* status) {
  int lb = 0;  // list buffers handed out so far
  bool ok = true;
  const Window w = make_window(g, lane);
  auto acquire = [&]() {  // wait until list buffer lb % kLists is free
    if (lane == 0) ok = mbar_wait(s32(&sm.list_empty[lb % kLists]), ((lb / kLists) & 1) ^ 1, abort, status);
    ok = __shfl_sync(0xffffffffu, ok, 0);
  };
  for (int it = 0; ok; ++it) {
    int item = 0;
    // the first item of a CTA is its own index; later ones come from the queue, which counts from 0
    if (lane == 0) item = it == 0 ? (int)blockIdx.x : atomicAdd(work_counter, 1) + (int)gridDim.x;
    item = __shfl_sync(0xffffffffu, item, 0);
    acquire();
    if (!ok) break;
    if (item >= queue.positions) {
      if (lane == 0) { sm.info[lb % kLists].n = -1; mbar_arrive(s32(&sm.list_full[lb % kLists])); }
      break;
    }
    int u, in_unit, first, width, hb[4], hc[4];
    queue_item(queue, item, ipu, u, in_unit, first, width);
    const int valid = item_halves(g, in_unit, hb, hc);
    int jsel[4];  // the four rows of block_idx, fetched together
#pragma unroll
    for (int h = 0; h < 4; ++h)
      jsel[h] = lane < g.topk ? __ldg(block_idx + ((long long)u * g.m + hb[h]) * g.topk + lane) : -1;
    for (int part = 0; part < (PLAN == kPlanSplit ? 2 : 1); ++part) {
      if (part > 0) {
        acquire();
        if (!ok) break;
      }
      int n = 0;
#pragma unroll 1
      for (int h = 0; h < 4; ++h) {  // (one copy of the code: with four, 186.0 us instead of 183.0 in the pass named at Window)
        const int blk = h == 0 ? hb[0] : h == 1 ? hb[1] : h == 2 ? hb[2] : hb[3];
        const int j = h == 0 ? jsel[0] : h == 1 ? jsel[1] : h == 2 ? jsel[2] : jsel[3];
        unsigned bits = 0;  // the halves of this block
#pragma unroll
        for (int h2 = 0; h2 < 4; ++h2) bits |= ((valid >> h2) & 1) && hb[h2] == blk ? 1u << h2 : 0u;
        if (!((valid >> h) & 1) || (bits & ((1u << h) - 1u))) continue;  // missing, or listed with the block's first half
        const int loc = PLAN != kPlanSplit || part == 1 ? local_id(g, w, blk) : -1;
        const int sel = PLAN != kPlanSplit || part == 0 ? selected_id(g, w, blk, j, lane, status) : -1;
        n = merge_list(loc, bits, sel, PLAN == kPlanTagged ? bits << 4 : bits, sm.tmp_ids, sm.tmp_mask, n, lane);
      }
      if (g.cpb == 1 && valid == 0xF && part == 0) {
        // Four different query blocks: which two share a 128-row tile is free.  Take the pairing whose tiles have
        // the most entries in common (fewest products with a masked half); ties keep the first pairing.  (Split
        // lists: the selected blocks decide; the local sets of neighbouring blocks overlap alike.)
        int o01 = 0, o23 = 0, o02 = 0, o13 = 0, o03 = 0, o12 = 0;
        for (int e0 = 0; e0 < n; e0 += 32) {
          const unsigned mk = e0 + lane < n ? who_attends(sm.tmp_mask[e0 + lane]) : 0u;
          o01 += __popc(__ballot_sync(0xffffffffu, (mk & 3u) == 3u));
          o23 += __popc(__ballot_sync(0xffffffffu, (mk & 12u) == 12u));
          o02 += __popc(__ballot_sync(0xffffffffu, (mk & 5u) == 5u));
          o13 += __popc(__ballot_sync(0xffffffffu, (mk & 10u) == 10u));
          o03 += __popc(__ballot_sync(0xffffffffu, (mk & 9u) == 9u));
          o12 += __popc(__ballot_sync(0xffffffffu, (mk & 6u) == 6u));
        }
        const int s0 = o01 + o23, s1 = o02 + o13, s2 = o03 + o12;
        const int pick = (s1 > s0 && s1 >= s2) ? 1 : (s2 > s0 && s2 > s1) ? 2 : 0;
        if (pick != 0) {
          // new half k is old half perm[k]: (0,2,1,3) pairs the blocks vertically, (0,3,1,2) diagonally
          const int p1 = pick == 1 ? 2 : 3, p2 = 1, p3 = pick == 1 ? 3 : 2;
          for (int e = lane; e < n; e += 32) {
            const unsigned mk = sm.tmp_mask[e];
            sm.tmp_mask[e] = (unsigned char)((mk & 0x11u) | (((mk >> p1) & 0x11u) << 1) | (((mk >> p2) & 0x11u) << 2) |
                                             (((mk >> p3) & 0x11u) << 3));
          }
          const int b1 = hb[p1], b2 = hb[p2], b3 = hb[p3], c1 = hc[p1], c2 = hc[p2], c3 = hc[p3];
          hb[1] = b1; hb[2] = b2; hb[3] = b3;
          hc[1] = c1; hc[2] = c2; hc[3] = c3;
          __syncwarp();
        }
      }
      const int buf = lb % kLists;
      interleave_tiles(sm.tmp_ids, sm.tmp_mask, n, sm.ids[buf], sm.mask[buf], lane);
      // A part keeps the order of the whole item's list: a row's result must not depend on where the queue cuts, which
      // depends on the number of units and of SMs.  (A 32 x 64 grid, all of which is cut: 30.4 us a pass with lists of the
      // parts' own blocks, 32.0 so.)
      if (width < 4) n = keep_part(sm.ids[buf], sm.mask[buf], n, first, width, lane);
      tile_steps(sm.mask[buf], n, sm.steps[buf], sm.info[buf].nsteps, lane);
      if (lane == 0) {
        RowItem& inf = sm.info[buf];
        inf.n = n; inf.unit = u; inf.hvalid = (int)part_mask((unsigned)valid, first, width); inf.branch = part;
      }
      if (lane < 4) {
        RowItem& inf = sm.info[buf];
        const int from = first + (lane < width ? lane : 0);
        const int b = from == 0 ? hb[0] : from == 1 ? hb[1] : from == 2 ? hb[2] : hb[3];
        const int c = from == 0 ? hc[0] : from == 1 ? hc[1] : from == 2 ? hc[2] : hc[3];
        const int by = quick_div(b, g.nbw, w.inv_nbw);
        inf.hb[lane] = b;
        inf.hx[lane] = (b - by * g.nbw) * g.bw;
        inf.hy[lane] = by * g.bh + c * g.crows;
      }
      __syncwarp();
      ++lb;
#ifdef MOSAIC_TEST_WITHHOLD_FIRST_LIST  // test build only: the CTA's first list is never published, so every consumer's wait runs out
      if (lb == 1) continue;
#endif
      if (lane == 0) mbar_arrive(s32(&sm.list_full[buf]));
    }
  }
}

// Producer warp: the key and value chunks of a list through the ring (`step`: ring position of the next chunk).  The whole warp
// walks the list, and its lanes work out where 32 entries lie at once: in the forward of 192 units of 28800 tokens (64-token
// blocks) one lane that divided once per entry took 830 cycles a chunk beside the row threads (conversions and reciprocals queue
// behind their exponentials).  Returns false after a failed wait.
template <int STAGES, class SM>
__device__ __forceinline__ bool produce_chunks(SM& sm, const Geo& g, const CUtensorMap* map_k, const CUtensorMap* map_v, int buf,
                                               int n, int ukv, uint32_t& step, int lane, volatile int* abort, int* status) {
  for (int e0 = 0; e0 < n; e0 += 32) {
    const int e = e0 + lane, j = e < n ? sm.ids[buf][e] : 0, by = j / g.nbw, x = (j - by * g.nbw) * g.bw, y = by * g.bh;
    const unsigned m = e < n ? who_attends(sm.mask[buf][e]) : 0u;
    const int here = min(32, n - e0);
    for (int i = 0; i < here; ++i) {
      const int cx = __shfl_sync(0xffffffffu, x, i);
      int cy = __shfl_sync(0xffffffffu, y, i);
      const unsigned mk = __shfl_sync(0xffffffffu, m, i);
      for (int c = 0; c < g.cpb; ++c, ++step, cy += g.crows) {
        const uint32_t st = step % STAGES, full = s32(&sm.kv_full[step % kFullBars]), empty = s32(&sm.kv_empty[st]);
        if (!warp_wait(empty, ((step / STAGES) & 1) ^ 1, abort, status)) return false;
        if (elect_one()) {
          mbar_expect_tx(full, 2 * kTile);
          tma_load_4d(s32(sm.kv[st][0]), map_k, full, 0, cx, cy, ukv);
          tma_load_4d(s32(sm.kv[st][1]), map_v, full, 0, cx, cy, ukv);
          // a tile that does not attend this entry never looks at the stage: its release is given here (the other
          // tile's release, after its products, is what lets the stage be reused)
          if (!(mk & 3u)) mbar_arrive(empty);
          if (!(mk & 12u)) mbar_arrive(empty);
        }
        __syncwarp();
      }
    }
  }
  return true;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
      "[%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
}  // namespace

// Cuts the last, partly filled round of items (one item per SM and round) into parts, as finely as they still fit one round: a
// part walks a shorter list, alone on its SM.  Forward in us, uncut and cut, at items = full rounds x 148 + rest (one unit of
// 2 x 2 groups of 64-token blocks, top-k 8; 128-token blocks alike): 20 items 27.8 / 20.2, 37 (the most for quarters) 29.1 /
// 20.7, 38 (halves) 28.6 / 23.8, 74 (the most for halves) 29.5 / 24.3, 148 + 2 48.0 / 39.5, 148 + 42 48.7 / 43.6, 296 + 34
// 67.8 / 59.7, 444 + 6 86.5 / 78.0, 592 + 38 105.7 / 101.0, 888 + 16 142.9 / 134.9; a rest that is not cut changes nothing.
inline Queue make_queue(long long items, int sms) {
  const int rem = (int)(items % sms), pieces = rem * 4 <= sms ? 4 : rem * 2 <= sms ? 2 : 1;
  Queue q;
  q.full = (int)items - rem;
  q.pieces = pieces;
  q.positions = q.full + rem * pieces;
  return q;
}

// ---- host side (tmap.cu) -------------------------------------------------------------------
// TMA descriptors are cached per (device, base pointer, geometry), so a call that sees the same tensors
// again encodes nothing.
// [units, nlat, nlon, d] bf16 view, box = one 64-token chunk {d, bw, 64/bw, 1}, 128-byte swizzle.
bool make_map(CUtensorMap* map, const void* base, const Geo& g, int units);
// [units, nlat, nlon] fp32 view (one value per token), box = the 64 tokens of one chunk {bw, 64/bw, 1}, no swizzle.
bool make_map_rows(CUtensorMap* map, const void* base, const Geo& g, int units);
}  // namespace mosaic

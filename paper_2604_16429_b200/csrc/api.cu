// C ABI of the library: argument validation, workspace carving, kernel launches.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include "common.cuh"

namespace mosaic {

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

int validate(const mosaic_bsa_params* p, Geo* g) {
  if (!p) return MOSAIC_E_INVALID_ARG;
  if (p->B <= 0 || p->H <= 0 || p->nlat <= 0 || p->nlon <= 0 || p->bh <= 0 || p->bw <= 0 || p->topk < 0 ||
      p->rlat < 0 || p->rlon < 0 || (p->flags & ~(MOSAIC_FLAG_LOCAL_GROUPS | MOSAIC_FLAG_FP16)) != 0)
    return MOSAIC_E_INVALID_ARG;
  if (p->nlat % p->bh || p->nlon % p->bw) return MOSAIC_E_INVALID_ARG;
  if (!(p->scale == p->scale) || isinf(p->scale)) return MOSAIC_E_INVALID_ARG;
  if (p->d != kD) return MOSAIC_E_UNSUPPORTED;
  if (!(p->bw == 8 || p->bw == 16)) return MOSAIC_E_UNSUPPORTED;
  const int crows = kChunk / p->bw;
  if (p->bh % crows) return MOSAIC_E_UNSUPPORTED;
  const int cpb = p->bh * p->bw / kChunk;
  if (!(cpb == 1 || cpb % 2 == 0)) return MOSAIC_E_UNSUPPORTED;
  const bool groups = (p->flags & MOSAIC_FLAG_LOCAL_GROUPS) != 0;
  if (groups && (p->rlat < 1 || p->rlon < 1)) return MOSAIC_E_INVALID_ARG;
  if (p->topk > kMaxTopk) return MOSAIC_E_UNSUPPORTED;
  if (groups ? (long long)p->rlat * p->rlon > 32 : (p->rlat > 2 || p->rlon > 2)) return MOSAIC_E_UNSUPPORTED;
  const int nlocal = groups ? p->rlat * p->rlon : (2 * p->rlat + 1) * (2 * p->rlon + 1);
  if (nlocal + p->topk > kMaxList) return MOSAIC_E_UNSUPPORTED;
  const long long U = (long long)p->B * p->H, N = (long long)p->nlat * p->nlon;
  const long long m = (long long)(p->nlat / p->bh) * (p->nlon / p->bw);
  if (U > (1 << 24) || m > (1 << 24) || U * m * cpb > 0x7fffffffll || U * N > (1ll << 40)) return MOSAIC_E_UNSUPPORTED;
  const int hkv = p->Hkv == 0 ? p->H : p->Hkv;
  if (hkv <= 0 || p->H % hkv) return MOSAIC_E_INVALID_ARG;
  g->U = (int)U;
  g->H = p->H; g->Hkv = hkv; g->Ukv = p->B * hkv;
  g->nlat = p->nlat; g->nlon = p->nlon; g->bh = p->bh; g->bw = p->bw;
  g->nbh = p->nlat / p->bh; g->nbw = p->nlon / p->bw; g->m = (int)m;
  g->b = p->bh * p->bw; g->cpb = cpb; g->crows = crows;
  g->rlat = p->rlat; g->rlon = p->rlon; g->topk = p->topk;
  g->local_groups = groups ? 1 : 0;
  g->f16 = (p->flags & MOSAIC_FLAG_FP16) ? 1 : 0;
  g->scale = p->scale > 0.f ? p->scale : 1.0f / sqrtf((float)p->d);
  g->scale_log2 = g->scale * 1.4426950408889634f;
  g->N = N;
  return MOSAIC_OK;
}

SelectWs select_layout(const Geo& g) {
  SelectWs w;
  const size_t pooled = align256(sizeof(float) * (size_t)g.U * g.m * kD), norms = align256(sizeof(float) * (size_t)g.U * g.m);
  w.pq = kStatusBytes;
  w.pk = w.pq + pooled;
  w.nq = w.pk + pooled;
  w.nk = w.nq + norms;
  w.total = w.nk + norms;
  return w;
}

BranchWs branch_layout(const Geo& g) {
  BranchWs w;
  const size_t pooled = align256(sizeof(float) * (size_t)g.U * g.m * kD);
  w.pq = kStatusBytes;
  w.pk = w.pq + pooled;
  w.pv = w.pk + pooled;
  w.ocg = w.pv + pooled;
  w.total = w.ocg + pooled;
  return w;
}

namespace {

struct BwdWs { size_t neg_d, neg_lse2, gate, gated_do, off, q, order, total; };
// `planes`: sets of row statistics (two, and the gates, in the three-branch form)
BwdWs bwd_layout(const Geo& g, int planes, size_t at) {
  BwdWs w;
  const size_t rows = align256(sizeof(float) * (size_t)planes * g.U * g.N);
  w.neg_d = at; at += rows;
  w.neg_lse2 = at; at += rows;
  w.gate = at; at += planes > 1 ? rows : 0;
  w.gated_do = at; at += planes > 1 ? align256(2 * (size_t)planes * g.U * g.N * kD) : 0;
  w.off = at; at = align256(at + sizeof(int32_t) * (size_t)g.U * (g.m + 1));
  w.q = at; at = align256(at + sizeof(int32_t) * (size_t)g.U * g.m * (g.topk > 0 ? g.topk : 1));
  // dK/dV items (two 128-row tiles per 256-row item of a key/value unit), longest first, and their cost classes
  w.order = at; at = align256(at + 2 * sizeof(int32_t) * 2 * (size_t)g.Ukv * items_per_unit(g));
  w.total = at;
  return w;
}
// Scratch of the three-branch backward: the forward's (pooled sums, obar), the block-level backward's vectors and the
// attention backward's own scratch.
struct BwdBranchWs {
  BranchWs f;
  size_t lse_cg, dob, dqm, dkm, dvm;
  BwdWs b;
};
BwdBranchWs bwd_branch_layout(const Geo& g) {
  BwdBranchWs w;
  w.f = branch_layout(g);
  const size_t pooled = align256(sizeof(float) * (size_t)g.U * g.m * kD), blocks = align256(sizeof(float) * (size_t)g.U * g.m);
  size_t at = w.f.total;
  w.lse_cg = at; at += blocks;
  w.dob = at; at += pooled;
  w.dqm = at; at += pooled;
  w.dkm = at; at += pooled;
  w.dvm = at; at += pooled;
  w.b = bwd_layout(g, 2, at);
  return w;
}
PoolArgs branch_pool(const Geo& g, const void* q, const void* k, const void* v, float* pq, float* pk, float* pv) {
  PoolArgs a = {};
  a.n = 3;
  a.job[0] = {q, pq, nullptr, nullptr, g.U};
  a.job[1] = {k, pk, nullptr, nullptr, g.Ukv};
  a.job[2] = {v, pv, nullptr, nullptr, g.Ukv};
  return a;
}
size_t select_total(const Geo& g) { return select_layout(g).total; }

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

int device_ok() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MOSAIC_E_CUDA;
  if (dev < 64 && cached[dev]) return cached[dev] > 0 ? MOSAIC_OK : MOSAIC_E_UNSUPPORTED;
  int major = 0;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return MOSAIC_E_CUDA;
  if (dev < 64) cached[dev] = major == 10 ? 1 : -1;
  return major == 10 ? MOSAIC_OK : MOSAIC_E_UNSUPPORTED;
}

// Clears the status block.  A memset there ended the overlap of launches: a pass over 2048 tokens 40.4 against 38.0 us.
__global__ void reset_kernel(int* status) { status[threadIdx.x + await_stream()] = 0; }

// `reset`: the status block is cleared here (otherwise the op's first kernel does it)
int begin(const mosaic_bsa_params* p, void* ws, size_t ws_bytes, size_t need, void* stream, HostCtx* c, bool reset) {
  int rc = validate(p, &c->g);
  if (rc) return rc;
  if (!ws) return MOSAIC_E_INVALID_ARG;
  if (!aligned(ws, 256)) return MOSAIC_E_MISALIGNED;
  if (ws_bytes < need) return MOSAIC_E_WORKSPACE_TOO_SMALL;
  if ((rc = device_ok())) return rc;
  c->stream = (cudaStream_t)stream;
  c->status = (int*)ws;
  return reset ? launch_kernel(reset_kernel, dim3(1), kStatusBytes / 4, 0, c->stream, true, 0, c->status) : MOSAIC_OK;
}

}  // namespace
}  // namespace mosaic

using namespace mosaic;

extern "C" {

size_t mosaic_bsa_workspace_bytes(const mosaic_bsa_params* p, int op) {
  Geo g;
  if (validate(p, &g)) return 0;
  switch (op) {
    case MOSAIC_OP_SELECT: return select_total(g);
    case MOSAIC_OP_FWD: return kStatusBytes;
    case MOSAIC_OP_BWD: return bwd_layout(g, 1, kStatusBytes).total;
    case MOSAIC_OP_FWD_BRANCHES: return branch_layout(g).total;
    case MOSAIC_OP_BWD_BRANCHES: return bwd_branch_layout(g).b.total;
    default: return 0;
  }
}

int mosaic_bsa_select(const mosaic_bsa_params* p, const void* q, const void* k, int32_t* block_idx, void* ws,
                      size_t ws_bytes, void* cuda_stream) {
  HostCtx c;
  Geo g;
  int rc = validate(p, &g);
  if (rc) return rc;
  if (!q || !k || (!block_idx && g.topk > 0)) return MOSAIC_E_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k, 16) || !aligned(block_idx, 4)) return MOSAIC_E_MISALIGNED;
  if ((rc = begin(p, ws, ws_bytes, select_total(g), cuda_stream, &c, false))) return rc;
  const SelectWs w = select_layout(g);
  char* base = (char*)ws;
  return launch_select(c, q, k, block_idx, (float*)(base + w.pq), (float*)(base + w.pk), (float*)(base + w.nq),
                       (float*)(base + w.nk));
}

int mosaic_bsa_fwd(const mosaic_bsa_params* p, const void* q, const void* k, const void* v,
                   const int32_t* block_idx, void* o, float* lse, void* ws, size_t ws_bytes, void* cuda_stream) {
  HostCtx c;
  Geo g;
  int rc = validate(p, &g);
  if (rc) return rc;
  if (!q || !k || !v || !o || !lse || (!block_idx && g.topk > 0)) return MOSAIC_E_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k, 16) || !aligned(v, 16) || !aligned(o, 16) || !aligned(lse, 4) ||
      !aligned(block_idx, 4))
    return MOSAIC_E_MISALIGNED;
  if ((rc = begin(p, ws, ws_bytes, kStatusBytes, cuda_stream, &c, true))) return rc;
  FwdOut out = {};
  out.o = (__nv_bfloat16*)o;
  out.lse = lse;
  return launch_fwd_tc(c, kFwdUnion, q, k, v, block_idx, out, c.status + 1);
}

int mosaic_bsa_fwd_branches(const mosaic_bsa_params* p, const void* q, const void* k, const void* v,
                            const int32_t* block_idx, const float* gates, void* o, float* lse_fg, float* lse_l, void* ws,
                            size_t ws_bytes, void* cuda_stream) {
  HostCtx c;
  Geo g;
  int rc = validate(p, &g);
  if (rc) return rc;
  if (!q || !k || !v || !gates || !o || !lse_fg || !lse_l || (!block_idx && g.topk > 0)) return MOSAIC_E_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k, 16) || !aligned(v, 16) || !aligned(o, 16) || !aligned(gates, 4) ||
      !aligned(lse_fg, 4) || !aligned(lse_l, 4) || !aligned(block_idx, 4))
    return MOSAIC_E_MISALIGNED;
  const BranchWs w = branch_layout(g);
  if ((rc = begin(p, ws, ws_bytes, w.total, cuda_stream, &c, false))) return rc;
  char* base = (char*)ws;
  float *pq = (float*)(base + w.pq), *pk = (float*)(base + w.pk), *pv = (float*)(base + w.pv);
  float* ocg = (float*)(base + w.ocg);
  // compression branch: pooled sums of Q, K and V, then block-level attention
  if ((rc = launch_pool(c, branch_pool(g, q, k, v, pq, pk, pv)))) return rc;
  if ((rc = launch_compress(c, pq, pk, pv, ocg, nullptr))) return rc;
  // selection and local branch, each with its own softmax, and the gated sum
  FwdOut out = {};
  out.o = (__nv_bfloat16*)o;
  out.lse = lse_fg;
  out.lse_l = lse_l;
  out.gates = gates;
  out.ocg = ocg;
  return launch_fwd_tc(c, kFwdBranches, q, k, v, block_idx, out, c.status + 1);
}

int mosaic_bsa_bwd(const mosaic_bsa_params* p, const void* q, const void* k, const void* v, const void* o,
                   const float* lse, const void* d_o, const int32_t* block_idx, void* dq, void* dk, void* dv,
                   void* ws, size_t ws_bytes, void* cuda_stream) {
  HostCtx c;
  Geo g;
  int rc = validate(p, &g);
  if (rc) return rc;
  if (!q || !k || !v || !o || !lse || !d_o || !dq || !dk || !dv || (!block_idx && g.topk > 0))
    return MOSAIC_E_INVALID_ARG;
  const void* ptrs[] = {q, k, v, o, d_o, dq, dk, dv};
  for (const void* x : ptrs)
    if (!aligned(x, 16)) return MOSAIC_E_MISALIGNED;
  if (!aligned(lse, 4) || !aligned(block_idx, 4)) return MOSAIC_E_MISALIGNED;
  if (2 * (size_t)g.m * sizeof(int) + (size_t)g.m * g.topk / 8 + 8 > 200 * 1024) return MOSAIC_E_UNSUPPORTED;  // transposed-pattern kernel
  const BwdWs w = bwd_layout(g, 1, kStatusBytes);
  if ((rc = begin(p, ws, ws_bytes, w.total, cuda_stream, &c, false))) return rc;
  char* base = (char*)ws;
  float *neg_d = (float*)(base + w.neg_d), *neg_lse2 = (float*)(base + w.neg_lse2);
  if ((rc = launch_rowdot(c, o, d_o, lse, neg_d, neg_lse2))) return rc;
  RowStats st = {};
  st.neg_lse2 = neg_lse2;
  st.neg_d = neg_d;
  return launch_bwd(c, q, k, v, st, d_o, block_idx, dq, dk, dv, (int32_t*)(base + w.off), (int32_t*)(base + w.q),
                    (int32_t*)(base + w.order), c.status + 1);
}

int mosaic_bsa_bwd_branches(const mosaic_bsa_params* p, const void* q, const void* k, const void* v,
                            const int32_t* block_idx, const float* gates, const void* d_o, void* dq, void* dk,
                            void* dv, float* dgates, void* ws, size_t ws_bytes, void* cuda_stream) {
  HostCtx c;
  Geo g;
  int rc = validate(p, &g);
  if (rc) return rc;
  if (!q || !k || !v || !gates || !d_o || !dq || !dk || !dv || !dgates || (!block_idx && g.topk > 0))
    return MOSAIC_E_INVALID_ARG;
  const void* ptrs[] = {q, k, v, d_o, dq, dk, dv};
  for (const void* x : ptrs)
    if (!aligned(x, 16)) return MOSAIC_E_MISALIGNED;
  if (!aligned(gates, 4) || !aligned(dgates, 4) || !aligned(block_idx, 4)) return MOSAIC_E_MISALIGNED;
  if (2 * (size_t)g.m * sizeof(int) + (size_t)g.m * g.topk / 8 + 8 > 200 * 1024) return MOSAIC_E_UNSUPPORTED;  // transposed-pattern kernel
  const BwdBranchWs w = bwd_branch_layout(g);
  if ((rc = begin(p, ws, ws_bytes, w.b.total, cuda_stream, &c, false))) return rc;
  char* base = (char*)ws;
  auto F = [&](size_t off) { return (float*)(base + off); };
  float *pq = F(w.f.pq), *pk = F(w.f.pk), *pv = F(w.f.pv), *ocg = F(w.f.ocg);
  // the forward again: pooled sums (and the gated block sums of dO), block-level attention with its log-sum-exp, and of the
  // attention branches the gate gradients and row statistics
  PoolArgs pool = branch_pool(g, q, k, v, pq, pk, pv);
  pool.job[pool.n++] = {d_o, F(w.dob), nullptr, gates, g.U};
  if ((rc = launch_pool(c, pool))) return rc;
  if ((rc = launch_compress(c, pq, pk, pv, ocg, F(w.lse_cg)))) return rc;
  FwdOut out = {};
  out.gates = gates;
  out.ocg = ocg;
  out.d_o = (const __nv_bfloat16*)d_o;
  out.dgates = dgates;
  out.neg_lse2 = F(w.b.neg_lse2);
  out.neg_d = F(w.b.neg_d);
  out.gate = F(w.b.gate);
  out.gated_do = base + w.b.gated_do;
  if ((rc = launch_fwd_tc(c, kFwdStats, q, k, v, block_idx, out, c.status + 1))) return rc;
  // compression branch on the block level
  const CompressBwd cb = {pq, pk, pv, F(w.dob), ocg, F(w.lse_cg), F(w.dqm), F(w.dkm), F(w.dvm)};
  if ((rc = launch_compress_bwd(c, cb))) return rc;
  // both attention branches in one pass, with the block level's share added in the epilogues
  RowStats st = {};
  st.neg_lse2 = out.neg_lse2;
  st.neg_d = out.neg_d;
  st.gate = out.gate;
  st.gated_do = out.gated_do;
  st.dqm = F(w.dqm);
  st.dkm = F(w.dkm);
  st.dvm = F(w.dvm);
  return launch_bwd(c, q, k, v, st, d_o, block_idx, dq, dk, dv, (int32_t*)(base + w.b.off), (int32_t*)(base + w.b.q),
                    (int32_t*)(base + w.b.order), c.status + 2);
}

int mosaic_bsa_rope(const mosaic_bsa_params* p, const void* q, const void* k, const float* pos, float theta, void* q_out,
                    void* k_out, void* cuda_stream) {
  HostCtx c;
  int rc = validate(p, &c.g);
  if (rc) return rc;
  if (!q || !k || !pos || !q_out || !k_out || !(theta > 0.f)) return MOSAIC_E_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k, 16) || !aligned(q_out, 16) || !aligned(k_out, 16) || !aligned(pos, 4))
    return MOSAIC_E_MISALIGNED;
  if ((rc = device_ok())) return rc;
  c.stream = (cudaStream_t)cuda_stream;
  c.status = nullptr;
  return launch_rope(c, q, k, pos, (double)theta, q_out, k_out);
}

int mosaic_bsa_last_status(const void* ws, void* cuda_stream) {
  if (!ws) return MOSAIC_E_INVALID_ARG;
  if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) return MOSAIC_E_CUDA;
  int st = 0;
  if (cudaMemcpy(&st, ws, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return MOSAIC_E_CUDA;
  return st;
}

const char* mosaic_bsa_strerror(int code) {
  switch (code) {
    case MOSAIC_OK: return "ok";
    case MOSAIC_E_INVALID_ARG: return "invalid argument";
    case MOSAIC_E_UNSUPPORTED: return "unsupported shape, option or device";
    case MOSAIC_E_WORKSPACE_TOO_SMALL: return "workspace too small";
    case MOSAIC_E_MISALIGNED: return "misaligned pointer";
    case MOSAIC_E_CUDA: return "CUDA call failed";
    case MOSAIC_E_DEVICE_TIMEOUT: return "device: bounded wait ran out";
    case MOSAIC_E_DEVICE_BAD_INDEX: return "device: block id out of range, inside the local set, or repeated in its row";
    default: return "unknown code";
  }
}

}  // extern "C"

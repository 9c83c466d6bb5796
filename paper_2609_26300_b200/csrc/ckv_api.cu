// Host side of the C ABI declared in include/compkv.h: validation, buffer partitioning, launches.
#include <math.h>
#include <new>
#include <string.h>

#include <algorithm>

#include "ckv_internal.cuh"
#include "ckv_pipe.cuh"

namespace {

thread_local int g_last_cuda_error = 0;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

int check_layout(const ckv_layout *L) {
  if (L == nullptr) return CKV_ERR_INVALID_ARG;
  if (L->head_dim != CKV_D || L->page_size != CKV_PAGE) return CKV_ERR_BAD_LAYOUT;
  if (L->num_kv_heads <= 0 || L->num_q_heads <= 0 || L->num_q_heads % L->num_kv_heads != 0) return CKV_ERR_BAD_LAYOUT;
  const int G = L->num_q_heads / L->num_kv_heads;
  if (G != 1 && G != 2 && G != 4 && G != 8) return CKV_ERR_BAD_LAYOUT;
  if (L->block_size != 16 && L->block_size != 32 && L->block_size != 64) return CKV_ERR_BAD_LAYOUT;
  if (!is_pow2(L->var_groups) || !(L->var_groups <= CKV_D / 2 || L->var_groups == CKV_D)) return CKV_ERR_BAD_LAYOUT;
  if (L->group_layout != 0 && L->group_layout != 1) return CKV_ERR_BAD_LAYOUT;
  if (L->kv_dtype != CKV_BF16 && L->kv_dtype != CKV_F32) return CKV_ERR_BAD_LAYOUT;
  if (L->max_batch <= 0 || L->max_blocks_per_seq <= 0 || L->num_pages <= 0) return CKV_ERR_BAD_LAYOUT;
  if ((long long)L->max_blocks_per_seq * L->block_size > (1ll << 30)) return CKV_ERR_BAD_LAYOUT;
  if ((long long)L->max_batch * L->num_kv_heads > 65535) return CKV_ERR_BAD_LAYOUT;   // grid.y
  if (L->sink_blocks < 0 || L->recent_blocks < 0) return CKV_ERR_BAD_LAYOUT;
  if (!(L->sm_scale >= 0.f) || !isfinite(L->sm_scale)) return CKV_ERR_BAD_LAYOUT;
  if (L->variant & ~(CKV_VARIANT_FIRST_ORDER_MASS | CKV_VARIANT_RANK_BY_MASS | CKV_VARIANT_DROP)) return CKV_ERR_BAD_LAYOUT;
  if (L->stat_bf16 != 0 && L->stat_bf16 != 1) return CKV_ERR_BAD_LAYOUT;
  // the kernels divide the count of a step's scan tiles (32 blocks each) with a float reciprocal that is exact below
  // 2^24 (those many tiles would be half a terabyte of summaries), and unit indices by a multiplication
  if ((long long)L->max_batch * L->num_kv_heads * ((L->max_blocks_per_seq + CKV_SCAN_TILE - 1) / CKV_SCAN_TILE) >= (1ll << 24))
    return CKV_ERR_BAD_LAYOUT;
  if ((long long)L->max_batch * L->num_kv_heads * L->num_kv_heads >= (1ll << 32)) return CKV_ERR_BAD_LAYOUT;
  if (L->stat_bf16 == 1 && (L->kv_dtype != CKV_BF16 || L->var_groups == CKV_D)) return CKV_ERR_BAD_LAYOUT;
  return CKV_OK;
}

struct Regions {
  size_t kmean, dbar, vmean, stats_total;
  size_t ls, lz, scores, comp, attn, status, done, stage_q, stage_knew, stage_vnew, stage_out, stage_ids, stage_cnt, work_total;
};

Regions regions(const ckv_layout *L) {
  Regions R;
  const size_t units = (size_t)L->max_batch * L->num_kv_heads;
  const size_t rows = units * L->max_blocks_per_seq;
  const int G = L->num_q_heads / L->num_kv_heads;
  const size_t esz = L->kv_dtype == CKV_BF16 ? 2 : 4;
  size_t o = 0;
  const size_t mean_row = L->stat_bf16 ? CKV_D * 2 : CKV_D * 4;   // bf16 values, or split pairs with fp32 precision
  R.kmean = o; o = align_up(o + rows * mean_row, 256);
  R.dbar = o;  o = align_up(o + rows * L->var_groups * 4, 256);
  R.vmean = o; o = align_up(o + rows * mean_row, 256);
  R.stats_total = o;
  o = 0;
  R.status = o; o = align_up(o + 256, 256);
  R.done = o;   o = align_up(o + units * 4, 256);
  R.ls = o;     o = align_up(o + rows * G * sizeof(float), 256);
  R.lz = o;     o = align_up(o + rows * G * sizeof(float), 256);
  R.scores = o; o = align_up(o + rows * 4, 256);
  R.comp = o;   o = align_up(o + (2 * units + CKV_MAX_SCAN_CTAS + 1) * CKV_SCAN_WARPS * G * CKV_PART_STRIDE * 4, 256);
  R.attn = o;   o = align_up(o + units * CKV_MAX_SPLITS * G * CKV_PART_STRIDE * 4, 256);
  R.stage_q = o;    o = align_up(o + (size_t)L->max_batch * L->num_q_heads * CKV_D * esz, 256);
  R.stage_knew = o; o = align_up(o + units * CKV_D * esz, 256);
  R.stage_vnew = o; o = align_up(o + units * CKV_D * esz, 256);
  R.stage_out = o;  o = align_up(o + (size_t)L->max_batch * L->num_q_heads * CKV_D * esz, 256);
  R.stage_ids = o;  o = align_up(o + units * (size_t)L->max_blocks_per_seq * 4, 256);
  R.stage_cnt = o;  o = align_up(o + units * 4, 256);
  R.work_total = o;
  return R;
}

inline int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return CKV_ERR_CUDA;
}
#define CKV_CUDA(expr)                                \
  do {                                                \
    cudaError_t e__ = (expr);                         \
    if (e__ != cudaSuccess) return cuda_fail(e__);    \
  } while (0)

}  // namespace

int ckv_record_cuda_error(cudaError_t e) { return cuda_fail(e); }

namespace {

int check_step_args(const ckv_ctx *c, int batch, int max_len) {
  if (c == nullptr) return CKV_ERR_INVALID_ARG;
  if (batch <= 0 || batch > c->layout.max_batch) return CKV_ERR_INVALID_ARG;
  if (max_len <= 0 || (long long)max_len > (long long)c->layout.max_blocks_per_seq * c->layout.block_size)
    return CKV_ERR_INVALID_ARG;
  return CKV_OK;
}

}  // namespace

extern "C" {

int ckv_version(void) { return 100; }

const char *ckv_strerror(int status) {
  switch (status) {
    case CKV_OK: return "ok";
    case CKV_ERR_INVALID_ARG: return "invalid argument";
    case CKV_ERR_BAD_LAYOUT: return "unsupported layout";
    case CKV_ERR_BUDGET_TOO_SMALL: return "budget smaller than the mandatory blocks";
    case CKV_ERR_CAPACITY: return "caller buffer too small";
    case CKV_ERR_CUDA: return "CUDA runtime error";
    case CKV_ERR_TIMEOUT: return "device-side wait timed out";
  }
  return "unknown status";
}

int ckv_last_cuda_error(void) { return g_last_cuda_error; }

int ckv_query_sizes(const ckv_layout *layout, size_t *stats_bytes, size_t *workspace_bytes) {
  const int st = check_layout(layout);
  if (st != CKV_OK) return st;
  if (stats_bytes == nullptr || workspace_bytes == nullptr) return CKV_ERR_INVALID_ARG;
  const Regions R = regions(layout);
  *stats_bytes = R.stats_total;
  *workspace_bytes = R.work_total;
  return CKV_OK;
}

int ckv_stats_offsets(const ckv_layout *layout, size_t *kmean_off, size_t *dbar_off, size_t *vmean_off) {
  const int st = check_layout(layout);
  if (st != CKV_OK) return st;
  if (kmean_off == nullptr || dbar_off == nullptr || vmean_off == nullptr) return CKV_ERR_INVALID_ARG;
  const Regions R = regions(layout);
  *kmean_off = R.kmean;
  *dbar_off = R.dbar;
  *vmean_off = R.vmean;
  return CKV_OK;
}

int ckv_create(const ckv_layout *layout, void *stats_dev, size_t stats_bytes, void *work_dev, size_t work_bytes,
               ckv_stream stream, ckv_ctx **out) {
  const int st = check_layout(layout);
  if (st != CKV_OK) return st;
  if (stats_dev == nullptr || work_dev == nullptr || out == nullptr) return CKV_ERR_INVALID_ARG;
  if (((uintptr_t)stats_dev & 255) != 0 || ((uintptr_t)work_dev & 255) != 0) return CKV_ERR_INVALID_ARG;
  const Regions R = regions(layout);
  if (stats_bytes < R.stats_total || work_bytes < R.work_total) return CKV_ERR_CAPACITY;
  ckv_ctx *c = new (std::nothrow) ckv_ctx();
  if (c == nullptr) return CKV_ERR_INVALID_ARG;
  c->layout = *layout;
  if (c->layout.sm_scale == 0.f) c->layout.sm_scale = 1.0f / sqrtf((float)layout->head_dim);
  char *sb = (char *)stats_dev, *wb = (char *)work_dev;
  CkvDev &P = c->dev;
  P.Hq = layout->num_q_heads; P.Hkv = layout->num_kv_heads; P.G = P.Hq / P.Hkv;
  P.bs = layout->block_size; P.ppb = layout->block_size / layout->page_size;
  P.r = layout->var_groups; P.glayout = layout->group_layout;
  P.max_blocks = layout->max_blocks_per_seq; P.max_pages_per_seq = P.max_blocks * P.ppb;
  P.num_pages = layout->num_pages; P.sink = layout->sink_blocks; P.recent = layout->recent_blocks;
  P.scale = c->layout.sm_scale;
  P.row_elems = layout->stat_bf16 ? CKV_D : CKV_ROW_ELEMS;
  P.variant = layout->variant;
  P.half_var = (layout->variant & CKV_VARIANT_FIRST_ORDER_MASS) ? 0.f : 0.5f;
  P.kmean = (__nv_bfloat16 *)(sb + R.kmean); P.dbar = (float *)(sb + R.dbar); P.vmean = (__nv_bfloat16 *)(sb + R.vmean);
  P.status = (int *)(wb + R.status); P.unit_done = (int *)(wb + R.done);
  P.lu = (float *)(wb + R.ls); P.lz = (float *)(wb + R.lz); P.scores = (float *)(wb + R.scores);
  P.comp_part = (float *)(wb + R.comp); P.attn_part = (float *)(wb + R.attn);
  P.spin_limit = ckv_pipe::kSpinLimit; P.debug = 0;
  // the default layout (bf16 pages, full-precision summaries, four variance groups) reads the mean values as hi halves
  P.vhi = (layout->kv_dtype == CKV_BF16 && !layout->stat_bf16 && layout->var_groups == 4) ? 1 : 0;
  P.scan_tile = (layout->stat_bf16 || P.vhi) ? CKV_SCAN_TILE_HS : CKV_SCAN_TILE;
  P.lg_bs = P.bs == 16 ? 4 : (P.bs == 32 ? 5 : 6);
  P.lg_tile = P.scan_tile == 32 ? 5 : 6;
  P.hkv_magic = (unsigned)((1ull << 32) / (unsigned)P.Hkv) + 1u;   // unused when Hkv == 1 (where it wraps)
  c->work = wb; c->work_bytes = work_bytes;
  c->stage_q = R.stage_q; c->stage_knew = R.stage_knew; c->stage_vnew = R.stage_vnew;
  c->stage_out = R.stage_out; c->stage_ids = R.stage_ids; c->stage_cnt = R.stage_cnt;
  c->launches = 0;
  cudaError_t e = ckv_configure_kernels();
  if (e == cudaSuccess) e = ckv_configure_scan(c);
  if (e == cudaSuccess) e = ckv_configure_attn(c);
  if (e == cudaSuccess) e = ckv_configure_attn_mma(c);
  if (e == cudaSuccess) e = ckv_configure_unit_step(c);
  int dev_id = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev_id);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, dev_id);
  if (e == cudaSuccess) e = cudaMemsetAsync(P.status, 0, R.ls - R.status, (cudaStream_t)stream);   // status word, split counters
  if (e != cudaSuccess) { delete c; return cuda_fail(e); }
  // one pinned word for ckv_step_host: its last kernel stores the call's number there and the host waits on the
  // word instead of on the driver (without it the call falls back to a stream synchronisation)
  void *flag = nullptr;
  if (cudaHostAlloc(&flag, 64, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) {
    c->host_flag = (volatile int *)flag;
    *c->host_flag = 0;
    void *dflag = nullptr;
    if (cudaHostGetDevicePointer(&dflag, flag, 0) == cudaSuccess) c->host_flag_dev = (int *)dflag;
    else { cudaFreeHost(flag); c->host_flag = nullptr; }
  } else {
    (void)cudaGetLastError();
  }
  *out = c;
  return CKV_OK;
}

void ckv_destroy(ckv_ctx *ctx) {
  if (ctx != nullptr && ctx->hg_exec != nullptr) cudaGraphExecDestroy((cudaGraphExec_t)ctx->hg_exec);
  if (ctx != nullptr && ctx->host_flag != nullptr) cudaFreeHost((void *)ctx->host_flag);
  delete ctx;
}

int ckv_stats_build(ckv_ctx *c, const void *k_pool, const void *v_pool, const int32_t *page_table,
                    const int32_t *seq_lens, int batch, int max_seq_len_host, ckv_stream stream) {
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!k_pool || !v_pool || !page_table || !seq_lens) return CKV_ERR_INVALID_ARG;
  CKV_CUDA(ckv_launch_stats_build(c, k_pool, v_pool, page_table, seq_lens, batch, max_seq_len_host,
                                  (cudaStream_t)stream));
  return CKV_OK;
}

int ckv_stats_export(ckv_ctx *c, int batch, float *kmean, float *dbar, float *vmean, ckv_stream stream) {
  if (c == nullptr || batch <= 0 || batch > c->layout.max_batch) return CKV_ERR_INVALID_ARG;
  if (!kmean || !dbar || !vmean) return CKV_ERR_INVALID_ARG;
  CKV_CUDA(ckv_launch_stats_export(c, batch, kmean, dbar, vmean, (cudaStream_t)stream));
  return CKV_OK;
}

int ckv_append(ckv_ctx *c, void *k_pool, void *v_pool, const int32_t *page_table, int32_t *seq_lens,
               const void *k_new, const void *v_new, int batch, ckv_stream stream) {
  if (c == nullptr || batch <= 0 || batch > c->layout.max_batch) return CKV_ERR_INVALID_ARG;
  if (!k_pool || !v_pool || !page_table || !seq_lens || !k_new || !v_new) return CKV_ERR_INVALID_ARG;
  CKV_CUDA(ckv_launch_append(c, k_pool, v_pool, page_table, seq_lens, k_new, v_new, batch, (cudaStream_t)stream));
  return CKV_OK;
}

int ckv_prefill(ckv_ctx *c, void *k_pool, void *v_pool, const int32_t *page_table, int32_t *seq_lens, const void *k_src,
                const void *v_src, const int32_t *new_lens, int src_stride_tokens, int batch, int max_new_host,
                ckv_stream stream) {
  if (c == nullptr || batch <= 0 || batch > c->layout.max_batch) return CKV_ERR_INVALID_ARG;
  if (!k_pool || !v_pool || !page_table || !seq_lens || !k_src || !v_src || !new_lens) return CKV_ERR_INVALID_ARG;
  if (src_stride_tokens <= 0 || max_new_host < 0 || max_new_host > src_stride_tokens) return CKV_ERR_INVALID_ARG;
  CKV_CUDA(ckv_launch_prefill(c, k_pool, v_pool, page_table, seq_lens, k_src, v_src, new_lens, src_stride_tokens, batch,
                              max_new_host, (cudaStream_t)stream));
  return CKV_OK;
}

namespace {

// ---- host-buffer entry point: device-visible host memory is moved by kernels, not by the copy engines ----

// The address under which the GPU can reach a host buffer, if it can (pinned or registered memory, managed
// memory; a device pointer passes through).  Pageable memory: false.
bool device_view(const void *host, void **dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, host) != cudaSuccess) { (void)cudaGetLastError(); return false; }
  if (a.type == cudaMemoryTypeUnregistered || a.devicePointer == nullptr) return false;
  *dev = a.devicePointer;
  return true;
}
constexpr size_t kHostReadBytes = 160 * 1024;   // see ckv_step_host
bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// three source ranges to three destination ranges, 16 bytes per thread and iteration (sizes are multiples of 16)
__global__ void __launch_bounds__(1024) ckv_move3_kernel(const uint4 *__restrict__ a, uint4 *__restrict__ da, int na,
                                                        const uint4 *__restrict__ b, uint4 *__restrict__ db, int nb,
                                                        const uint4 *__restrict__ c, uint4 *__restrict__ dc, int nc,
                                                        const int *__restrict__ tail_src, int *__restrict__ tail_dst,
                                                        int n_tail, int *done_flag, int *done_count) {
  const int stride = gridDim.x * blockDim.x;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < na + nb + nc; i += stride) {
    if (i < na) da[i] = a[i];
    else if (i < na + nb) db[i - na] = b[i - na];
    else dc[i - na - nb] = c[i - na - nb];
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_tail; i += stride) tail_dst[i] = tail_src[i];   // 4-byte leftovers
  if (done_flag != nullptr) {   // single-CTA launches only: everything above is in host memory before the word is
    __threadfence_system();
    __syncthreads();
    // the call's number is counted on the device, so that a captured launch can be replayed
    if (threadIdx.x == 0) { const int e = *done_count + 1; *done_count = e; *(volatile int *)done_flag = e; __threadfence_system(); }
  }
}

cudaError_t ckv_launch_host_in(ckv_ctx *c, const void *hq, const void *hk, const void *hv, void *dq, void *dk, void *dv,
                               size_t q_bytes, size_t kv_bytes, cudaStream_t s) {
  const int nq = (int)(q_bytes / 16), nkv = (int)(kv_bytes / 16);
  const int grid = std::max(1, std::min((nq + 2 * nkv + 255) / 256, 64));
  ckv_move3_kernel<<<grid, 256, 0, s>>>((const uint4 *)hq, (uint4 *)dq, nq, (const uint4 *)hk, (uint4 *)dk, nkv,
                                        (const uint4 *)hv, (uint4 *)dv, nkv, nullptr, nullptr, 0, nullptr, nullptr);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t ckv_launch_host_out(ckv_ctx *c, const void *dout, const int32_t *dids, const int32_t *dcnt, void *ho, void *hi,
                                void *hc, size_t out_bytes, size_t ids_bytes, size_t cnt_bytes, int *done_flag,
                                int *done_count, cudaStream_t s) {
  // out rows are multiples of 16 bytes; the id array is moved in 16-byte pieces with a 4-byte remainder; the counts
  // (one int per unit) go as the 4-byte tail of the same launch.  One CTA: a few tens of KB, and the completion
  // word must follow every store of the launch.
  const int no = (int)(out_bytes / 16), ni = (int)(ids_bytes / 16);
  if (ids_bytes % 16 != 0)   // at most three ids
    ckv_move3_kernel<<<1, 32, 0, s>>>(nullptr, nullptr, 0, nullptr, nullptr, 0, nullptr, nullptr, 0,
                                      dids + ni * 4, (int *)hi + ni * 4, (int)((ids_bytes % 16) / 4), nullptr, nullptr);
  ckv_move3_kernel<<<1, 1024, 0, s>>>((const uint4 *)dout, (uint4 *)ho, no, (const uint4 *)dids, (uint4 *)hi, ni,
                                      nullptr, nullptr, 0, dcnt, (int *)hc, (int)(cnt_bytes / 4), done_flag, done_count);
  c->launches++;
  return cudaGetLastError();
}

// How a step is arranged: one launch, or separate ones with the last block left to the scan's tail CTAs or not.  The
// arrangements agree to rounding only, so a call decides once, from the length bound it was given.
struct Route { bool one, tail; CkvStepPlan plan; };
Route route_of(const ckv_ctx *c, int batch, int max_len, int kcap) {
  Route r = {};
  r.one = ckv_unit_step_plan(c, batch, max_len, kcap, &r.plan);
  r.tail = !r.one && ckv_scan_wants_tail(c, batch, max_len);
  return r;
}

// The launches of a sparse decode step; ev (may be null) receives 5 events bracketing them.  With `fresh` the step's new
// token is appended by its only launch, or by the scan launch (its tail CTAs do, beside the scan CTAs).  route: null, or
// what the caller has decided.
int decode_impl(ckv_ctx *c, const void *q, const void *k_pool, const void *v_pool, const int32_t *page_table,
                const int32_t *seq_lens, int batch, int max_seq_len_host, int budget_tokens, void *out, float *lse,
                int32_t *sel_ids, int32_t *sel_cnt, cudaStream_t s, cudaEvent_t *ev, const CkvNewToken *fresh = nullptr,
                const Route *route = nullptr) {
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!q || !k_pool || !v_pool || !page_table || !seq_lens || !out || !sel_ids || !sel_cnt) return CKV_ERR_INVALID_ARG;
  const ckv_layout &L = c->layout;
  const int kcap = budget_tokens / L.block_size;
  if (budget_tokens <= 0 || kcap <= 0) return CKV_ERR_BUDGET_TOO_SMALL;
  if (kcap < L.sink_blocks + L.recent_blocks && (long long)kcap * L.block_size < max_seq_len_host)
    return CKV_ERR_BUDGET_TOO_SMALL;
  Route rt;
  if (route != nullptr) rt = *route;
  else if (ev == nullptr) rt = route_of(c, batch, max_seq_len_host, kcap);
  else rt = Route{false, ckv_scan_wants_tail(c, batch, max_seq_len_host), {}};   // the profile is of the separate launches
  if (rt.one) {
    CKV_CUDA(ckv_launch_unit_step(c, rt.plan, q, k_pool, v_pool, page_table, seq_lens, fresh, batch, kcap, sel_ids, sel_cnt, out, lse, CkvHostDone{}, s));
    return CKV_OK;
  }
  int scan_grid = 0, n_splits = 0;
  c->dev.tail = rt.tail ? 1 : 0;   // one mode for the step's launches
  if (ev) CKV_CUDA(cudaEventRecord(ev[0], s));
  CKV_CUDA(ckv_launch_scan(c, q, seq_lens, batch, max_seq_len_host, fresh, &scan_grid, s));
  if (ev) CKV_CUDA(cudaEventRecord(ev[1], s));
  CKV_CUDA(ckv_launch_select(c, seq_lens, batch, kcap, scan_grid, sel_ids, sel_cnt, s));
  if (ev) CKV_CUDA(cudaEventRecord(ev[2], s));
  bool merged = false;
  CKV_CUDA(ckv_launch_attn(c, false, q, k_pool, v_pool, page_table, seq_lens, sel_ids, sel_cnt, kcap, batch,
                           max_seq_len_host, scan_grid, out, lse, &n_splits, &merged, s));
  if (ev) CKV_CUDA(cudaEventRecord(ev[3], s));
  if (!merged) CKV_CUDA(ckv_launch_merge(c, false, seq_lens, sel_cnt, n_splits, scan_grid, batch, out, lse, s));
  if (ev) CKV_CUDA(cudaEventRecord(ev[4], s));
  return CKV_OK;
}

// One step; route: null, or what the caller has decided.
int step_impl(ckv_ctx *c, const void *q, const void *k_new, const void *v_new, void *k_pool, void *v_pool,
              const int32_t *page_table, int32_t *seq_lens, int batch, int max_seq_len_host, int budget_tokens, void *out,
              float *lse, int32_t *sel_ids, int32_t *sel_cnt, cudaStream_t s, const Route *route) {
  // validate the decode half before anything is appended, so that a refused step leaves the cache untouched
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!q || !out || !sel_ids || !sel_cnt) return CKV_ERR_INVALID_ARG;
  const ckv_layout &L = c->layout;
  const int kcap = budget_tokens / L.block_size;
  if (budget_tokens <= 0 || kcap <= 0) return CKV_ERR_BUDGET_TOO_SMALL;
  if (kcap < L.sink_blocks + L.recent_blocks && (long long)kcap * L.block_size < max_seq_len_host)
    return CKV_ERR_BUDGET_TOO_SMALL;
  if (!k_pool || !v_pool || !page_table || !seq_lens || !k_new || !v_new) return CKV_ERR_INVALID_ARG;
  const Route rt = route != nullptr ? *route : route_of(c, batch, max_seq_len_host, kcap);
  CkvNewToken fresh = {k_pool, v_pool, page_table, seq_lens, k_new, v_new};
  const bool rides = rt.one || rt.tail;   // the append rides in the step's only launch, or in the scan launch (three per step)
  if (!rides) CKV_CUDA(ckv_launch_append(c, k_pool, v_pool, page_table, seq_lens, k_new, v_new, batch, s));
  return decode_impl(c, q, k_pool, v_pool, page_table, seq_lens, batch, max_seq_len_host, budget_tokens, out, lse, sel_ids,
                     sel_cnt, s, nullptr, rides ? &fresh : nullptr, &rt);
}

}  // namespace

int ckv_decode(ckv_ctx *c, const void *q, const void *k_pool, const void *v_pool, const int32_t *page_table,
               const int32_t *seq_lens, int batch, int max_seq_len_host, int budget_tokens, void *out, float *lse,
               int32_t *sel_ids, int32_t *sel_cnt, ckv_stream stream) {
  return decode_impl(c, q, k_pool, v_pool, page_table, seq_lens, batch, max_seq_len_host, budget_tokens, out, lse,
                     sel_ids, sel_cnt, (cudaStream_t)stream, nullptr);
}

int ckv_step(ckv_ctx *c, const void *q, const void *k_new, const void *v_new, void *k_pool, void *v_pool,
             const int32_t *page_table, int32_t *seq_lens, int batch, int max_seq_len_host, int budget_tokens, void *out,
             float *lse, int32_t *sel_ids, int32_t *sel_cnt, ckv_stream stream) {
  return step_impl(c, q, k_new, v_new, k_pool, v_pool, page_table, seq_lens, batch, max_seq_len_host, budget_tokens, out, lse,
                   sel_ids, sel_cnt, (cudaStream_t)stream, nullptr);
}

int ckv_decode_profile(ckv_ctx *c, const void *q, const void *k_pool, const void *v_pool, const int32_t *page_table,
                       const int32_t *seq_lens, int batch, int max_seq_len_host, int budget_tokens, void *out,
                       float *lse, int32_t *sel_ids, int32_t *sel_cnt, ckv_stream stream, float *stage_ms_host) {
  if (stage_ms_host == nullptr) return CKV_ERR_INVALID_ARG;
  cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  int rc = CKV_OK;
  for (int i = 0; i < 5 && rc == CKV_OK; ++i)
    if (cudaEventCreate(&ev[i]) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  if (rc == CKV_OK)
    rc = decode_impl(c, q, k_pool, v_pool, page_table, seq_lens, batch, max_seq_len_host, budget_tokens, out, lse,
                     sel_ids, sel_cnt, (cudaStream_t)stream, ev);
  if (rc == CKV_OK && cudaEventSynchronize(ev[4]) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  for (int i = 0; i < 4 && rc == CKV_OK; ++i)
    if (cudaEventElapsedTime(&stage_ms_host[i], ev[i], ev[i + 1]) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  for (int i = 0; i < 5; ++i)
    if (ev[i]) cudaEventDestroy(ev[i]);
  return rc;
}

int ckv_scan_profile(ckv_ctx *c, const void *q, const int32_t *seq_lens, int batch, int max_seq_len_host, int reps,
                     ckv_stream stream, float *avg_ms_host) {
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!q || !seq_lens || !avg_ms_host || reps <= 0) return CKV_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  int rc = CKV_OK;
  for (int i = 0; i < 2 && rc == CKV_OK; ++i)
    if (cudaEventCreate(&ev[i]) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  int scan_grid = 0;
  if (rc == CKV_OK && cudaEventRecord(ev[0], s) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  for (int i = 0; i < reps && rc == CKV_OK; ++i) {
    c->dev.tail = ckv_scan_wants_tail(c, batch, max_seq_len_host) ? 1 : 0;
    const cudaError_t e = ckv_launch_scan(c, q, seq_lens, batch, max_seq_len_host, nullptr, &scan_grid, s);
    if (e != cudaSuccess) rc = cuda_fail(e);
  }
  if (rc == CKV_OK && cudaEventRecord(ev[1], s) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  if (rc == CKV_OK && cudaEventSynchronize(ev[1]) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  float ms = 0.f;
  if (rc == CKV_OK && cudaEventElapsedTime(&ms, ev[0], ev[1]) != cudaSuccess) rc = cuda_fail(cudaGetLastError());
  if (rc == CKV_OK) *avg_ms_host = ms / (float)reps;
  for (int i = 0; i < 2; ++i)
    if (ev[i]) cudaEventDestroy(ev[i]);
  return rc;
}

int ckv_dense_decode(ckv_ctx *c, const void *q, const void *k_pool, const void *v_pool, const int32_t *page_table,
                     const int32_t *seq_lens, int batch, int max_seq_len_host, void *out, float *lse,
                     ckv_stream stream) {
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!q || !k_pool || !v_pool || !page_table || !seq_lens || !out) return CKV_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int n_splits = 0;
  bool merged = false;
  CKV_CUDA(ckv_launch_attn(c, true, q, k_pool, v_pool, page_table, seq_lens, nullptr, nullptr, 0, batch,
                           max_seq_len_host, 0, out, lse, &n_splits, &merged, s));
  if (!merged) CKV_CUDA(ckv_launch_merge(c, true, seq_lens, nullptr, n_splits, 0, batch, out, lse, s));
  return CKV_OK;
}

int ckv_exact_blocks(ckv_ctx *c, const void *q, const void *k_pool, const int32_t *page_table, const int32_t *seq_lens,
                     int batch, int max_seq_len_host, float *logZ, float *zmean, float *zvar, ckv_stream stream) {
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!q || !k_pool || !page_table || !seq_lens || !logZ || !zmean || !zvar) return CKV_ERR_INVALID_ARG;
  CKV_CUDA(ckv_launch_exact_blocks(c, q, k_pool, page_table, seq_lens, batch, max_seq_len_host, logZ, zmean, zvar,
                                   (cudaStream_t)stream));
  return CKV_OK;
}

int ckv_copy_scores(ckv_ctx *c, float *dst, int batch, ckv_stream stream) {
  if (c == nullptr || dst == nullptr || batch <= 0 || batch > c->layout.max_batch) return CKV_ERR_INVALID_ARG;
  const size_t bytes = (size_t)batch * c->layout.num_kv_heads * c->layout.max_blocks_per_seq * sizeof(float);
  CKV_CUDA(cudaMemcpyAsync(dst, c->dev.scores, bytes, cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
  return CKV_OK;
}

int ckv_step_host(ckv_ctx *c, const void *q_host, const void *k_new_host, const void *v_new_host, void *k_pool,
                  void *v_pool, const int32_t *page_table, int32_t *seq_lens, int batch, int max_seq_len_host,
                  int budget_tokens, void *out_host, int32_t *sel_ids_host, int32_t *sel_cnt_host,
                  ckv_stream stream) {
  const int st = check_step_args(c, batch, max_seq_len_host);
  if (st != CKV_OK) return st;
  if (!q_host || !k_new_host || !v_new_host || !out_host || !sel_ids_host || !sel_cnt_host) return CKV_ERR_INVALID_ARG;
  const ckv_layout &L = c->layout;
  const size_t esz = L.kv_dtype == CKV_BF16 ? 2 : 4;
  const size_t q_bytes = (size_t)batch * L.num_q_heads * CKV_D * esz;
  const size_t kv_bytes = (size_t)batch * L.num_kv_heads * CKV_D * esz;
  const int kcap = budget_tokens / L.block_size;
  if (kcap <= 0) return CKV_ERR_BUDGET_TOO_SMALL;
  if (kcap > L.max_blocks_per_seq) return CKV_ERR_INVALID_ARG;
  const size_t ids_bytes = (size_t)batch * L.num_kv_heads * kcap * 4;
  const size_t cnt_bytes = (size_t)batch * L.num_kv_heads * 4;
  cudaStream_t s = (cudaStream_t)stream;
  void *dq = c->work + c->stage_q, *dk = c->work + c->stage_knew, *dv = c->work + c->stage_vnew;
  void *dout = c->work + c->stage_out;
  int32_t *dids = (int32_t *)(c->work + c->stage_ids), *dcnt = (int32_t *)(c->work + c->stage_cnt);
  // Pinned (or otherwise device-visible) host buffers are read and written by two small kernels of the library,
  // one before and one after the step, instead of three copy-engine transfers each way: the six transfers cost
  // about 40 us of a 145 us call.  Pageable buffers take the copies.
  void *hq = nullptr, *hk = nullptr, *hv = nullptr, *ho = nullptr, *hi = nullptr, *hc = nullptr;
  // (asked on every call: a buffer may have been freed and its address reused by pageable memory since the last one)
  const bool direct = device_view(q_host, &hq) && device_view(k_new_host, &hk) && device_view(v_new_host, &hv) &&
                      device_view(out_host, &ho) && device_view(sel_ids_host, &hi) && device_view(sel_cnt_host, &hc) &&
                      aligned16(hq) && aligned16(hk) && aligned16(hv) && aligned16(ho) && aligned16(hi);
  const bool flagged = direct && c->host_flag != nullptr;
  int *done_count = c->dev.status + CKV_HOST_EPOCH_WORD;
  const Route rt = route_of(c, batch, max_seq_len_host, kcap);
  // the three parts of the call as launches on `on`: inputs in, the step, results out (+ completion word)
  auto enqueue = [&](cudaStream_t on, int max_len) -> int {
    if (direct) {
      CKV_CUDA(ckv_launch_host_in(c, hq, hk, hv, dq, dk, dv, q_bytes, kv_bytes, on));
    } else {
      CKV_CUDA(cudaMemcpyAsync(dq, q_host, q_bytes, cudaMemcpyHostToDevice, on));
      CKV_CUDA(cudaMemcpyAsync(dk, k_new_host, kv_bytes, cudaMemcpyHostToDevice, on));
      CKV_CUDA(cudaMemcpyAsync(dv, v_new_host, kv_bytes, cudaMemcpyHostToDevice, on));
    }
    const int r = step_impl(c, dq, dk, dv, k_pool, v_pool, page_table, seq_lens, batch, max_len, budget_tokens, dout, nullptr,
                            dids, dcnt, on, &rt);
    if (r != CKV_OK) return r;
    if (direct) {
      CKV_CUDA(ckv_launch_host_out(c, dout, dids, dcnt, ho, hi, hc, q_bytes, ids_bytes, cnt_bytes,
                                   flagged ? c->host_flag_dev : nullptr, done_count, on));
    } else {
      CKV_CUDA(cudaMemcpyAsync(out_host, dout, q_bytes, cudaMemcpyDeviceToHost, on));
      CKV_CUDA(cudaMemcpyAsync(sel_ids_host, dids, ids_bytes, cudaMemcpyDeviceToHost, on));
      CKV_CUDA(cudaMemcpyAsync(sel_cnt_host, dcnt, cnt_bytes, cudaMemcpyDeviceToHost, on));
    }
    return CKV_OK;
  };
  // wait on the word the last kernel stores (its stores to the caller's buffers precede it); if it does not show
  // up in a long while something failed: the stream synchronisation reports it
  auto wait_done = [&]() -> int {
    const int epoch = ++c->host_epoch;
    for (long long spin = 0; spin < 200000000ll; ++spin)
      if (*c->host_flag == epoch) return CKV_OK;
    CKV_CUDA(cudaStreamSynchronize(s));
    c->host_epoch = *c->host_flag;
    return CKV_OK;
  };

  // A step that is one launch reads its inputs from the pinned buffers and writes its results there itself, completion
  // word included: nothing is staged and there is one kernel to launch (a graph of copy-in, step and copy-out took 76 us
  // a call at 128K where this takes 57 to 59).  Every CTA of a unit reads the unit's queries over the bus; past kHostReadBytes
  // a kernel brings the inputs in first, in a launch of its own.  That is the documented count of launches and not a
  // crossover: read over the bus / copied first, 38.0 / 38.8 us a call (128 KB), 42.8 / 43.2 (256 KB), 47.3 / 50.6 (288 KB).
  if (flagged && rt.one) {
    const CkvStepPlan &plan = rt.plan;
    if (!k_pool || !v_pool || !page_table || !seq_lens) return CKV_ERR_INVALID_ARG;
    if (kcap < L.sink_blocks + L.recent_blocks && (long long)kcap * L.block_size < max_seq_len_host) return CKV_ERR_BUDGET_TOO_SMALL;
    const void *sq = hq, *sk = hk, *sv = hv;
    if (q_bytes * plan.cluster > kHostReadBytes) {
      CKV_CUDA(ckv_launch_host_in(c, hq, hk, hv, dq, dk, dv, q_bytes, kv_bytes, s));
      sq = dq; sk = dk; sv = dv;
    }
    const CkvNewToken fresh = {k_pool, v_pool, page_table, seq_lens, sk, sv};
    CKV_CUDA(ckv_launch_unit_step(c, plan, sq, k_pool, v_pool, page_table, seq_lens, &fresh, batch, kcap, (int *)hi, (int *)hc, ho, nullptr,
                                  CkvHostDone{c->host_flag_dev, done_count, c->dev.status + CKV_CTA_COUNTER_WORD}, s));
    return wait_done();
  }

  // A caller that comes back with the same buffers and sizes (a decode loop) gets its second call captured as a
  // CUDA graph and every later one replayed: one driver call instead of five launches.  The length bound is part
  // of the captured launches, so it is rounded up (it only has to be an upper bound) and the graph lasts 1024 steps; the
  // arrangement is the one of the bound that was given, and part of the key.
  cudaStreamCaptureStatus cap_state = cudaStreamCaptureStatusActive;
  const bool own_stream = s != nullptr && s != cudaStreamLegacy && s != cudaStreamPerThread &&
                          cudaStreamIsCapturing(s, &cap_state) == cudaSuccess && cap_state == cudaStreamCaptureStatusNone;
  if (flagged && own_stream && !c->hg_disabled) {
    const int cap_tokens = L.max_blocks_per_seq * L.block_size;
    const int len_r = std::min((max_seq_len_host + 1023) / 1024 * 1024, cap_tokens);
    const void *key[10] = {q_host, k_new_host, v_new_host, out_host, sel_ids_host, sel_cnt_host, k_pool, v_pool, page_table, seq_lens};
    const int ints[5] = {batch, len_r, budget_tokens, c->tail_mode, rt.tail ? 1 : 0};
    const bool same = c->hg_key_valid && memcmp(key, c->hg_key, sizeof(key)) == 0 && memcmp(ints, c->hg_ints, sizeof(ints)) == 0;
    if (same && c->hg_exec == nullptr) {   // second call in a row with this key: capture it
      const int64_t before = c->launches;
      cudaGraph_t graph = nullptr;
      cudaGraphExec_t exec = nullptr;
      bool ok = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
      if (ok) {
        ok = enqueue(s, len_r) == CKV_OK;
        ok = (cudaStreamEndCapture(s, &graph) == cudaSuccess) && ok && graph != nullptr;
      }
      if (ok) ok = cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
      if (graph != nullptr) cudaGraphDestroy(graph);
      c->hg_launches = (int)(c->launches - before);
      c->launches = before;
      if (ok) c->hg_exec = exec;
      else { (void)cudaGetLastError(); c->hg_disabled = true; }
    }
    if (same && c->hg_exec != nullptr) {
      CKV_CUDA(cudaGraphLaunch((cudaGraphExec_t)c->hg_exec, s));
      c->launches += c->hg_launches;
      return wait_done();
    }
    if (!same) {   // a new key: remember it, drop the graph of the old one
      if (c->hg_exec != nullptr) { cudaGraphExecDestroy((cudaGraphExec_t)c->hg_exec); c->hg_exec = nullptr; }
      memcpy(c->hg_key, key, sizeof(key));
      memcpy(c->hg_ints, ints, sizeof(ints));
      c->hg_key_valid = true;
    }
  }
  const int r = enqueue(s, max_seq_len_host);
  if (r != CKV_OK) return r;
  if (flagged) return wait_done();
  CKV_CUDA(cudaStreamSynchronize(s));
  return CKV_OK;
}

int ckv_read_status(ckv_ctx *c, int32_t *host_status, ckv_stream stream) {
  if (c == nullptr || host_status == nullptr) return CKV_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  CKV_CUDA(cudaMemcpyAsync(host_status, c->dev.status, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CKV_CUDA(cudaMemsetAsync(c->dev.status, 0, sizeof(int32_t), s));
  CKV_CUDA(cudaStreamSynchronize(s));
  return CKV_OK;
}

int64_t ckv_launch_count(const ckv_ctx *c) { return c == nullptr ? 0 : c->launches; }

int ckv_debug_set(ckv_ctx *c, uint32_t spin_limit, int flags) {
  if (c == nullptr || (flags & ~CKV_DEBUG_SKIP_FILL) != 0) return CKV_ERR_INVALID_ARG;
  c->dev.spin_limit = spin_limit == 0 ? ckv_pipe::kSpinLimit : spin_limit;
  c->dev.debug = flags;
  return CKV_OK;
}

int ckv_set_tail_mode(ckv_ctx *c, int mode) {
  if (c == nullptr || mode < CKV_TAIL_AUTO || mode > CKV_TAIL_ON) return CKV_ERR_INVALID_ARG;
  c->tail_mode = mode;
  return CKV_OK;
}

}  // extern "C"

// extern "C" entry points of libtreelstm_b200 (declared in include/treelstm.h): argument checks,
// parameter copies, workspace layout and the launch sequence of one forward / backward call.
#include <string.h>

#include <new>
#include <type_traits>

#include "common.cuh"

namespace tl {

WsLayout ws_layout(const treelstm* ctx, int n, bool with_backward) {
  WsLayout L{};
  const size_t nn = n < 1 ? 1 : (size_t)n;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += round_up_sz(bytes, 256); return o; };
  L.status = take(sizeof(DevStatus));
  L.parent = take(4 * nn);
  L.pending = take(4 * nn);
  L.order_tmp = take(4 * nn);
  L.level_offset = take(4 * (nn + 2));
  L.roots = take(4 * nn);
  L.table = take(4 * (size_t)kRadixBins * ((nn + kRadixChunk - 1) / kRadixChunk));
  L.slot = take(4 * nn);
  L.part_order = L.part_offset = L.part_spill = L.xin = L.ain = L.cin = off;
  if (ctx->precision == TREELSTM_BF16) {
    L.part_order = take(4 * nn);                     // node ids by (sub-forest, level, id)
    L.part_offset = take(4 * (kMaxParts + 1));
    L.part_spill = take(4 * (nn + kMaxParts + 1));   // wavefront boundaries of very deep sub-forests
    L.xin = take(2 * nn * (size_t)ctx->Ep);          // leaf embedding rows in ready order
    L.ain = take(2 * nn * 2 * (size_t)ctx->Hp);      // [h_l | h_r] of every position, bf16
    L.cin = take(4 * nn * 2 * (size_t)row_pitch(ctx->H));       // [c_l | c_r] of every position, fp32
  }
  L.walks = off;
  if (with_backward || ctx->cell == 0) L.walks = take(saved_walks_bytes(ctx, (int)nn));
  L.gates = L.dh = L.dc = L.dz = L.tok_slot = off;
  if (with_backward) {
    const size_t H = (size_t)ctx->H;
    L.gates = take(4 * nn * 5 * (size_t)row_pitch(ctx->H));
    L.dh = take(4 * nn * H);
    L.dc = take(4 * nn * H);
    L.dz = take(4 * nn * 5 * H);
    L.tok_slot = take(4 * ((size_t)ctx->vocab + 4 + ((size_t)ctx->vocab + 127) / 128));   // vocab + 1 entries in use, the scan
                                                                   // reads whole quads; then one count per 128 ids
  }
  L.img_dz = L.img_x0 = L.img_x1 = L.img_end = off;
  // forests that the tree kernels may be too slow for: operands of the backward pass split into bf16 pieces
  if (with_backward && wide_backward_bytes(ctx) > 0 && !trees_always_pay(ctx->cell, ctx->H, (int)nn, true)) {
    L.img_dz = take(image_bytes((int)nn, 5 * gate_pitch(ctx->H)));
    L.img_x0 = take(image_bytes((int)nn, ctx->E + 1));
    L.img_x1 = take(image_bytes((int)nn, 2 * ctx->H + 1));
    L.img_end = off;
  }
  L.trace = off;
#ifdef TREELSTM_TRACE
  L.trace = take(2 * sizeof(long long) * kTraceSlots * kTraceLevels);   // grid kernel | cluster kernel
#endif
  L.check = off;
#ifdef TREELSTM_CHECKED
  L.check = take(3 * 4 * nn);
#endif
  L.total = off;
  return L;
}

namespace {

int copy_params(treelstm* ctx, const float* emb, const float* W, const float* b, cudaStream_t s) {
  const size_t H = ctx->H, E = ctx->E, V = ctx->vocab;
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->emb, emb, sizeof(float) * V * E, cudaMemcpyDeviceToDevice, s));
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->W, W, sizeof(float) * (E + 2 * H) * 5 * H, cudaMemcpyDeviceToDevice, s));
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->b, b, sizeof(float) * 5 * H, cudaMemcpyDeviceToDevice, s));
  if (ctx->precision == TREELSTM_BF16) {
    int rc = pack_weights_bf16(ctx, s);
    if (rc == TREELSTM_OK) rc = pack_trees_tc(ctx, s);
    if (rc != TREELSTM_OK) return rc;
  }
  int rc = pack_trees(ctx, true, true, s);
  if (rc == TREELSTM_OK) rc = pack_wide_backward(ctx, s);
  if (rc != TREELSTM_OK) return rc;
  TL_CUDA(ctx, cudaStreamSynchronize(s));
  return TREELSTM_OK;
}

// Room for a classifier, and the images of the weights that only a backward pass reads: a context that never gets a
// classifier has none, and treelstm_update_weights keeps them up to date from then on.  One allocation (each costs a third of
// a millisecond).  The caller waits for `s`.
int ensure_backward_memory(treelstm* ctx, cudaStream_t s) {
  if (ctx->memory_bwd) return TREELSTM_OK;
  const size_t trees = tree_backward_bytes(ctx), wide = wide_backward_bytes(ctx);
  int dev = -1;
  TL_CUDA(ctx, cudaGetDevice(&dev));
  if (dev != ctx->device) {              // the classifier may be set with another device current
    TL_CUDA(ctx, cudaSetDevice(ctx->device));
    s = nullptr;
  }
  int rc = TREELSTM_OK;
  const cudaError_t e = cudaMalloc((void**)&ctx->memory_bwd, trees + wide + sizeof(float) * ((size_t)ctx->H + 1) * kMaxClasses);
  if (e != cudaSuccess) {
    ctx->cuda_error = (int)e;
    cudaGetLastError();
    ctx->memory_bwd = nullptr;
    rc = TREELSTM_ERR_CUDA;
  } else {
    ctx->trees.Wb = trees ? reinterpret_cast<float*>(ctx->memory_bwd) : nullptr;
    ctx->wsp = wide ? ctx->memory_bwd + trees : nullptr;
    ctx->Wc = reinterpret_cast<float*>(ctx->memory_bwd + trees + wide);
    rc = pack_trees(ctx, false, true, s);
    if (rc == TREELSTM_OK) rc = pack_wide_backward(ctx, s);
    if (rc == TREELSTM_OK && dev != ctx->device && cudaStreamSynchronize(s) != cudaSuccess) rc = TREELSTM_ERR_CUDA;
    if (rc != TREELSTM_OK) {
      cudaFree(ctx->memory_bwd);
      ctx->memory_bwd = nullptr; ctx->trees.Wb = nullptr; ctx->wsp = nullptr; ctx->Wc = nullptr;
    }
  }
  if (dev != ctx->device) TL_CUDA(ctx, cudaSetDevice(dev));
  return rc;
}

void free_host_path(treelstm* ctx) {
  auto& p = ctx->hp;
  if (p.owned) {
    cudaFree(p.forest); cudaFree(p.level); cudaFree(p.order);
    cudaFree(p.n_levels); cudaFree(p.roots_pack); cudaFree(p.n_roots); cudaFree(p.h); cudaFree(p.c);
    cudaFree(p.ws);
  }
  unsigned char* ext = p.ext;
  const size_t ext_bytes = p.ext_bytes;
  p = treelstm::HostPath{};
  p.ext = ext; p.ext_bytes = ext_bytes;
}

// Device staging of treelstm_forward_host for forests of up to `cap` nodes: offsets of its parts in
// one buffer (every part 256-byte aligned) and the total.
struct HostStaging {
  size_t forest, level, order, n_levels, roots_pack, n_roots, h, c, ws, ws_bytes, total;
};
HostStaging host_staging_layout(const treelstm* ctx, size_t cap) {
  HostStaging L{};
  const size_t H = ctx->H;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += round_up_sz(bytes, 256); return o; };
  L.forest = take(12 * cap);
  L.level = take(4 * cap);
  L.order = take(4 * cap);
  L.n_levels = take(256);
  L.roots_pack = take((4 + 8 * H) * cap);
  L.n_roots = take(256);
  L.h = take(4 * cap * H);
  L.c = take(4 * cap * H);
  L.ws_bytes = ws_layout(ctx, (int)cap, false).total;
  L.ws = take(L.ws_bytes);
  L.total = off;
  return L;
}

// True if the calling thread's current device is the one the context was created on.
bool on_own_device(const treelstm* ctx) {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess && dev == ctx->device;
}

// Read the control block and the level table back (one synchronisation).
int read_levels(treelstm* ctx) {
  auto& L = ctx->last;
  char* base = static_cast<char*>(L.ws);
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->host_status, base + L.lay.status, sizeof(DevStatus),
                               cudaMemcpyDeviceToHost, L.stream));
  // the level table is at most (n + 1) / 2 + 1 entries; small forests are copied whole, large
  // ones after the count is known
  const int quick = 4096;
  int cap_needed = L.n + 2 < quick ? L.n + 2 : quick;
  if (ctx->host_level_cap < cap_needed || !ctx->host_level_offset) {
    if (ctx->host_level_offset) cudaFreeHost(ctx->host_level_offset);
    ctx->host_level_offset = nullptr;
    TL_CUDA(ctx, cudaMallocHost((void**)&ctx->host_level_offset, sizeof(int32_t) * cap_needed));
    ctx->host_level_cap = cap_needed;
  }
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->host_level_offset, L.level_offset, sizeof(int32_t) * cap_needed,
                               cudaMemcpyDeviceToHost, L.stream));
  TL_CUDA(ctx, cudaStreamSynchronize(L.stream));
  const DevStatus* hs = reinterpret_cast<const DevStatus*>(ctx->host_status);
  if (hs->status != 0) return hs->status;
  const int n_levels = hs->n_levels;
  if (n_levels + 1 > cap_needed) {
    cudaFreeHost(ctx->host_level_offset);
    ctx->host_level_offset = nullptr;
    TL_CUDA(ctx, cudaMallocHost((void**)&ctx->host_level_offset, sizeof(int32_t) * (n_levels + 1)));
    ctx->host_level_cap = n_levels + 1;
    TL_CUDA(ctx, cudaMemcpyAsync(ctx->host_level_offset, L.level_offset,
                                 sizeof(int32_t) * (n_levels + 1), cudaMemcpyDeviceToHost, L.stream));
    TL_CUDA(ctx, cudaStreamSynchronize(L.stream));
  }
  L.n_levels = n_levels;
  L.host_levels_valid = true;
  return TREELSTM_OK;
}

}  // namespace

// What the stream of the last call, which the caller has waited for, left behind: the status, and a hint about the hand-over to
// the cluster kernel.
int settle(treelstm* ctx, int status, int hint) {
  auto& L = ctx->last;
  if (status != 0) L.valid = false;
  else if (hint != kTailUnknown && L.says_tail && ctx->tail_ok && ctx->precision == TREELSTM_BF16 && L.mode == TREELSTM_PERSISTENT) ctx->tail_skip = hint == kNoTail;
  return status;
}

// Waits for the stream of the last call, whose control block is then in ctx->host_status, and says what it holds.
int finish_status(treelstm* ctx) {
  TL_CUDA(ctx, cudaStreamSynchronize(ctx->last.stream));
  const DevStatus* hs = reinterpret_cast<const DevStatus*>(ctx->host_status);
  return settle(ctx, hs->status, tail_hint(hs->status, hs->n_levels, hs->tail_from));
}

// Pinned host memory of a context: a copy of the control block and, on a line of its own, the word that backward passes write.
int make_host_status(treelstm* ctx) {
  const size_t bytes = round_up_sz(sizeof(DevStatus), 256) + 256;
  TL_CUDA(ctx, cudaMallocHost((void**)&ctx->host_status, bytes));
  memset(ctx->host_status, 0, bytes);
  ctx->bwd_status = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(ctx->host_status) + bytes - 256);
  return TREELSTM_OK;
}

// Whether a kernel may write to `bytes` bytes of host memory at `ptr` (pinned, at the same address on the device): the first
// and the last of them are looked at, since a registered range may be shorter than what the caller says.  NULL: nothing to write.
bool gpu_writable(const void* ptr, size_t bytes) {
  if (!ptr || bytes == 0) return true;
  for (const char* at : {static_cast<const char*>(ptr), static_cast<const char*>(ptr) + bytes - 1}) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, at) != cudaSuccess) { cudaGetLastError(); return false; }
    if (a.type != cudaMemoryTypeHost || a.devicePointer != at) return false;
  }
  return true;
}

// used by backward.cu
int ensure_host_levels(treelstm* ctx) {
  if (ctx->last.host_levels_valid) return TREELSTM_OK;
  return read_levels(ctx);
}

}  // namespace tl

using namespace tl;

extern "C" {

int treelstm_create(treelstm_t** out, int H, int E, int vocab, const float* emb, const float* W,
                    const float* b, int precision, void* stream) {
  if (!out) return TREELSTM_ERR_INVALID_ARG;
  *out = nullptr;
  if (H <= 0 || E <= 0 || vocab <= 0 || !emb || !W || !b) return TREELSTM_ERR_INVALID_ARG;
  if (precision != TREELSTM_FP32 && precision != TREELSTM_BF16) return TREELSTM_ERR_INVALID_ARG;
  if (H > 8192 || E > 8192) return TREELSTM_ERR_UNSUPPORTED;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return TREELSTM_ERR_NO_DEVICE;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return TREELSTM_ERR_NO_DEVICE;
  if (prop.major != 10) return TREELSTM_ERR_NO_DEVICE;  // kernels are built for sm_100a only
  treelstm* ctx = new (std::nothrow) treelstm();
  if (!ctx) return TREELSTM_ERR_INVALID_ARG;
  ctx->H = H; ctx->E = E; ctx->vocab = vocab; ctx->precision = precision;
  ctx->Hp = round_up(H, kKBlock);
  ctx->Ep = round_up(E, kKBlock);
  ctx->device = dev;
  ctx->sm_count = prop.multiProcessorCount;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t Hs = H, Es = E, V = vocab;
  auto fail = [&](int rc) { treelstm_destroy(ctx); return rc; };
  const size_t Hp = ctx->Hp, Ep = ctx->Ep, groups = Hp / kUnitGroup;
  const size_t trees = plan_trees(ctx);
  // one allocation (a call costs about a millisecond for every couple of megabytes it maps)
  for (int pass = 0; pass < 2; ++pass) {
    size_t off = 0;
    auto take = [&](auto& ptr, size_t bytes) {
      if (pass) ptr = reinterpret_cast<std::remove_reference_t<decltype(ptr)>>(ctx->memory + off);
      off += round_up_sz(bytes, 256);
    };
    unsigned char* images = nullptr;
    take(ctx->emb, sizeof(float) * V * Es);
    take(ctx->W, sizeof(float) * (Es + 2 * Hs) * 5 * Hs);
    take(ctx->b, sizeof(float) * 5 * Hs);
    if (precision == TREELSTM_BF16) {
      take(ctx->emb_bf, 2 * V * Ep);
      take(ctx->Wp_h, 2 * groups * 40 * 2 * Hp);
      take(ctx->Wp_x, 2 * groups * 24 * Ep);
      take(ctx->Wp_t, trees_tc_bytes(ctx));
      take(ctx->bp_h, 4 * groups * 40);
      take(ctx->bp_x, 4 * groups * 24);
    }
    take(images, trees);
    if (!pass && (cudaMalloc((void**)&ctx->memory, off) != cudaSuccess || make_host_status(ctx) != TREELSTM_OK))
      return fail(TREELSTM_ERR_CUDA);
    if (pass && init_trees(ctx, images, s) != TREELSTM_OK) return fail(TREELSTM_ERR_CUDA);
  }
  int rc = init_schedule_attributes(ctx);
  if (rc == TREELSTM_OK && precision == TREELSTM_BF16) rc = init_tc_attributes(ctx);
  if (rc == TREELSTM_OK) rc = init_dweight_tc_attributes(ctx);
  if (rc != TREELSTM_OK) return fail(rc);
  rc = copy_params(ctx, emb, W, b, s);
  if (rc != TREELSTM_OK) return fail(rc);
  ctx->sf = subforest_plan(ctx);
  ctx->tail_ok = ctx->sf.ok && init_tail_attributes(ctx) == TREELSTM_OK;
  init_trees_tc(ctx);
  *out = ctx;
  return TREELSTM_OK;
}

int treelstm_create_recursive(treelstm_t** out, int cell, int H, int vocab, const float* emb, const float* W,
                              const float* b, const float* V, void* stream) {
  if (!out) return TREELSTM_ERR_INVALID_ARG;
  *out = nullptr;
  if (cell != TREELSTM_CELL_TREERNN && cell != TREELSTM_CELL_RNTN) return TREELSTM_ERR_INVALID_ARG;
  if (H <= 0 || vocab <= 0 || !emb || !W || !b || (cell == TREELSTM_CELL_RNTN && !V)) return TREELSTM_ERR_INVALID_ARG;
  if (H > 4096 || (cell == TREELSTM_CELL_RNTN && H > 128)) return TREELSTM_ERR_UNSUPPORTED;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return TREELSTM_ERR_NO_DEVICE;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return TREELSTM_ERR_NO_DEVICE;
  if (prop.major != 10) return TREELSTM_ERR_NO_DEVICE;
  treelstm* ctx = new (std::nothrow) treelstm();
  if (!ctx) return TREELSTM_ERR_INVALID_ARG;
  ctx->H = H; ctx->E = H; ctx->vocab = vocab; ctx->precision = TREELSTM_FP32; ctx->cell = cell;
  ctx->Hp = round_up(H, kKBlock); ctx->Ep = ctx->Hp;
  ctx->device = dev;
  ctx->sm_count = prop.multiProcessorCount;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t Hs = H, V_ = vocab, K2 = 2 * Hs, KQ = cell == TREELSTM_CELL_RNTN ? K2 * K2 : 0;
  auto fail = [&](int rc) { treelstm_destroy(ctx); return rc; };
  const size_t trees = plan_trees(ctx), emb_bytes = round_up_sz(sizeof(float) * V_ * Hs, 256),
               w_bytes = round_up_sz(sizeof(float) * (KQ + K2) * Hs, 256), b_bytes = round_up_sz(sizeof(float) * Hs, 256);
  if (cudaMalloc((void**)&ctx->memory, emb_bytes + w_bytes + b_bytes + trees) != cudaSuccess || make_host_status(ctx) != TREELSTM_OK)
    return fail(TREELSTM_ERR_CUDA);
  ctx->emb = reinterpret_cast<float*>(ctx->memory);
  ctx->Wcat = reinterpret_cast<float*>(ctx->memory + emb_bytes);
  ctx->b = reinterpret_cast<float*>(ctx->memory + emb_bytes + w_bytes);
  if (init_trees(ctx, ctx->memory + emb_bytes + w_bytes + b_bytes, s) != TREELSTM_OK) return fail(TREELSTM_ERR_CUDA);
  int rc = init_schedule_attributes(ctx);
  if (rc != TREELSTM_OK) return fail(rc);
  if (cudaMemcpyAsync(ctx->emb, emb, sizeof(float) * V_ * Hs, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(ctx->b, b, sizeof(float) * Hs, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return fail(TREELSTM_ERR_CUDA);
  rc = pack_weights_rec(ctx, W, V, s);
  if (rc == TREELSTM_OK) rc = pack_trees(ctx, true, false, s);
  if (rc != TREELSTM_OK) return fail(rc);
  if (cudaStreamSynchronize(s) != cudaSuccess) return fail(TREELSTM_ERR_CUDA);
  *out = ctx;
  return TREELSTM_OK;
}

int treelstm_update_weights(treelstm_t* ctx, const float* emb, const float* W, const float* b,
                            void* stream) {
  if (!ctx || !emb || !W || !b) return TREELSTM_ERR_INVALID_ARG;
  if (ctx->cell != 0) return TREELSTM_ERR_UNSUPPORTED;   // TreeRNN / RNTN contexts are created anew
  return copy_params(ctx, emb, W, b, static_cast<cudaStream_t>(stream));
}

int treelstm_set_classifier(treelstm_t* ctx, int C, const float* Wc, const float* bc, void* stream) {
  if (!ctx || !Wc || !bc || C < 1) return TREELSTM_ERR_INVALID_ARG;
  if (C > kMaxClasses) return TREELSTM_ERR_UNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (ctx->C > 0) {                      // a backward on another stream may still read the old one
    int dev = -1;
    TL_CUDA(ctx, cudaGetDevice(&dev));
    if (dev != ctx->device) TL_CUDA(ctx, cudaSetDevice(ctx->device));
    const cudaError_t e = cudaDeviceSynchronize();
    if (dev != ctx->device) TL_CUDA(ctx, cudaSetDevice(dev));
    TL_CUDA(ctx, e);
  }
  ctx->C = 0;
  const int rc = ensure_backward_memory(ctx, s);
  if (rc != TREELSTM_OK) return rc;
  ctx->bc = ctx->Wc + (size_t)ctx->H * C;
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->Wc, Wc, sizeof(float) * ctx->H * C, cudaMemcpyDeviceToDevice, s));
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->bc, bc, sizeof(float) * C, cudaMemcpyDeviceToDevice, s));
  TL_CUDA(ctx, cudaStreamSynchronize(s));
  ctx->C = C;
  return TREELSTM_OK;
}

int treelstm_set_option(treelstm_t* ctx, int key, long long value) {
  if (!ctx || value < 0) return TREELSTM_ERR_INVALID_ARG;
  switch (key) {
    case TREELSTM_OPT_SCHED_SINGLE_CTA_MAX:
      ctx->opt.sched_single_cta_max = value > kSchedSingleMaxNodes ? kSchedSingleMaxNodes : (int)value;
      return TREELSTM_OK;
    case TREELSTM_OPT_WAIT_LIMIT_CYCLES:
      if (value < 1 || value > (1ll << 24)) return TREELSTM_ERR_INVALID_ARG;
      ctx->opt.wait_limit_kcycles = value;
      return TREELSTM_OK;
    case TREELSTM_OPT_MAX_CTAS:
      ctx->opt.max_ctas = value > 65535 ? 65535 : (int)value;
      return TREELSTM_OK;
    case TREELSTM_OPT_TAIL_WIDTH:
      ctx->opt.tail_width = value > 64 ? 64 : (int)value;
      ctx->tail_skip = false;
      return TREELSTM_OK;
    case TREELSTM_OPT_TAIL_MIN_LEVELS:
      ctx->opt.tail_min_levels = value > (1 << 20) ? (1 << 20) : (int)value;
      ctx->tail_skip = false;
      return TREELSTM_OK;
    case TREELSTM_OPT_LEAVES_FIRST_MIN_NODES:
      return TREELSTM_OK;                    // (no effect any more)
    case TREELSTM_OPT_OVERLAP_LAUNCH:
      ctx->opt.overlap_launch = value != 0;
      return TREELSTM_OK;
    case TREELSTM_OPT_DW_TENSOR_CORES:
      ctx->opt.dw_tensor_cores = value != 0;
      return TREELSTM_OK;
    case TREELSTM_OPT_TAIL_MAX_NODES:
      ctx->opt.tail_max_nodes = value > (1 << 30) ? (1 << 30) : (int)value;
      return TREELSTM_OK;
    case TREELSTM_OPT_TIME_WAVEFRONT_KERNEL:
      if (value && !ctx->ev_begin) {
        TL_CUDA(ctx, cudaEventCreate(&ctx->ev_begin));
        TL_CUDA(ctx, cudaEventCreate(&ctx->ev_end));
      }
      ctx->opt.time_kernel = value != 0;
      return TREELSTM_OK;
    default:
      return TREELSTM_ERR_INVALID_ARG;
  }
}

size_t treelstm_workspace_bytes(const treelstm_t* ctx, int max_nodes, int with_backward) {
  if (!ctx || max_nodes < 0) return 0;
  return ws_layout(ctx, max_nodes, with_backward != 0).total;
}

int treelstm_forward(treelstm_t* ctx, int n_nodes, const int32_t* left, const int32_t* right,
                     const int32_t* token, float* h, float* c, int32_t* level, int32_t* order,
                     int32_t* level_offset, int32_t* n_levels, int flags, void* workspace,
                     size_t workspace_bytes, void* stream) {
  if (!ctx) return TREELSTM_ERR_INVALID_ARG;
  ctx->last.valid = false;
  ctx->launches = 0;
  ctx->status_expected = 0;
  ctx->bwd_counters_clear = false;
  if (!on_own_device(ctx)) return TREELSTM_ERR_STATE;
  if (n_nodes < 0 || !n_levels || !workspace) return TREELSTM_ERR_INVALID_ARG;
  if (n_nodes > 0 && (!left || !right || !token || !h || (!c && ctx->cell == 0) || !level || !order))
    return TREELSTM_ERR_INVALID_ARG;
  if (flags & ~(TREELSTM_PERSISTENT | TREELSTM_SAVE_FOR_BACKWARD | TREELSTM_SUBFORESTS)) return TREELSTM_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return TREELSTM_ERR_INVALID_ARG;
  const bool save = (flags & TREELSTM_SAVE_FOR_BACKWARD) != 0;
  const WsLayout lay = ws_layout(ctx, n_nodes, save);
  if (workspace_bytes < lay.total) return TREELSTM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* base = static_cast<char*>(workspace);
  int32_t* lvl_off = level_offset ? level_offset : reinterpret_cast<int32_t*>(base + lay.level_offset);

  auto& L = ctx->last;
  L.n = n_nodes; L.flags = flags; L.left = left; L.right = right; L.token = token;
  L.h = h; L.c = c; L.level = level; L.order = order; L.level_offset = lvl_off;
  L.ws = workspace; L.lay = lay; L.stream = s; L.host_levels_valid = false; L.n_levels = 0; L.says_tail = true;

  // Sub-forest mode needs the cluster plan of this context and a forest the single-CTA scheduler
  // can deal out; anything else runs the grid-wide persistent kernel instead.
  const int single_max = ctx->opt.sched_single_cta_max < kSchedPartMaxNodes ? ctx->opt.sched_single_cta_max
                                                                             : kSchedPartMaxNodes;
  const bool subforests = (flags & TREELSTM_SUBFORESTS) && ctx->precision == TREELSTM_BF16 && ctx->sf.ok &&
                          n_nodes > 0 && n_nodes <= single_max;
  int rc = launch_check_clear(ctx, n_nodes, workspace, lay, s);
  if (rc != TREELSTM_OK) return rc;
  const bool asked = trees_tc_asked(ctx, n_nodes, flags);
  rc = asked
           ? launch_schedule_trees_tc(ctx, n_nodes, left, right, token, h, c, level, order, lvl_off, n_levels, save, workspace, lay, s)
           : launch_schedule(ctx, n_nodes, left, right, token, level, order, lvl_off, n_levels, workspace, lay, subforests ? ctx->sf.n_parts : 0, s);
  if (rc != TREELSTM_OK) return rc;
  const bool persistent = (flags & (TREELSTM_PERSISTENT | TREELSTM_SUBFORESTS)) != 0;
  L.mode = subforests ? TREELSTM_SUBFORESTS : (persistent ? TREELSTM_PERSISTENT : TREELSTM_PER_LEVEL);
  L.valid = true;
  ctx->bwd_counters_clear = true;                          // with the whole control block
  if (n_nodes == 0) return TREELSTM_OK;
  ctx->ev_valid = false;
  if (asked && trees_tc_always_take(ctx, n_nodes)) {
    L.says_tail = false;
    rc = launch_check_counts(ctx, n_nodes, order, left, workspace, lay, s);
    if (rc != TREELSTM_OK) L.valid = false;
    return rc;
  }

  if (!persistent) {
    rc = read_levels(ctx);
    if (rc != TREELSTM_OK) { L.valid = false; return rc; }
  }
  if (ctx->opt.time_kernel) TL_CUDA(ctx, cudaEventRecord(ctx->ev_begin, s));
  if (ctx->cell != 0)
    rc = launch_forward_rec(ctx, n_nodes, left, right, token, h, order, lvl_off, ctx->host_level_offset, L.n_levels,
                            persistent ? (flags | TREELSTM_PERSISTENT) : flags, workspace, lay, s);
  else if (subforests)
    rc = launch_forward_bf16_subforest(ctx, n_nodes, left, right, token, h, c, level, flags, workspace, lay, s);
  else if (ctx->precision == TREELSTM_BF16)
    rc = launch_forward_bf16(ctx, n_nodes, left, right, token, h, c, order, lvl_off,
                             ctx->host_level_offset, L.n_levels, persistent ? (flags | TREELSTM_PERSISTENT) : flags,
                             workspace, lay, s);
  else
    rc = launch_forward_fp32(ctx, n_nodes, left, right, token, h, c, order, lvl_off,
                             ctx->host_level_offset, L.n_levels, persistent ? (flags | TREELSTM_PERSISTENT) : flags,
                             workspace, lay, s);
  if (ctx->opt.time_kernel && rc == TREELSTM_OK) {
    TL_CUDA(ctx, cudaEventRecord(ctx->ev_end, s));
    ctx->ev_valid = true;
  }
  if (rc == TREELSTM_OK)
    rc = launch_check_counts(ctx, n_nodes, subforests ? reinterpret_cast<const int32_t*>(base + lay.part_order) : order,
                             left, workspace, lay, s);
  if (rc != TREELSTM_OK) L.valid = false;
  return rc;
}

int treelstm_last_kernel_ms(treelstm_t* ctx, float* ms) {
  if (!ctx || !ms) return TREELSTM_ERR_INVALID_ARG;
  if (!ctx->ev_valid) return TREELSTM_ERR_STATE;
  TL_CUDA(ctx, cudaEventSynchronize(ctx->ev_end));
  TL_CUDA(ctx, cudaEventElapsedTime(ms, ctx->ev_begin, ctx->ev_end));
  return TREELSTM_OK;
}

int treelstm_status_sync(treelstm_t* ctx) {
  if (!ctx) return TREELSTM_ERR_INVALID_ARG;
  auto& L = ctx->last;
  if (!L.ws) return TREELSTM_ERR_STATE;
  char* base = static_cast<char*>(L.ws);
  if (ctx->status_expected != 0 && ctx->status_stream == L.stream) {   // the last kernel of the backward pass writes it
    TL_CUDA(ctx, cudaStreamSynchronize(L.stream));
    const unsigned long long word = *const_cast<const volatile unsigned long long*>(ctx->bwd_status);
    if ((int)(word >> 32) == ctx->status_expected) return settle(ctx, -(int)(word & 0xFFFFu), (int)(word >> 16 & 0xFFFFu));
    // (a backward pass on another stream has written it since: the control block itself says it)
  }
  TL_CUDA(ctx, cudaMemcpyAsync(ctx->host_status, base + L.lay.status, sizeof(DevStatus),
                               cudaMemcpyDeviceToHost, L.stream));
  return finish_status(ctx);
}

int treelstm_roots(treelstm_t* ctx, int max_roots, int32_t* root_ids, float* root_h, float* root_c,
                   int32_t* n_roots, void* stream) {
  if (!ctx || max_roots < 0 || !n_roots) return TREELSTM_ERR_INVALID_ARG;
  if (!ctx->last.valid) return TREELSTM_ERR_STATE;
  return launch_gather_roots(ctx, max_roots, root_ids, root_h, root_c, n_roots, nullptr,
                             static_cast<cudaStream_t>(stream));
}

int treelstm_backward(treelstm_t* ctx, const int32_t* labels, float* loss, float* dW, float* db,
                      float* dWc, float* dbc, int32_t* touched_ids, float* dEmb_rows,
                      int32_t* n_touched, void* stream) {
  if (!ctx || !labels || !loss || !dW || !db || !dWc || !dbc || !touched_ids || !dEmb_rows ||
      !n_touched)
    return TREELSTM_ERR_INVALID_ARG;
  if (!ctx->last.valid || !(ctx->last.flags & TREELSTM_SAVE_FOR_BACKWARD) || ctx->C < 1)
    return TREELSTM_ERR_STATE;
  if (ctx->cell != 0) return TREELSTM_ERR_STATE;   // TreeRNN / RNTN contexts: treelstm_backward_recursive
  if (!on_own_device(ctx)) return TREELSTM_ERR_STATE;
  ctx->launches = 0;
  ctx->status_expected = 0;
  return launch_backward(ctx, labels, loss, dW, db, dWc, dbc, touched_ids, dEmb_rows, n_touched,
                         static_cast<cudaStream_t>(stream));
}

int treelstm_backward_recursive(treelstm_t* ctx, const int32_t* labels, float* loss, float* dW, float* db, float* dV,
                                float* dWc, float* dbc, int32_t* touched_ids, float* dEmb_rows,
                                int32_t* n_touched, void* stream) {
  if (!ctx || !labels || !loss || !dW || !db || !dWc || !dbc || !touched_ids || !dEmb_rows || !n_touched)
    return TREELSTM_ERR_INVALID_ARG;
  if (ctx->cell == 0) return TREELSTM_ERR_STATE;
  if (ctx->cell == TREELSTM_CELL_RNTN && !dV) return TREELSTM_ERR_INVALID_ARG;
  if (!ctx->last.valid || !(ctx->last.flags & TREELSTM_SAVE_FOR_BACKWARD) || ctx->C < 1)
    return TREELSTM_ERR_STATE;
  if (!on_own_device(ctx)) return TREELSTM_ERR_STATE;
  ctx->launches = 0;
  ctx->status_expected = 0;
  return launch_backward_rec(ctx, labels, loss, dW, db, dV, dWc, dbc, touched_ids, dEmb_rows, n_touched,
                             static_cast<cudaStream_t>(stream));
}

int treelstm_forward_host(treelstm_t* ctx, int n_nodes, const int32_t* left, const int32_t* right,
                          const int32_t* token, float* h, float* c, int32_t* level, int32_t* order,
                          int32_t* n_levels, int max_roots, int32_t* root_ids, float* root_h,
                          float* root_c, int32_t* n_roots, int flags, void* stream) {
  if (!ctx || n_nodes < 0 || max_roots < 0) return TREELSTM_ERR_INVALID_ARG;
  if (n_nodes > 0 && (!left || !right || !token)) return TREELSTM_ERR_INVALID_ARG;
  if (flags & TREELSTM_SAVE_FOR_BACKWARD) return TREELSTM_ERR_INVALID_ARG;
  if (ctx->cell != 0) c = root_c = nullptr;   // these cells have no cell state
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!on_own_device(ctx)) return TREELSTM_ERR_STATE;
  auto& p = ctx->hp;
  const size_t H = ctx->H;
  if (p.ext) {
    // the caller's staging memory: carved up anew whenever the forest outgrows the last carving
    if (n_nodes > p.cap_nodes || !p.ws || p.owned) {
      const size_t cap = n_nodes < 1 ? 1 : (size_t)n_nodes;
      const HostStaging L = host_staging_layout(ctx, cap);
      if (L.total > p.ext_bytes) return TREELSTM_ERR_INVALID_ARG;
      free_host_path(ctx);
      unsigned char* b = p.ext;
      p.forest = reinterpret_cast<int32_t*>(b + L.forest);
      p.level = reinterpret_cast<int32_t*>(b + L.level);
      p.order = reinterpret_cast<int32_t*>(b + L.order);
      p.n_levels = reinterpret_cast<int32_t*>(b + L.n_levels);
      p.roots_pack = b + L.roots_pack;
      p.n_roots = reinterpret_cast<int32_t*>(b + L.n_roots);
      p.h = reinterpret_cast<float*>(b + L.h);
      p.c = reinterpret_cast<float*>(b + L.c);
      p.ws = b + L.ws;
      p.ws_bytes = L.ws_bytes;
      p.cap_nodes = (int)cap;
      p.owned = false;
    }
  } else if (n_nodes > p.cap_nodes || !p.ws) {
    free_host_path(ctx);
    const size_t cap = n_nodes < 1024 ? 1024 : (size_t)n_nodes + n_nodes / 4;
    p.ws_bytes = ws_layout(ctx, (int)cap, false).total;
    p.owned = true;
    // the three forest arrays share one buffer, the root outputs another: when the caller's host
    // arrays are adjacent in the same way, each group moves in a single copy
    if (cudaMalloc((void**)&p.forest, 12 * cap) != cudaSuccess || cudaMalloc((void**)&p.level, 4 * cap) != cudaSuccess ||
        cudaMalloc((void**)&p.order, 4 * cap) != cudaSuccess || cudaMalloc((void**)&p.n_levels, 256) != cudaSuccess ||
        cudaMalloc((void**)&p.roots_pack, (4 + 8 * H) * cap) != cudaSuccess || cudaMalloc((void**)&p.n_roots, 256) != cudaSuccess ||
        cudaMalloc((void**)&p.h, 4 * cap * H) != cudaSuccess || cudaMalloc((void**)&p.c, 4 * cap * H) != cudaSuccess ||
        cudaMalloc(&p.ws, p.ws_bytes) != cudaSuccess) {
      ctx->cuda_error = (int)cudaGetLastError();
      free_host_path(ctx);
      return TREELSTM_ERR_CUDA;
    }
    p.cap_nodes = (int)cap;
  }
  const size_t nb = 4 * (size_t)n_nodes;
  p.left = p.forest; p.right = p.forest + n_nodes; p.token = p.forest + 2 * (size_t)n_nodes;
  if (n_nodes > 0) {
    if (right == left + n_nodes && token == right + n_nodes) {
      TL_CUDA(ctx, cudaMemcpyAsync(p.left, left, 3 * nb, cudaMemcpyHostToDevice, s));
    } else {
      TL_CUDA(ctx, cudaMemcpyAsync(p.left, left, nb, cudaMemcpyHostToDevice, s));
      TL_CUDA(ctx, cudaMemcpyAsync(p.right, right, nb, cudaMemcpyHostToDevice, s));
      TL_CUDA(ctx, cudaMemcpyAsync(p.token, token, nb, cudaMemcpyHostToDevice, s));
    }
  }
  ctx->behind_copy = true;
  int rc = treelstm_forward(ctx, n_nodes, p.left, p.right, p.token, p.h, p.c, p.level, p.order, nullptr,
                            p.n_levels, flags, p.ws, p.ws_bytes, s);
  ctx->behind_copy = false;
  if (rc != TREELSTM_OK) return rc;
  const int launches_fwd = ctx->launches;
  const bool want_roots = root_ids || root_h || root_c || n_roots;
  int max_r = max_roots < n_nodes ? max_roots : n_nodes;
  p.root_ids = reinterpret_cast<int32_t*>(p.roots_pack);
  p.root_h = reinterpret_cast<float*>(p.root_ids + max_r);
  p.root_c = p.root_h + (size_t)max_r * H;
  // Roots whose destinations are pinned are written there by the gathering kernel itself, and so is the control
  // block: two copies less behind it on the stream.
  const size_t id_bytes = 4 * (size_t)max_r, row_bytes = id_bytes * H;
  const bool one_range = root_ids && root_h == reinterpret_cast<float*>(root_ids + max_r) && root_c == root_h + (size_t)max_r * H;
  const bool direct = want_roots && max_r > 0 &&
                      (one_range ? gpu_writable(root_ids, id_bytes + 2 * row_bytes)
                                 : gpu_writable(root_ids, id_bytes) && gpu_writable(root_h, row_bytes) &&
                                       gpu_writable(root_c, row_bytes));
  if (want_roots) {
    rc = direct ? launch_gather_roots(ctx, max_r, root_ids, root_h, root_c, nullptr, ctx->host_status, s)
                : launch_gather_roots(ctx, max_r, p.root_ids, p.root_h, p.root_c, p.n_roots, nullptr, s);
    if (rc != TREELSTM_OK) return rc;
  }
  if (n_nodes > 0) {
    if (h) TL_CUDA(ctx, cudaMemcpyAsync(h, p.h, nb * H, cudaMemcpyDeviceToHost, s));
    if (c) TL_CUDA(ctx, cudaMemcpyAsync(c, p.c, nb * H, cudaMemcpyDeviceToHost, s));
    if (level) TL_CUDA(ctx, cudaMemcpyAsync(level, p.level, nb, cudaMemcpyDeviceToHost, s));
    if (order) TL_CUDA(ctx, cudaMemcpyAsync(order, p.order, nb, cudaMemcpyDeviceToHost, s));
  }
  if (want_roots && max_r > 0 && !direct) {
    // the number of roots is not known on the host yet: copy max_r rows (rows past n_roots are
    // unspecified) - callers pass the number of trees they submitted
    if (one_range && max_r == max_roots) {
      TL_CUDA(ctx, cudaMemcpyAsync(root_ids, p.root_ids, id_bytes + 2 * row_bytes, cudaMemcpyDeviceToHost, s));
    } else {
      if (root_ids) TL_CUDA(ctx, cudaMemcpyAsync(root_ids, p.root_ids, id_bytes, cudaMemcpyDeviceToHost, s));
      if (root_h) TL_CUDA(ctx, cudaMemcpyAsync(root_h, p.root_h, row_bytes, cudaMemcpyDeviceToHost, s));
      if (root_c) TL_CUDA(ctx, cudaMemcpyAsync(root_c, p.root_c, row_bytes, cudaMemcpyDeviceToHost, s));
    }
  }
  // the level and root counts come back with the control block that the status read copies anyway
  rc = direct ? finish_status(ctx) : treelstm_status_sync(ctx);
  const DevStatus* hs = reinterpret_cast<const DevStatus*>(ctx->host_status);
  const bool ok = rc == TREELSTM_OK;
  if (n_levels) *n_levels = ok ? hs->n_levels : 0;
  if (n_roots) *n_roots = ok ? (hs->n_roots < max_r ? hs->n_roots : max_r) : 0;
  ctx->launches = launches_fwd + (want_roots ? 1 : 0);
  return rc;
}

size_t treelstm_host_staging_bytes(const treelstm_t* ctx, int max_nodes) {
  if (!ctx || max_nodes < 0) return 0;
  return host_staging_layout(ctx, max_nodes < 1 ? 1 : (size_t)max_nodes).total;
}

int treelstm_set_host_staging(treelstm_t* ctx, void* device_buffer, size_t bytes) {
  if (!ctx) return TREELSTM_ERR_INVALID_ARG;
  if (device_buffer && reinterpret_cast<uintptr_t>(device_buffer) % 256 != 0) return TREELSTM_ERR_INVALID_ARG;
  free_host_path(ctx);
  ctx->hp.ext = static_cast<unsigned char*>(device_buffer);
  ctx->hp.ext_bytes = device_buffer ? bytes : 0;
  ctx->last.valid = false;
  return TREELSTM_OK;
}

int treelstm_selftest_waits(treelstm_t* ctx, void* workspace, size_t workspace_bytes, int32_t* result,
                            void* stream) {
  if (!ctx || !workspace || !result || workspace_bytes < sizeof(DevStatus)) return TREELSTM_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return TREELSTM_ERR_INVALID_ARG;
  ctx->last.valid = false;   // the control block of an earlier forward may be the one overwritten
  ctx->last.ws = nullptr;    // and its workspace is no longer this context's to read
  return launch_selftest_waits(ctx, workspace, result, static_cast<cudaStream_t>(stream));
}

#ifdef TREELSTM_TRACE
// Trace builds only (not part of the public header): copies the cycle stamps of the last forward to
// the host, kTraceSlots per wavefront; which = 0 grid-wide kernel, 1 cluster kernel.  Synchronises.
TREELSTM_API int treelstm_trace_read(treelstm_t* ctx, int which, long long* out, int max_entries) {
  if (!ctx || !out || which < 0 || which > 2 || !ctx->last.ws) return TREELSTM_ERR_INVALID_ARG;
  if (which == 2) {   // the scheduler's phase stamps: the unused words of the control block
    DevStatus hs;
    TL_CUDA(ctx, cudaStreamSynchronize(ctx->last.stream));
    TL_CUDA(ctx, cudaMemcpy(&hs, static_cast<const char*>(ctx->last.ws) + ctx->last.lay.status, sizeof(hs), cudaMemcpyDeviceToHost));
    int cnt = 0;
    for (; cnt < 16 && cnt < max_entries; ++cnt) out[cnt] = hs.pad[cnt];
    return cnt;
  }
  const int total = kTraceSlots * kTraceLevels;
  const int cnt = max_entries < total ? max_entries : total;
  const char* src = static_cast<const char*>(ctx->last.ws) + ctx->last.lay.trace + (size_t)which * total * sizeof(long long);
  TL_CUDA(ctx, cudaStreamSynchronize(ctx->last.stream));
  TL_CUDA(ctx, cudaMemcpy(out, src, sizeof(long long) * cnt, cudaMemcpyDeviceToHost));
  return cnt;
}
#endif

int treelstm_last_launch_count(const treelstm_t* ctx) { return ctx ? ctx->launches : 0; }

int treelstm_last_mode(const treelstm_t* ctx) { return ctx && ctx->last.valid ? ctx->last.mode : -1; }

int treelstm_subforest_count(const treelstm_t* ctx) { return ctx && ctx->sf.ok ? ctx->sf.n_parts : 0; }

int treelstm_last_cuda_error(const treelstm_t* ctx) { return ctx ? ctx->cuda_error : 0; }

int treelstm_destroy(treelstm_t* ctx) {
  if (!ctx) return TREELSTM_OK;
  cudaFree(ctx->memory); cudaFree(ctx->memory_bwd);
  if (ctx->host_level_offset) cudaFreeHost(ctx->host_level_offset);
  if (ctx->host_status) cudaFreeHost(ctx->host_status);
  free_host_path(ctx);
  if (ctx->ev_begin) cudaEventDestroy(ctx->ev_begin);
  if (ctx->ev_end) cudaEventDestroy(ctx->ev_end);
  delete ctx;
  return TREELSTM_OK;
}

const char* treelstm_strerror(int status) {
  switch (status) {
    case TREELSTM_OK: return "ok";
    case TREELSTM_ERR_INVALID_ARG: return "invalid argument";
    case TREELSTM_ERR_INVALID_FOREST: return "forest is not a set of disjoint binary trees";
    case TREELSTM_ERR_TOKEN_OUT_OF_RANGE: return "leaf token outside the vocabulary";
    case TREELSTM_ERR_LABEL_OUT_OF_RANGE: return "label outside the classifier's classes";
    case TREELSTM_ERR_TIMEOUT: return "a bounded device-side wait expired";
    case TREELSTM_ERR_CUDA: return "CUDA runtime error";
    case TREELSTM_ERR_NO_DEVICE: return "no sm_100 CUDA device";
    case TREELSTM_ERR_UNSUPPORTED: return "size not supported";
    case TREELSTM_ERR_STATE: return "call order violated";
    case TREELSTM_ERR_CHECK: return "checked build: index out of range or state row written a wrong number of times";
    default: return "unknown status";
  }
}

}  // extern "C"

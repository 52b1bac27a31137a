// On-device ready-set construction for a forest given as child-index arrays.
//
// Paper, Section 4.1.1: an operation with no unresolved input is ready; when an operation
// completes, the operations that waited on it and have all inputs resolved become ready.  For a
// tree node this gives wavefront ("level") 0 for leaves and 1 + max(level of children) for
// internal nodes.  Section 4.1.2: every invocation keeps a pointer to its caller -> parent[].
// The ready order reported to the caller is canonical: ascending (level, node id).
//
// Two implementations produce identical arrays:
//   * k_schedule_single and k_schedule_cluster (schedule.cuh): one CTA or one cluster, dependency words in shared memory;
//   * a multi-CTA path (dependency counters walked up from the leaves, LSD radix sort with
//     per-chunk histograms) for anything larger.
#include "schedule.cuh"

namespace tl {
namespace {

__global__ void __launch_bounds__(kSingleThreads, 1)
k_schedule_single(int n, const int* left, const int* right, const int* token,
                  int vocab, int* parent, int* level, int* order,
                  int* order_tmp, int* level_offset, int* roots, int* n_levels_out, DevStatus* st,
                  int n_parts, int* part_order, int* part_offset, int* slot, int cache_children) {
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_last(left, right, token);
  schedule_single(smem, false, n, left, right, token, vocab, parent, level, order, order_tmp, level_offset, roots, n_levels_out, st, n_parts,
                  part_order, part_offset, slot, cache_children);
}
__global__ void __launch_bounds__(kSingleThreads, 1)
k_schedule_cluster(int n, const int* left, const int* right, const int* token,
                   int vocab, int* level, int* order, int* order_tmp, int* level_offset, int* roots, int* n_levels_out,
                   DevStatus* st, int sh) {
  extern __shared__ __align__(16) unsigned char smem[];
  wait_for_last(left, right, token);
  schedule_cluster(smem, false, n, left, right, token, vocab, level, order, order_tmp, level_offset, roots, n_levels_out, st, sh);
}

// ------------------------------------------------------------------------------------------ //
// multi-CTA path
// ------------------------------------------------------------------------------------------ //
__global__ void k_sched_init(int n, const int* __restrict__ left, const int* __restrict__ right,
                             const int* __restrict__ token, int vocab, int* parent, int* level,
                             DevStatus* st) {
  // parent[] was set to -1 and pending[] to 0 by memsets enqueued before this kernel
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int l = left[k], r = right[k];
  bool leaf;
  int err = check_node(n, k, l, r, token, vocab, &leaf);
  if (err == 0 && !leaf) {
    if (atomicCAS(&parent[l], -1, k) != -1) err = TREELSTM_ERR_INVALID_FOREST;
    if (atomicCAS(&parent[r], -1, k) != -1) err = TREELSTM_ERR_INVALID_FOREST;
  }
  if (err) report(st, err);
  level[k] = (err == 0 && leaf) ? 0 : -1;
}

// Dependency counters: every leaf walks towards its root; at each caller the first child to
// arrive stops, the second one knows both children are resolved, assigns the level and goes on.
__global__ void k_sched_walkup(int n, const int* __restrict__ left, const int* __restrict__ right,
                               const int* parent, int* pending, int* level, DevStatus* st) {
  if (ld_volatile(&st->status) != 0) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n || left[k] >= 0) return;
  int cur = k, lvl = 0;
  for (int step = 0; step < n; ++step) {  // a path has fewer than n edges
    const int p = parent[cur];
    if (p < 0) break;
    __threadfence();
    if (atomicAdd(&pending[p], 1) == 0) return;  // sibling subtree still running
    __threadfence();
    const int sib = left[p] == cur ? right[p] : left[p];
    lvl = 1 + max(lvl, ld_volatile(&level[sib]));
    *(volatile int*)&level[p] = lvl;
    cur = p;
  }
  atomicMax(&st->max_level, lvl);
}

__global__ void k_sched_check(int n, const int* level, DevStatus* st) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0 && st->status == 0) st->n_levels = n > 0 ? st->max_level + 1 : 0;
  if (k < n && level[k] < 0) report(st, TREELSTM_ERR_INVALID_FOREST);  // cycle
}

// mode 0: key = digit `pass` of level; mode 1: key = has-a-caller flag.
__device__ __forceinline__ int sort_key(int mode, int pass, int item, const int* level,
                                        const int* parent) {
  return mode == 0 ? ((level[item] >> (8 * pass)) & 255) : (parent[item] >= 0 ? 1 : 0);
}

__device__ __forceinline__ int passes_needed(int n_levels) {
  int passes = 1;
  while (passes < 4 && (n_levels - 1) >> (8 * passes)) ++passes;
  return passes;
}

// Which buffer pass p reads and writes, so that the last needed pass lands in `order`.
__device__ __forceinline__ void pass_buffers(int mode, int pass, int passes, int* order,
                                             int* order_tmp, int* roots, const int** src,
                                             int** dst) {
  if (mode == 1) { *src = nullptr; *dst = roots; return; }
  *dst = ((passes - 1 - pass) & 1) ? order_tmp : order;
  *src = pass == 0 ? nullptr : (*dst == order ? order_tmp : order);
}

// One warp per CTA, chunk of kRadixChunk consecutive source items; table is [256][n_chunks].
__global__ void __launch_bounds__(32)
k_radix_hist(int n, int mode, int pass, const int* level, const int* parent, int* order,
             int* order_tmp, int* roots, int* table, int n_chunks, const DevStatus* st) {
  if (st->status != 0) return;
  const int passes = mode == 0 ? passes_needed(st->n_levels) : 1;
  if (pass >= passes) return;
  __shared__ int hist[kRadixBins];
  const int lane = threadIdx.x, chunk = blockIdx.x;
  for (int i = lane; i < kRadixBins; i += 32) hist[i] = 0;
  __syncwarp();
  const int* src; int* dst;
  pass_buffers(mode, pass, passes, order, order_tmp, roots, &src, &dst);
  const int begin = chunk * kRadixChunk, end = min(n, begin + kRadixChunk);
  for (int r = begin + lane; r < end; r += 32) {
    const int item = src ? src[r] : r;
    atomicAdd(&hist[sort_key(mode, pass, item, level, parent)], 1);
  }
  __syncwarp();
  for (int i = lane; i < kRadixBins; i += 32) table[(size_t)i * n_chunks + chunk] = hist[i];
}

// Exclusive scan of the whole table by one CTA.
__global__ void __launch_bounds__(1024)
k_radix_scan(int mode, int pass, int* table, int n_chunks, DevStatus* st) {
  if (st->status != 0) return;
  const int passes = mode == 0 ? passes_needed(st->n_levels) : 1;
  if (pass >= passes) return;
  __shared__ int warp_sum[32];
  __shared__ int carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long total = (long long)kRadixBins * n_chunks;
  if (tid == 0) carry = 0;
  __syncthreads();
  for (long long base = 0; base < total; base += 1024) {
    const long long i = base + tid;
    const int v = i < total ? table[i] : 0;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int t = __shfl_up_sync(kWarpMask, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int w = warp_sum[lane], wi = w;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        int t = __shfl_up_sync(kWarpMask, wi, d);
        if (lane >= d) wi += t;
      }
      warp_sum[lane] = wi - w;
    }
    __syncthreads();
    const int excl = carry + warp_sum[warp] + incl - v;
    if (i < total) table[i] = excl;
    if (mode == 1 && i == (long long)n_chunks) st->n_roots = excl;  // start of bin 1
    __syncthreads();
    if (tid == 1023) carry = excl + v;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(32)
k_radix_scatter(int n, int mode, int pass, const int* level, const int* parent, int* order,
                int* order_tmp, int* roots, const int* table, int n_chunks, const DevStatus* st) {
  if (st->status != 0) return;
  const int passes = mode == 0 ? passes_needed(st->n_levels) : 1;
  if (pass >= passes) return;
  __shared__ int base_of[kRadixBins];
  const int lane = threadIdx.x, chunk = blockIdx.x;
  for (int i = lane; i < kRadixBins; i += 32) base_of[i] = table[(size_t)i * n_chunks + chunk];
  __syncwarp();
  const int* src; int* dst;
  pass_buffers(mode, pass, passes, order, order_tmp, roots, &src, &dst);
  const int begin = chunk * kRadixChunk, end = min(n, begin + kRadixChunk);
  for (int r0 = begin; r0 < end; r0 += 32) {
    const int r = r0 + lane;
    const bool valid = r < end;
    const unsigned act = __ballot_sync(kWarpMask, valid);
    int item = 0, k = 0, base = 0;
    unsigned peers = 0;
    if (valid) {
      item = src ? src[r] : r;
      k = sort_key(mode, pass, item, level, parent);
      peers = __match_any_sync(act, k);
      base = base_of[k];
    }
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) base_of[k] = base + __popc(peers);
    __syncwarp();
    if (valid) dst[base + __popc(peers & lanemask_lt())] = item;
  }
}

__global__ void k_sched_offsets(int n, const int* level, const int* order, int* level_offset,
                                const DevStatus* st) {
  if (st->status != 0) return;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r == 0) level_offset[st->n_levels] = n;
  if (r >= n) return;
  const int a = level[order[r]];
  if (r == 0 || level[order[r - 1]] != a) level_offset[a] = r;
}

__global__ void k_gather_roots(int max_roots, int H, const int* roots, const float* h,
                               const float* c, int* root_ids, float* root_h, float* root_c,
                               int* n_roots_out, const DevStatus* st, int* status_out) {
  asm volatile("griddepcontrol.wait;" ::: "memory");      // (comes up while the kernel ahead ends)
  const int n_roots = st->status == 0 ? min(st->n_roots, max_roots) : 0;
  if (blockIdx.x == 0 && threadIdx.x == 0 && n_roots_out) *n_roots_out = n_roots;
  // the control block to pinned host memory (the destinations may lie there as well): no copy behind this kernel
  if (blockIdx.x == 0 && status_out && threadIdx.x < sizeof(DevStatus) / sizeof(int))
    status_out[threadIdx.x] = reinterpret_cast<const int*>(st)[threadIdx.x];
  for (int t = blockIdx.x; t < n_roots; t += gridDim.x) {
    const int node = roots[t];   // written by the scheduler from ids below n
    if (threadIdx.x == 0 && root_ids) root_ids[t] = node;
    // Half of the threads take h, the others c; 16 bytes each where every row starts on such a boundary (host memory behind PCIe:
    // the size of the pieces matters).
    const int half = (int)blockDim.x / 2, side = (int)threadIdx.x >= half, at = (int)threadIdx.x - side * half;
    float* const to = side ? root_c : root_h;
    const float* const from = side ? c : h;
    if (!to) continue;
    const size_t src = (size_t)node * H, dst = (size_t)t * H;
    if (H % 4 == 0 && ((reinterpret_cast<uintptr_t>(to) | reinterpret_cast<uintptr_t>(from)) & 15) == 0) {
      for (int j = at; j < H / 4; j += half) reinterpret_cast<float4*>(to + dst)[j] = reinterpret_cast<const float4*>(from + src)[j];
    } else {
      for (int j = at; j < H; j += half) to[dst + j] = from[src + j];
    }
  }
}

}  // namespace

int init_schedule_attributes(treelstm* ctx) {
  TL_CUDA(ctx, cudaFuncSetAttribute(k_schedule_single, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)single_smem_bytes(kSchedSingleMaxNodes, false)));
  // sixteen CTAs where the device has room for such a cluster, else the portable eight
  const int kMost = (int)cl_smem_bytes(13);              // 8192 nodes per CTA
  TL_CUDA(ctx, cudaFuncSetAttribute(k_schedule_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost));
  TL_CUDA(ctx, cudaFuncSetAttribute(k_schedule_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  for (int cs = 16; cs >= 8 && ctx->sched_cluster == 0; cs /= 2) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cs; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(cs); cfg.blockDim = dim3(kSingleThreads); cfg.dynamicSmemBytes = kMost;
    cfg.attrs = &at; cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_schedule_cluster, &cfg) == cudaSuccess && clusters > 0) ctx->sched_cluster = cs;
    else cudaGetLastError();
  }
  return TREELSTM_OK;
}

// Whether the kernel that schedules n nodes lets the next one on the stream start beside it.
bool scheduler_lets_start(const treelstm* ctx, int n) {
  return schedules_on_cluster(ctx, n) || n <= (ctx->opt.sched_single_cta_max < kSchedSingleMaxNodes ? ctx->opt.sched_single_cta_max : kSchedSingleMaxNodes);
}

// Forests scheduled by one cluster: from kClusterMinNodes nodes on (below that a single CTA is done before the CTAs of
// a cluster have met a few times), as long as a warp can keep its share in registers.  A lowered
// TREELSTM_OPT_SCHED_SINGLE_CTA_MAX asks for the multi-CTA path.
bool schedules_on_cluster(const treelstm* ctx, int n) {
  const int cs = ctx->sched_cluster;
  return cs > 0 && n >= kClusterMinNodes && ctx->opt.sched_single_cta_max >= kSchedSingleMaxNodes &&
         n <= (long long)cs * kClMaxPer;
}

int launch_schedule(treelstm* ctx, int n, const int32_t* left, const int32_t* right,
                    const int32_t* token, int32_t* level, int32_t* order, int32_t* level_offset,
                    int32_t* n_levels_out, void* ws, const WsLayout& lay, int n_parts, cudaStream_t stream) {
  char* base = static_cast<char*>(ws);
  DevStatus* st = reinterpret_cast<DevStatus*>(base + lay.status);
  int* parent = reinterpret_cast<int*>(base + lay.parent);
  int* pending = reinterpret_cast<int*>(base + lay.pending);
  int* order_tmp = reinterpret_cast<int*>(base + lay.order_tmp);
  int* roots = reinterpret_cast<int*>(base + lay.roots);
  int* table = reinterpret_cast<int*>(base + lay.table);

  const int single_max = ctx->opt.sched_single_cta_max < kSchedSingleMaxNodes
                             ? ctx->opt.sched_single_cta_max : kSchedSingleMaxNodes;
  if (n > 0 && n_parts == 0 && schedules_on_cluster(ctx, n)) {
    const int cs = ctx->sched_cluster;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1] = behind_last(ctx, stream);
    cfg.gridDim = dim3(cs); cfg.blockDim = dim3(kSingleThreads); cfg.dynamicSmemBytes = cl_smem_bytes(cl_shift(n, cs)); cfg.stream = stream;
    cfg.attrs = at; cfg.numAttrs = 2;
    TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_schedule_cluster, n, left, right, token, ctx->vocab, level, order, order_tmp,
                                    level_offset, roots, n_levels_out, st, cl_shift(n, cs)));
    ctx->launches += 1;
    return TREELSTM_OK;
  }
  if (n > 0 && n <= single_max) {
    // the kernel clears the control block itself and writes the level count to the caller
    const bool parts = n_parts > 0 && n <= kSchedPartMaxNodes;
    const bool cache = single_caches_children(n, parts);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = behind_last(ctx, stream);
    cfg.gridDim = dim3(1); cfg.blockDim = dim3(kSingleThreads); cfg.dynamicSmemBytes = single_smem_bytes(n, parts) + (cache ? (size_t)n * 4 + 16 : 0); cfg.stream = stream;
    cfg.attrs = &at; cfg.numAttrs = 1;
    TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_schedule_single, n, left, right, token, ctx->vocab, parent, level, order, order_tmp, level_offset, roots,
                                    n_levels_out, st, parts ? n_parts : 0, reinterpret_cast<int*>(base + lay.part_order),
                                    reinterpret_cast<int*>(base + lay.part_offset), reinterpret_cast<int*>(base + lay.slot), cache ? 1 : 0));
    ctx->launches += 1;
    return TREELSTM_OK;
  }

  TL_CUDA(ctx, cudaMemsetAsync(st, 0, sizeof(DevStatus), stream));
  if (n == 0) {
    TL_CUDA(ctx, cudaMemsetAsync(n_levels_out, 0, sizeof(int), stream));
    return TREELSTM_OK;
  }
  TL_CUDA(ctx, cudaMemsetAsync(parent, 0xFF, sizeof(int) * (size_t)n, stream));
  TL_CUDA(ctx, cudaMemsetAsync(pending, 0, sizeof(int) * (size_t)n, stream));
  const int tpb = 256, blocks = (n + tpb - 1) / tpb;
  k_sched_init<<<blocks, tpb, 0, stream>>>(n, left, right, token, ctx->vocab, parent, level, st);
  k_sched_walkup<<<blocks, tpb, 0, stream>>>(n, left, right, parent, pending, level, st);
  k_sched_check<<<blocks, tpb, 0, stream>>>(n, level, st);
  ctx->launches += 3;
  const int n_chunks = (n + kRadixChunk - 1) / kRadixChunk;
  // a forest of n nodes has at most (n + 1) / 2 levels; later passes switch themselves off on
  // the device once the actual level count is known
  int host_passes = 1;
  while (host_passes < 4 && (((n + 1) / 2 - 1) >> (8 * host_passes))) ++host_passes;
  for (int p = 0; p < host_passes; ++p) {
    k_radix_hist<<<n_chunks, 32, 0, stream>>>(n, 0, p, level, parent, order, order_tmp, roots, table,
                                              n_chunks, st);
    k_radix_scan<<<1, 1024, 0, stream>>>(0, p, table, n_chunks, st);
    k_radix_scatter<<<n_chunks, 32, 0, stream>>>(n, 0, p, level, parent, order, order_tmp, roots,
                                                 table, n_chunks, st);
    ctx->launches += 3;
  }
  k_sched_offsets<<<blocks, tpb, 0, stream>>>(n, level, order, level_offset, st);
  k_radix_hist<<<n_chunks, 32, 0, stream>>>(n, 1, 0, level, parent, order, order_tmp, roots, table,
                                            n_chunks, st);
  k_radix_scan<<<1, 1024, 0, stream>>>(1, 0, table, n_chunks, st);
  k_radix_scatter<<<n_chunks, 32, 0, stream>>>(n, 1, 0, level, parent, order, order_tmp, roots,
                                               table, n_chunks, st);
  ctx->launches += 4;
  TL_CUDA(ctx, cudaGetLastError());
  TL_CUDA(ctx, cudaMemcpyAsync(n_levels_out, &st->n_levels, sizeof(int), cudaMemcpyDeviceToDevice, stream));
  return TREELSTM_OK;
}

#ifdef TREELSTM_CHECKED
namespace {
// After a forward: every node's h row written once (H units), every internal position's operand rows
// (bf16 path) twice - one half per child -, no leaf position's operand row at all.
__global__ void k_check_counts(int n, int H, int bf16, const int* rows, const int* left, const int* counts,
                               DevStatus* st) {
  if (st->status != 0) return;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  bool ok = counts[k] == H;
  if (bf16 && !st->trees_fwd) {          // (clusters that take whole trees hand states over in shared memory only)
    // rows[k]: the node whose operand row sits at position k (ready order, or the order by sub-forest)
    const int want = left[chk(st, rows[k], n)] < 0 ? 0 : 2 * H;
    ok = ok && counts[n + k] == want && counts[2 * n + k] == want;
  }
  if (!ok) report(st, TREELSTM_ERR_CHECK);
}
}  // namespace
#endif

int launch_check_clear(treelstm* ctx, int n, void* ws, const WsLayout& lay, cudaStream_t stream) {
#ifdef TREELSTM_CHECKED
  if (n > 0) TL_CUDA(ctx, cudaMemsetAsync(check_counters(ws, lay), 0, sizeof(int) * 3 * (size_t)n, stream));
#else
  (void)ctx; (void)n; (void)ws; (void)lay; (void)stream;
#endif
  return TREELSTM_OK;
}

int launch_check_counts(treelstm* ctx, int n, const int32_t* rows, const int32_t* left, void* ws, const WsLayout& lay,
                        cudaStream_t stream) {
#ifdef TREELSTM_CHECKED
  if (n > 0) {
    DevStatus* st = reinterpret_cast<DevStatus*>(static_cast<char*>(ws) + lay.status);
    k_check_counts<<<(n + 255) / 256, 256, 0, stream>>>(n, ctx->H, ctx->precision == TREELSTM_BF16 ? 1 : 0,
                                                        rows, left, check_counters(ws, lay), st);
    TL_CUDA(ctx, cudaGetLastError());
  }
#else
  (void)ctx; (void)n; (void)rows; (void)left; (void)ws; (void)lay; (void)stream;
#endif
  return TREELSTM_OK;
}

int launch_gather_roots(treelstm* ctx, int max_roots, int32_t* root_ids, float* root_h,
                        float* root_c, int32_t* n_roots, int* status_out, cudaStream_t stream) {
  const auto& L = ctx->last;
  char* base = static_cast<char*>(L.ws);
  const DevStatus* st = reinterpret_cast<const DevStatus*>(base + L.lay.status);
  const int* roots = reinterpret_cast<const int*>(base + L.lay.roots);
  int blocks = max_roots < 1 ? 1 : (max_roots < 1184 ? max_roots : 1184);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(128); cfg.stream = stream;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization; at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_gather_roots, max_roots, ctx->H, (const int*)roots, (const float*)L.h, (const float*)L.c, (int*)root_ids, root_h,
                                  L.c ? root_c : nullptr, (int*)n_roots, (const DevStatus*)st, status_out));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace tl

// ------------------------------------------------------------------------------------------ //
// Scheduling without any allocation: the scratch of the single-CTA scheduler in a fixed array of
// the device image.  Layout: control block | parent | order_tmp | roots, each for
// TREELSTM_STATIC_MAX_NODES nodes.
// ------------------------------------------------------------------------------------------ //
namespace {
constexpr size_t kStaticNodes = TREELSTM_STATIC_MAX_NODES;
constexpr size_t kStaticBytes = sizeof(tl::DevStatus) + 3 * sizeof(int) * kStaticNodes;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

constexpr int kMaxDevices = 64;
unsigned char* g_static_scratch_addr[kMaxDevices] = {};   // device address per device ordinal
}  // namespace

extern "C" int treelstm_schedule_static(int n_nodes, const int32_t* left, const int32_t* right,
                                        const int32_t* token, int vocab, int32_t* level,
                                        int32_t* order, int32_t* level_offset, int32_t* n_levels,
                                        int32_t* status, void* stream) {
  using namespace tl;
  if (n_nodes < 0 || vocab <= 0 || !level_offset || !n_levels || !status) return TREELSTM_ERR_INVALID_ARG;
  if (n_nodes > 0 && (!left || !right || !token || !level || !order)) return TREELSTM_ERR_INVALID_ARG;
  if (n_nodes > TREELSTM_STATIC_MAX_NODES) return TREELSTM_ERR_UNSUPPORTED;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return TREELSTM_ERR_NO_DEVICE;
  if (!g_static_scratch_addr[dev]) {
    // In host code the array's name is only a handle for the symbol; the address the kernel can
    // use has to be asked for, once per device, with that device current.
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || !addr) return TREELSTM_ERR_CUDA;
    if (cudaFuncSetAttribute(k_schedule_single, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)single_smem_bytes(kSchedSingleMaxNodes, false)) != cudaSuccess)
      return TREELSTM_ERR_CUDA;
    g_static_scratch_addr[dev] = static_cast<unsigned char*>(addr);
  }
  unsigned char* base = g_static_scratch_addr[dev];
  DevStatus* st = reinterpret_cast<DevStatus*>(base);
  int* parent = reinterpret_cast<int*>(base + sizeof(DevStatus));
  int* order_tmp = parent + kStaticNodes;
  int* roots = order_tmp + kStaticNodes;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (n_nodes > 0) {
    // the control block keeps the previous call's status and counts; the kernel's first step is
    // to clear it, everything else in the array is rewritten before it is read
    const bool cache = single_caches_children(n_nodes, false);
    k_schedule_single<<<1, kSingleThreads, single_smem_bytes(n_nodes, false) + (cache ? (size_t)n_nodes * 4 + 16 : 0), s>>>(
        n_nodes, left, right, token, vocab, parent, level, order, order_tmp, level_offset, roots, n_levels, st,
        0, nullptr, nullptr, nullptr, cache ? 1 : 0);
    if (cudaGetLastError() != cudaSuccess) return TREELSTM_ERR_CUDA;
  } else {
    if (cudaMemsetAsync(st, 0, sizeof(DevStatus), s) != cudaSuccess ||
        cudaMemsetAsync(level_offset, 0, sizeof(int32_t), s) != cudaSuccess ||
        cudaMemsetAsync(n_levels, 0, sizeof(int32_t), s) != cudaSuccess)
      return TREELSTM_ERR_CUDA;
  }
  if (cudaMemcpyAsync(status, &st->status, sizeof(int), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return TREELSTM_ERR_CUDA;
  return TREELSTM_OK;
}

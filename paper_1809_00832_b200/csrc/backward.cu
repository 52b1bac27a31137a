// Training step: per-node softmax classifier + mean cross-entropy, then backpropagation through
// structure over the wavefronts in reverse (parents before children).
//
// Paper, Section 4.2.2: the gradient computation recurses at the same positions as the forward
// computation; Sections 4.2.1 / 5: a gradient operation needs the previous gradient and the
// forward values of its own node instance.  Here those values live in dense per-node arrays
// (gates, c, h) indexed by node id, so no lookup structure is needed and nothing can be routed
// to the wrong instance.
//
//   dh_n  = Wc (p_n - e_y)/N + [dIn from the caller]          dc_n = dc_caller*f + dh_n o (1 - tanh^2 c)
//   dz_o = dh tanh(c) o(1-o)   dz_i = dc u i(1-i)   dz_u = dc i (1-u^2)   dz_f* = dc c_* f*(1-f*)
//   dIn  = W dz  (rows [0,E): embedding row of a leaf; rows [E,E+2H): dh of the two children)
//   dW   = sum_n in_n (x) dz_n,   db = sum_n dz_n
#include "split_tc.cuh"

namespace tl {

int ensure_host_levels(treelstm* ctx);  // api.cu

namespace {

constexpr unsigned kFull = 0xffffffffu;

struct BwdParams {
  int n, H, E, C, vocab, n_leaves;
  const int *left, *right, *token, *order, *labels;
  const float *emb, *W, *Wc, *bc, *h, *c, *gates;
  float *dh, *dc, *dz;
  float *loss, *dW, *db, *dWc, *dbc, *dEmb_rows;
  int *tok_slot, *touched_ids, *n_touched;
  int *pos_left, *pos_right;   // children of the node at every ready position (one-launch backward; scheduler scratch reused)
  DevStatus* st;
  long long* trace;   // cycle stamps of the one-launch backward (trace builds), else nullptr
};

// ---- touched embedding rows: flag, scan, compact ------------------------------------------- //
__global__ void k_bwd_mark_tokens(BwdParams p) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= p.n_leaves) return;
  p.tok_slot[chk(p.st, p.token[chk(p.st, p.order[r], p.n)], p.vocab)] = 1;  // level 0 occupies order[0 .. n_leaves)
}

// Exclusive scan of the flags over the vocabulary by one CTA; flagged ids are emitted in
// ascending order and tok_slot[id] becomes the row index of id in dEmb_rows.  A warp takes a
// contiguous run of 128-id groups: lane l holds ids 4 l .. 4 l + 3 of a group (one 16-byte load,
// eight groups in flight), four ballots per group (component c of every lane) kept in shared memory
// (s_mask, mask_cap words; groups beyond that are read again), a scan over the warps' counts, then
// a second pass that only stores.
// flags of ids id .. id + 3 (id a multiple of 4), zeros beyond the vocabulary or where `take` is false.  No
// branch: the compiler can then keep the loads of a batch in flight together.  The table has three
// spare entries behind its vocab + 1, so the last quad may be read whole.
__device__ __forceinline__ int4 load_flags4(const BwdParams& p, int id, bool take) {
  const int last_quad = ((p.vocab - 1) >> 2) << 2;
  int4 v = *reinterpret_cast<const int4*>(p.tok_slot + min(id, last_quad));
  v.x = take && id < p.vocab ? v.x : 0;
  v.y = take && id + 1 < p.vocab ? v.y : 0;
  v.z = take && id + 2 < p.vocab ? v.z : 0;
  v.w = take && id + 3 < p.vocab ? v.w : 0;
  return v;
}
__device__ void scan_tokens(const BwdParams& p, unsigned int* s_mask, int mask_cap) {   // blockDim a multiple of 32
  __shared__ int warp_sum[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int n_groups = (p.vocab + 127) / 128, per = (n_groups + nw - 1) / nw;
  const int g_lo = min(n_groups, warp * per), g_hi = min(n_groups, g_lo + per);
  constexpr int kBatch = 8;
  int count = 0;
  for (int g0 = g_lo; g0 < g_hi; g0 += kBatch) {
    int4 v[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b)
      v[b] = load_flags4(p, (g0 + b) * 128 + 4 * lane, g0 + b < g_hi);
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const unsigned int m0 = __ballot_sync(kFull, v[b].x != 0), m1 = __ballot_sync(kFull, v[b].y != 0);
      const unsigned int m2 = __ballot_sync(kFull, v[b].z != 0), m3 = __ballot_sync(kFull, v[b].w != 0);
      if (g0 + b < g_hi) {
        if (4 * (g0 + b) + 3 < mask_cap && lane < 4) s_mask[4 * (g0 + b) + lane] = lane == 0 ? m0 : (lane == 1 ? m1 : (lane == 2 ? m2 : m3));
        count += __popc(m0) + __popc(m1) + __popc(m2) + __popc(m3);
      }
    }
  }
  if (lane == 0) warp_sum[warp] = count;
  TL_STAMP(tid == 0 ? p.trace : nullptr, kTraceLevels - 1, 9);    // first warp: flags read
  __syncthreads();
  TL_STAMP(tid == 0 ? p.trace : nullptr, kTraceLevels - 1, 10);   // all warps: flags read
  if (warp == 0) {
    int w = lane < nw ? warp_sum[lane] : 0, wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int t = __shfl_up_sync(kFull, wi, d);
      if (lane >= d) wi += t;
    }
    warp_sum[lane] = wi - w;
  }
  __syncthreads();
  int base = warp_sum[warp];
  const unsigned int below = (1u << lane) - 1u;
  for (int g = g_lo; g < g_hi; ++g) {
    const int id = g * 128 + 4 * lane;
    unsigned int m0, m1, m2, m3;
    if (4 * g + 3 < mask_cap) {
      const uint4 m = *reinterpret_cast<const uint4*>(s_mask + 4 * g);
      m0 = m.x; m1 = m.y; m2 = m.z; m3 = m.w;
    } else {
      const int4 v = load_flags4(p, id, true);
      m0 = __ballot_sync(kFull, v.x != 0); m1 = __ballot_sync(kFull, v.y != 0);
      m2 = __ballot_sync(kFull, v.z != 0); m3 = __ballot_sync(kFull, v.w != 0);
    }
    // ids ascend lane by lane, component by component
    const int f0 = (m0 >> lane) & 1u, f1 = (m1 >> lane) & 1u, f2 = (m2 >> lane) & 1u, f3 = (m3 >> lane) & 1u;
    const int e0 = base + __popc(m0 & below) + __popc(m1 & below) + __popc(m2 & below) + __popc(m3 & below);
    const int e1 = e0 + f0, e2 = e1 + f1, e3 = e2 + f2;
    if (id + 3 < p.vocab) {
      *reinterpret_cast<int4*>(p.tok_slot + id) = make_int4(e0, e1, e2, e3);
    } else {
      if (id < p.vocab) p.tok_slot[id] = e0;
      if (id + 1 < p.vocab) p.tok_slot[id + 1] = e1;
      if (id + 2 < p.vocab) p.tok_slot[id + 2] = e2;
    }
    if (f0) p.touched_ids[e0] = id;       // a set flag implies id < vocab: flags beyond it were read as 0
    if (f1) p.touched_ids[e1] = id + 1;
    if (f2) p.touched_ids[e2] = id + 2;
    if (f3) p.touched_ids[e3] = id + 3;
    base += __popc(m0) + __popc(m1) + __popc(m2) + __popc(m3);
  }
  if (warp == nw - 1 && lane == 0) { *p.n_touched = base; p.st->n_touched = base; }
}
// The same scan spread over the CTAs of the one-launch backward, in two steps with a grid barrier between
// them: scan_count_groups writes the number of flagged ids of every 128-id group to group_count[], then
// scan_place_groups sums the counts before a group and places its ids.  Group g belongs to warp 0 of CTA
// gridDim.x - 1 - g % gridDim.x: the high-numbered CTAs, which have no block in a narrow wavefront, so that
// the second step runs beside the first wavefronts instead of ahead of them.
__device__ __forceinline__ void scan_count_groups(const BwdParams& p, int* group_count) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x, n_groups = (p.vocab + 127) / 128;
  for (int g = (int)(gridDim.x - 1 - blockIdx.x); g < n_groups; g += (int)gridDim.x) {
    const int4 v = load_flags4(p, g * 128 + 4 * lane, true);
    const int c = __popc(__ballot_sync(kFull, v.x != 0)) + __popc(__ballot_sync(kFull, v.y != 0)) +
                  __popc(__ballot_sync(kFull, v.z != 0)) + __popc(__ballot_sync(kFull, v.w != 0));
    if (lane == 0) group_count[g] = c;
  }
}
__device__ __forceinline__ void scan_place_groups(const BwdParams& p, const int* group_count) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x, n_groups = (p.vocab + 127) / 128;
  const unsigned int below = (1u << lane) - 1u;
  for (int g = (int)(gridDim.x - 1 - blockIdx.x); g < n_groups; g += (int)gridDim.x) {
    const int id = g * 128 + 4 * lane;
    const int4 v = load_flags4(p, id, true);          // the group's flags: nobody else touches them
    int base = 0;
    for (int q = lane; q < g; q += 32) base += group_count[q];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) base += __shfl_xor_sync(kFull, base, d);
    const unsigned int m0 = __ballot_sync(kFull, v.x != 0), m1 = __ballot_sync(kFull, v.y != 0);
    const unsigned int m2 = __ballot_sync(kFull, v.z != 0), m3 = __ballot_sync(kFull, v.w != 0);
    const int f0 = (m0 >> lane) & 1u, f1 = (m1 >> lane) & 1u, f2 = (m2 >> lane) & 1u, f3 = (m3 >> lane) & 1u;
    const int e0 = base + __popc(m0 & below) + __popc(m1 & below) + __popc(m2 & below) + __popc(m3 & below);
    const int e1 = e0 + f0, e2 = e1 + f1, e3 = e2 + f2;
    if (id + 3 < p.vocab) {
      *reinterpret_cast<int4*>(p.tok_slot + id) = make_int4(e0, e1, e2, e3);
    } else {
      if (id < p.vocab) p.tok_slot[id] = e0;
      if (id + 1 < p.vocab) p.tok_slot[id + 1] = e1;
      if (id + 2 < p.vocab) p.tok_slot[id + 2] = e2;
    }
    if (f0) p.touched_ids[e0] = id;
    if (f1) p.touched_ids[e1] = id + 1;
    if (f2) p.touched_ids[e2] = id + 2;
    if (f3) p.touched_ids[e3] = id + 3;
    if (g == n_groups - 1 && lane == 0) {
      const int total = base + __popc(m0) + __popc(m1) + __popc(m2) + __popc(m3);
      *p.n_touched = total; p.st->n_touched = total;
    }
  }
}
// The same without flags in memory, behind a single grid barrier: a CTA finds the leaf tokens of its own run of groups in the
// forest itself, every owner reading all of it, and keeps them as bits in shared memory.  The flags need two grid barriers more (cleared |
// set | counted | placed).
struct OwnTokens {
  int g0, g1;                                            // groups of 128 ids
  __device__ OwnTokens(int vocab) {
    const int n_groups = (vocab + 127) / 128, per = (n_groups + (int)gridDim.x - 1) / (int)gridDim.x;
    g0 = min(n_groups, (int)(gridDim.x - 1 - blockIdx.x) * per);
    g1 = min(n_groups, g0 + per);
  }
};
__device__ __forceinline__ void own_tokens_count(const BwdParams& p, const OwnTokens& t, unsigned int* s_mask, int* group_count) {
  if (t.g0 == t.g1) return;
  const int tid = threadIdx.x, words = 4 * (t.g1 - t.g0);
  for (int w = tid; w < words; w += blockDim.x) s_mask[w] = 0u;
  __syncthreads();
  constexpr int kBatch = 8;
  for (int i0 = tid; i0 < p.n; i0 += kBatch * (int)blockDim.x) {
    int left[kBatch], token[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int i = min(i0 + b * (int)blockDim.x, p.n - 1);      // (the last node more than once: the same bit)
      left[b] = __ldg(p.left + i);
      token[b] = __ldg(p.token + i);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const unsigned int at = (unsigned int)(token[b] - 128 * t.g0);
      if (left[b] < 0 && at < 32u * (unsigned int)words) atomicOr(s_mask + (at >> 5), 1u << (at & 31u));
    }
  }
  __syncthreads();
  for (int g = t.g0 + tid; g < t.g1; g += blockDim.x) {
    const uint4 m = reinterpret_cast<const uint4*>(s_mask)[g - t.g0];
    group_count[g] = __popc(m.x) + __popc(m.y) + __popc(m.z) + __popc(m.w);
  }
}
__device__ __forceinline__ void own_tokens_place(const BwdParams& p, const OwnTokens& t, const unsigned int* s_mask, const int* group_count) {
  if (threadIdx.x >= 32 || t.g0 == t.g1) return;
  const int lane = threadIdx.x, n_groups = (p.vocab + 127) / 128;
  int base = 0;
  for (int q = lane; q < t.g0; q += 32) base += ld_volatile(group_count + q);
  base = __reduce_add_sync(kFull, base);
  for (int g = t.g0; g < t.g1; ++g) {
    const unsigned int* m = s_mask + 4 * (g - t.g0);
    const unsigned int mine = m[lane >> 3], shift = 4u * (lane & 7u);
    int e = base + __popc(mine & ((1u << shift) - 1u));  // rows before this lane's four ids
    for (int w = 0; w < lane >> 3; ++w) e += __popc(m[w]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int id = 128 * g + 4 * lane + k;
      if ((mine >> (shift + k)) & 1u) { p.tok_slot[id] = e; p.touched_ids[e] = id; ++e; }
    }
    base += __popc(m[0]) + __popc(m[1]) + __popc(m[2]) + __popc(m[3]);
  }
  if (t.g1 == n_groups && lane == 0) { *p.n_touched = base; p.st->n_touched = base; }
}
constexpr int kScanMaskWords = 8192;
__global__ void __launch_bounds__(1024) k_bwd_scan_tokens(BwdParams p) {
  __shared__ __align__(16) unsigned int s_mask[kScanMaskWords];
  scan_tokens(p, s_mask, kScanMaskWords);
}

// ---- classifier: logits, softmax, loss, dlogits, dh (classifier part), dWc, dbc -------------- //
// One warp per node: the lanes share the contraction over h (lane j takes units j, j + 32, ...),
// a butterfly sum gives every lane all logits, lane k keeps class k (C <= 32).
constexpr int kClsWarps = 8;
constexpr int kClsNodesPerCta = 8;    // one node per warp and group: the chains of dependent loads of a node are long

// Up to 256 hidden units and 8 classes (instantiations for the units per lane): a lane keeps its units' part of dWc in
// registers over all nodes of its warp.  (One shared-memory add per node, unit and class instead is an add of
// floats in a compare-and-swap loop: 70 us for 14.6 k nodes, H = 256, 5 classes.)
// Wider states take at most five classes, which is what the registers of two CTAs per SM hold.
template <int NJ, int kClsRegC>
__device__ __forceinline__ void classifier_nodes(const BwdParams& p, int warp_first, int warp_step, float* s_dWc) {
  const int lane = threadIdx.x & 31, H = p.H, C = p.C;
  const float inv_n = 1.0f / (float)p.n;
  float wc[NJ][kClsRegC], acc[NJ][kClsRegC], loss = 0.f, acc_b = 0.f;
#pragma unroll
  for (int t = 0; t < NJ; ++t)
#pragma unroll
    for (int k = 0; k < kClsRegC; ++k) {
      const int j = lane + 32 * t;
      wc[t][k] = j < H && k < C ? __ldg(p.Wc + j * C + k) : 0.f;
      acc[t][k] = 0.f;
    }
  const float my_bias = lane < C ? __ldg(p.bc + lane) : 0.f;
  float hn[NJ];
  int y = 0;
  auto fetch = [&](int node) {           // the next node's states and label, while this one is worked on
    if (node >= p.n) return;
    y = p.labels[node];
#pragma unroll
    for (int t = 0; t < NJ; ++t) hn[t] = p.h[(size_t)node * H + min(lane + 32 * t, H - 1)];
  };
  fetch(warp_first);
  for (int node = warp_first; node < p.n; node += warp_step) {
    float h[NJ];
    const int label = y;
#pragma unroll
    for (int t = 0; t < NJ; ++t) h[t] = lane + 32 * t < H ? hn[t] : 0.f;
    fetch(node + warp_step);
    float part[kClsRegC];
#pragma unroll
    for (int k = 0; k < kClsRegC; ++k) {
      part[k] = 0.f;
      if (k < C) {
#pragma unroll
        for (int t = 0; t < NJ; ++t) part[k] = fmaf(h[t], wc[t][k], part[k]);
      }
    }
    float logit = -INFINITY;
#pragma unroll
    for (int k = 0; k < kClsRegC; ++k)
      if (k < C) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) part[k] += __shfl_xor_sync(kFull, part[k], d);
        if (lane == k) logit = part[k] + my_bias;
      }
    float m = logit;
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, d));   // the classes sit in the first eight lanes
    m = __shfl_sync(kFull, m, 0);
    const float e = lane < C ? expf(logit - m) : 0.f;
    float sum = e;
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
    sum = __shfl_sync(kFull, sum, 0);
    const bool y_ok = label >= 0 && label < C;
    if (!y_ok && lane == 0) report(p.st, TREELSTM_ERR_LABEL_OUT_OF_RANGE);
    const float logit_y = __shfl_sync(kFull, logit, y_ok ? label : 0);
    if (y_ok) loss += m + logf(sum) - logit_y;
    const float dlogit = lane < C ? (e / sum - (lane == label ? 1.f : 0.f)) * inv_n : 0.f;
    acc_b += dlogit;
    float dh[NJ];
#pragma unroll
    for (int t = 0; t < NJ; ++t) dh[t] = 0.f;
#pragma unroll
    for (int k = 0; k < kClsRegC; ++k)
      if (k < C) {
        const float dk = __shfl_sync(kFull, dlogit, k);
#pragma unroll
        for (int t = 0; t < NJ; ++t) {
          dh[t] = fmaf(wc[t][k], dk, dh[t]);
          acc[t][k] = fmaf(h[t], dk, acc[t][k]);
        }
      }
#pragma unroll
    for (int t = 0; t < NJ; ++t)
      if (lane + 32 * t < H) p.dh[(size_t)node * H + lane + 32 * t] = dh[t];
  }
#pragma unroll
  for (int t = 0; t < NJ; ++t)
#pragma unroll
    for (int k = 0; k < kClsRegC; ++k)
      if (lane + 32 * t < H && k < C) atomicAdd(&s_dWc[(lane + 32 * t) * C + k], acc[t][k]);
  if (lane < C) atomicAdd(&s_dWc[H * C + lane], acc_b);
  if (lane == 0 && loss != 0.f) atomicAdd(&s_dWc[H * C + C], loss * inv_n);
}

// The CTA takes the node groups vb_first, vb_first + vb_step, ...; s_dWc [H][C] + [C] collects its partial sums.
struct AlreadyCleared { __device__ bool operator()() const { return true; } };
// (s_dWc: the CTA's sums of dWc, dbc and the loss, H C + C + 1 words.  They are added to the outputs behind `cleared`, which says whether
// to go on; the nodes' dh need not wait for that.)
template <typename Cleared>
__device__ bool classifier_groups(const BwdParams& p, int vb_first, int vb_step, float* s_dWc, Cleared cleared) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int H = p.H, C = p.C;
  for (int i = tid; i < H * C + C + 1; i += blockDim.x) s_dWc[i] = 0.f;
  __syncthreads();
#ifdef TREELSTM_TRACE
  long long* const ctrace = blockIdx.x == 1 && tid == 0 ? p.trace : nullptr;   // the first CTA with nodes to classify
#endif
  TL_STAMP(ctrace, kTraceLevels - 1, 11);
  const float inv_n = 1.0f / (float)p.n;
  const int n_groups = (p.n + kClsNodesPerCta - 1) / kClsNodesPerCta;
  if (C <= (H <= 64 ? 8 : 5) && H <= 256) {
    const int first = vb_first * kClsWarps + warp, step = vb_step * kClsWarps;
    if (H <= 64) classifier_nodes<2, 8>(p, first, step, s_dWc);
    else if (H <= 160) classifier_nodes<5, 5>(p, first, step, s_dWc);
    else classifier_nodes<8, 5>(p, first, step, s_dWc);
  } else {
  for (int vb = vb_first; vb < n_groups; vb += vb_step)
  for (int q = warp; q < kClsNodesPerCta; q += kClsWarps) {
    const int node0 = vb * kClsNodesPerCta;
    const int node = node0 + q;
    if (node >= p.n) break;
    const float* hn = p.h + (size_t)node * H;
    const int y = p.labels[node];                       // asked for now: they arrive with the first h values
    const float my_bias = lane < C ? __ldg(p.bc + lane) : 0.f;
    float logit = -INFINITY;
    for (int k = 0; k < C; ++k) {
      float part = 0.f;
      for (int j = lane; j < H; j += 32) part = fmaf(hn[j], __ldg(p.Wc + j * C + k), part);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) part += __shfl_xor_sync(kFull, part, d);
      if (lane == k) logit = part + my_bias;
    }
    float m = logit;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, d));
    float e = lane < C ? expf(logit - m) : 0.f, sum = e;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
    const bool y_ok = y >= 0 && y < C;
    if (!y_ok && lane == 0) report(p.st, TREELSTM_ERR_LABEL_OUT_OF_RANGE);
    const float lse = m + logf(sum);
    const float logit_y = __shfl_sync(kFull, logit, y_ok ? y : 0);
    if (lane == 0 && y_ok) atomicAdd(&s_dWc[H * C + C], (lse - logit_y) * inv_n);
    const float dlogit = lane < C ? (e / sum - (lane == y ? 1.f : 0.f)) * inv_n : 0.f;
    if (lane < C) atomicAdd(&s_dWc[H * C + lane], dlogit);
    for (int j0 = 0; j0 < H; j0 += 32) {
      const int j = j0 + lane;
      const float hj = j < H ? hn[j] : 0.f;
      float dhj = 0.f;
      for (int k = 0; k < C; ++k) {
        const float dk = __shfl_sync(kFull, dlogit, k);
        if (j < H) {
          dhj = fmaf(p.Wc[j * C + k], dk, dhj);
          atomicAdd(&s_dWc[j * C + k], hj * dk);
        }
      }
      if (j < H) p.dh[(size_t)node * H + j] = dhj;
    }
    TL_STAMP(ctrace, kTraceLevels - 1, 12);   // first warp: a node done
  }
  }
  __syncthreads();
  TL_STAMP(ctrace, kTraceLevels - 1, 13);     // all warps: nodes done
  if (!cleared()) return false;
  if (vb_first >= n_groups) return true;   // a CTA without a group has nothing to add (and 300 CTAs adding zeros to the same H x C words queue up)
  for (int i = tid; i < H * C; i += blockDim.x) atomicAdd(&p.dWc[i], s_dWc[i]);
  for (int i = tid; i < C; i += blockDim.x) atomicAdd(&p.dbc[i], s_dWc[H * C + i]);
  if (tid == 0) atomicAdd(p.loss, s_dWc[H * C + C]);
  TL_STAMP(ctrace, kTraceLevels - 1, 14);     // partial sums sent
  return true;
}
__global__ void __launch_bounds__(kClsWarps * 32) k_bwd_classifier(BwdParams p) {
  extern __shared__ float s_dyn[];
  classifier_groups(p, blockIdx.x, gridDim.x, s_dyn, AlreadyCleared{});
}

// ---- gate gradients of one wavefront -------------------------------------------------------- //
__device__ __forceinline__ void gates_element(const BwdParams& p, int row_begin, long long idx, int leaf) {
  const int H = p.H;
  const int row = row_begin + (int)(idx / H), u = (int)(idx % H);
  const int node = chk(p.st, p.order[row], p.n);
  const int gs = row_pitch(H);
  const float* g = p.gates + (size_t)node * 5 * gs + u;
  const float gi = g[0], go = g[3 * gs], gu = g[4 * gs];
  const float cn = p.c[(size_t)node * H + u];
  const float tc = tanhf(cn);
  const float dhn = p.dh[(size_t)node * H + u];
  const float dcn = p.dc[(size_t)node * H + u] + dhn * go * (1.f - tc * tc);
  float* dz = p.dz + (size_t)node * 5 * H + u;
  dz[0] = dcn * gu * gi * (1.f - gi);
  dz[3 * H] = dhn * tc * go * (1.f - go);
  dz[4 * H] = dcn * gi * (1.f - gu * gu);
  if (leaf) {
    dz[H] = 0.f;
    dz[2 * H] = 0.f;
  } else {
    const int l = chk(p.st, p.left[node], p.n), r = chk(p.st, p.right[node], p.n);
    const float gfl = g[gs], gfr = g[2 * gs];
    dz[H] = dcn * p.c[(size_t)l * H + u] * gfl * (1.f - gfl);
    dz[2 * H] = dcn * p.c[(size_t)r * H + u] * gfr * (1.f - gfr);
    p.dc[(size_t)l * H + u] = dcn * gfl;  // every node has exactly one caller: plain stores
    p.dc[(size_t)r * H + u] = dcn * gfr;
  }
}
__global__ void k_bwd_gates(BwdParams p, int row_begin, int row_end, int leaf) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < (long long)(row_end - row_begin) * p.H) gates_element(p, row_begin, idx, leaf);
}

// ---- dIn = dz W^T for one wavefront --------------------------------------------------------- //
// out[row][k] = sum_j dz[row][j] * W[koff + k][j]; tile 64 rows x 64 outputs, 16 x 16 threads.
// The next chunk of the contraction is fetched into registers while the current one is
// multiplied out of shared memory (two buffers, one CTA barrier per chunk).
constexpr int BT = 64, BK = 32;
constexpr int kLd = BT * BK / 256;   // elements of each operand per thread and chunk

constexpr int kDiRow = BK + 4;       // row stride: float4 reads along the contraction, 16 rows spread over all banks
struct DinputSmem {
  __align__(16) float As[2][BT][kDiRow];
  __align__(16) float Bs[2][BT][kDiRow];
  int node[BT];
  int dst_a[BT], dst_b[BT];   // where a row's dIn goes: left / right child, or (leaves) its row of dEmb_rows
  int fnode[2][BT], fleft[2][BT], fright[2][BT];   // the same for the blocks of dinput_fused: two sets used in turn
};
__device__ void dinput_block(const BwdParams& p, int row_begin, int row_end, int leaf, int bx, int by, int nby,
                             DinputSmem& sm) {
  float (*As)[BT][kDiRow] = sm.As;
  float (*Bs)[BT][kDiRow] = sm.Bs;
  int* s_node = sm.node;
  const int H = p.H, E = p.E, J = 5 * H;
  const int K = leaf ? E : 2 * H, koff = leaf ? 0 : E;
  const int tiles_k = (K + BT - 1) / BT;
  const int row0 = row_begin + (bx / tiles_k) * BT, k0 = (bx % tiles_k) * BT;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  __syncthreads();   // a previous block of this CTA may still be reading the shared arrays
  // the index chains (order -> children, or order -> token -> touched row) are resolved once per block
  for (int i = tid; i < BT; i += 256) {
    int node = -1, da = 0, db = 0;
    if (row0 + i < row_end) {
      node = chk(p.st, p.order[row0 + i], p.n);
      if (leaf) da = chk(p.st, p.tok_slot[chk(p.st, p.token[node], p.vocab)], p.n_leaves);
      else { da = chk(p.st, p.left[node], p.n); db = chk(p.st, p.right[node], p.n); }
    }
    s_node[i] = node; sm.dst_a[i] = da; sm.dst_b[i] = db;
  }
  __syncthreads();
  float acc[4][4] = {};
  float ra[kLd], rb[kLd];
  // Loads without a branch (rows and columns outside the block clamped onto valid ones); what they brought for
  // elements outside is replaced by zeros at the store - a use right behind the loads would make the
  // multiply-adds of the current chunk wait for them.
  auto fetch = [&](int j0) {
#pragma unroll
    for (int q = 0; q < kLd; ++q) {
      const int e = tid + q * 256, i = e / BK, j = min(j0 + e % BK, J - 1);
      ra[q] = p.dz[(size_t)max(s_node[i], 0) * J + j];
      rb[q] = __ldg(p.W + (size_t)(koff + min(k0 + i, K - 1)) * J + j);
    }
  };
  auto stash = [&](int buf, int j0) {
#pragma unroll
    for (int q = 0; q < kLd; ++q) {
      const int e = tid + q * 256, i = e / BK, j = j0 + e % BK;
      As[buf][i][e % BK] = (s_node[i] >= 0 && j < J) ? ra[q] : 0.f;
      Bs[buf][i][e % BK] = (k0 + i < K && j < J) ? rb[q] : 0.f;
    }
  };
  // gridDim.y CTAs share the contraction: each takes a contiguous run of chunks and adds its
  // partial sums with atomics (few levels fill the GPU on their own, the chain of dependent
  // memory round trips per CTA is what costs time)
  const int chunks_all = (J + BK - 1) / BK;
  const int per_split = (chunks_all + nby - 1) / nby;
  const int c_lo = by * per_split, chunks = min(chunks_all, c_lo + per_split);
  if (c_lo >= chunks) return;
  fetch(c_lo * BK);
  stash(c_lo & 1, c_lo * BK);
  __syncthreads();
  for (int cidx = c_lo; cidx < chunks; ++cidx) {
    const int buf = cidx & 1;
    if (cidx + 1 < chunks) fetch((cidx + 1) * BK);
#pragma unroll
    for (int jj = 0; jj < BK; jj += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = *reinterpret_cast<const float4*>(&As[buf][ty + 16 * i][jj]);
        b[i] = *reinterpret_cast<const float4*>(&Bs[buf][tx + 16 * i][jj]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[i][q] = fmaf(a[i].x, b[q].x, acc[i][q]);
          acc[i][q] = fmaf(a[i].y, b[q].y, acc[i][q]);
          acc[i][q] = fmaf(a[i].z, b[q].z, acc[i][q]);
          acc[i][q] = fmaf(a[i].w, b[q].w, acc[i][q]);
        }
    }
    if (cidx + 1 < chunks) stash(buf ^ 1, (cidx + 1) * BK);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int node = s_node[ty + 16 * i];
    if (node < 0) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + tx + 16 * q;
      if (k >= K) continue;
      if (leaf) {
        atomicAdd(&p.dEmb_rows[(size_t)sm.dst_a[ty + 16 * i] * E + k], acc[i][q]);
      } else {
        const int child = k < H ? sm.dst_a[ty + 16 * i] : sm.dst_b[ty + 16 * i];
        atomicAdd(&p.dh[(size_t)child * H + (k < H ? k : k - H)], acc[i][q]);
      }
    }
  }
}
// How many CTAs share the contraction of one dIn tile.  A 64 x 64 tile costs about 4 k cycles per
// 32-wide chunk of the contraction whatever the number of valid rows, so a wavefront with few tiles
// spreads the chunks over as many CTAs as there are (about two per SM), down to one chunk each.
__host__ __device__ inline int dinput_splits(int tiles, int J) {
  const int chunks_all = (J + BK - 1) / BK;
  if (tiles >= 148) return 1;
  int s = 296 / (tiles > 0 ? tiles : 1);
  if (s < 6) s = 6;
  return s < chunks_all ? s : chunks_all;
}
__host__ __device__ inline int dinput_tiles(int rows, int K) { return ((rows + BT - 1) / BT) * ((K + BT - 1) / BT); }
__global__ void __launch_bounds__(256)
k_bwd_dinput(BwdParams p, int row_begin, int row_end, int leaf) {
  __shared__ DinputSmem sm;
  dinput_block(p, row_begin, row_end, leaf, blockIdx.x, blockIdx.y, gridDim.y, sm);
}

// ---- narrow internal wavefronts of the one-launch backward: gate gradients inside the contraction -- //
// A block of dIn = dz W^T forms the dz values of its chunk itself instead of reading them back, so a
// narrow wavefront needs neither a pass of its own for the gate gradients nor the grid barrier behind
// it.  What does not depend on the wavefront above - the rows' index triples (node, left, right; kept
// by position in pos_left / pos_right, filled once at the start) and the weight chunk - is asked for
// with cp.async before the CTA enters the grid barrier and lands in shared memory while it waits;
// after the barrier one round of loads brings dh, dc (just written by the wavefront above) together
// with the forward's gate activations and cell states.  Same expressions as gates_element.  The
// blocks of the first output tile (k0 == 0) also store dz for the dW contraction and hand dc to the
// children; every (node, gate column) belongs to exactly one of them.
struct FusedItem {
  int row0, rows, k0, c_lo, chunks;   // first row (position in the ready order), valid rows, first output, chunk range
};
__device__ __forceinline__ FusedItem fused_item(const BwdParams& p, int row_begin, int row_end, int bx, int by, int nby) {
  const int K = 2 * p.H, J = 5 * p.H;
  const int tiles_k = (K + BT - 1) / BT;
  const int chunks_all = (J + BK - 1) / BK, per_split = (chunks_all + nby - 1) / nby;
  FusedItem it;
  it.row0 = row_begin + (bx / tiles_k) * BT;
  it.rows = min(BT, row_end - it.row0);
  it.k0 = (bx % tiles_k) * BT;
  it.c_lo = by * per_split;
  it.chunks = min(chunks_all, it.c_lo + per_split);
  return it;
}
// What a block needs that does not depend on the wavefront above, fetched into registers (a 4-byte cp.async
// per element measured ~130 cycles of issue each: slower than holding nine registers across the barrier) ...
struct FusedFetch {
  int idx;          // thread t < 192: order / pos_left / pos_right of row t % 64
  float w[kLd];     // the thread's elements of the first weight chunk
};
__device__ __forceinline__ void fused_fetch(const BwdParams& p, const FusedItem& it, int j0, FusedFetch& f) {
  const int J = 5 * p.H, K = 2 * p.H, t = threadIdx.x;
  f.idx = 0;
  if (t < 3 * BT) {
    const int which = t / BT, i = t % BT;
    const int pos = it.row0 + min(i, it.rows - 1);
    f.idx = *(which == 0 ? p.order + pos : (which == 1 ? p.pos_left + pos : p.pos_right + pos));
  }
#pragma unroll
  for (int q = 0; q < kLd; ++q) {
    const int e = t + q * 256, i = min(it.k0 + e / BK, K - 1), j = min(j0 + e % BK, J - 1);
    f.w[q] = __ldg(p.W + (size_t)(p.E + i) * J + j);
  }
}
// ... and put into index set `ib` and operand buffer `buf` (a CTA barrier must follow)
__device__ __forceinline__ void fused_deposit(const BwdParams& p, const FusedItem& it, DinputSmem& sm, int ib, int buf,
                                              int j0, const FusedFetch& f) {
  const int J = 5 * p.H, K = 2 * p.H, t = threadIdx.x;
  if (t < 3 * BT) {
    const int which = t / BT, i = t % BT;
    *(which == 0 ? &sm.fnode[ib][i] : (which == 1 ? &sm.fleft[ib][i] : &sm.fright[ib][i])) = f.idx;
  }
#pragma unroll
  for (int q = 0; q < kLd; ++q) {
    const int e = t + q * 256;
    sm.Bs[buf][e / BK][e % BK] = (it.k0 + e / BK < K && j0 + e % BK < J) ? f.w[q] : 0.f;
  }
}
// weight chunk j0 of the block into operand buffer `buf` (later chunks of a block)
__device__ __forceinline__ void fused_weights(const BwdParams& p, const FusedItem& it, DinputSmem& sm, int buf, int j0) {
  const int J = 5 * p.H, K = 2 * p.H, t = threadIdx.x;
  float w[kLd];
#pragma unroll
  for (int q = 0; q < kLd; ++q) {
    const int e = t + q * 256, i = min(it.k0 + e / BK, K - 1), j = min(j0 + e % BK, J - 1);
    w[q] = __ldg(p.W + (size_t)(p.E + i) * J + j);
  }
#pragma unroll
  for (int q = 0; q < kLd; ++q) {
    const int e = t + q * 256;
    sm.Bs[buf][e / BK][e % BK] = (it.k0 + e / BK < K && j0 + e % BK < J) ? w[q] : 0.f;
  }
}
__device__ __forceinline__ int gate_of_column(int j, int H) { return (j >= H) + (j >= 2 * H) + (j >= 3 * H) + (j >= 4 * H); }
// dz values of chunk j0 for the block's rows -> operand buffer `buf`.  All loads first and without a
// branch (rows and columns beyond the block are clamped onto valid ones and discarded afterwards), so that
// they are in flight together: one round trip instead of one per element; then the arithmetic and the stores.
__device__ __forceinline__ void fused_gate_gradients(const BwdParams& p, const FusedItem& it, DinputSmem& sm, int ib,
                                                     int buf, int j0) {
  const int H = p.H, J = 5 * H, gs = row_pitch(H), tid = threadIdx.x;
  float dhn[kLd], dci[kLd], go[kLd], cn[kLd], g1[kLd], g2[kLd];
#pragma unroll
  for (int q = 0; q < kLd; ++q) {
    const int e = tid + q * 256, i = min(e / BK, it.rows - 1), j = min(j0 + e % BK, J - 1);
    const int node = chk(p.st, sm.fnode[ib][i], p.n);
    const int g = gate_of_column(j, H), u = j - g * H;
    const bool forget = g == 1 || g == 2;
    const int child = chk(p.st, g == 2 ? sm.fright[ib][i] : sm.fleft[ib][i], p.n);
    const float* gt = p.gates + (size_t)node * 5 * gs + u;
    dhn[q] = p.dh[(size_t)node * H + u];
    dci[q] = p.dc[(size_t)node * H + u];
    go[q] = gt[3 * gs];
    cn[q] = p.c[(size_t)node * H + u];
    g1[q] = gt[forget ? g * gs : 0];                                   // f_l / f_r, else i
    g2[q] = *(forget ? p.c + (size_t)child * H + u : gt + 4 * gs);   // the child's cell state, else u
  }
  const bool keep = it.k0 == 0;
#pragma unroll
  for (int q = 0; q < kLd; ++q) {
    const int e = tid + q * 256, i = e / BK, j = j0 + e % BK;
    float dz = 0.f;
    if (i < it.rows && j < J) {
      const int node = chk(p.st, sm.fnode[ib][i], p.n);
      const int g = gate_of_column(j, H), u = j - g * H;
      const float tc = tanhf(cn[q]);
      const float dcn = dci[q] + dhn[q] * go[q] * (1.f - tc * tc);
      if (g == 3) {
        dz = dhn[q] * tc * go[q] * (1.f - go[q]);
      } else if (g == 1 || g == 2) {
        const float gf = g1[q];
        dz = dcn * g2[q] * gf * (1.f - gf);
        if (keep) p.dc[(size_t)chk(p.st, g == 1 ? sm.fleft[ib][i] : sm.fright[ib][i], p.n) * H + u] = dcn * gf;
      } else {
        const float gi = g1[q], gu = g2[q];
        dz = g == 0 ? dcn * gu * gi * (1.f - gi) : dcn * gi * (1.f - gu * gu);
      }
      if (keep) p.dz[(size_t)node * J + j] = dz;
    }
    sm.As[buf][i][e % BK] = dz;
  }
}
// one chunk of the contraction for the first 16 NI rows of the tile (thread (tx, ty): rows ty + 16 i, outputs tx + 16 q)
template <int NI>
__device__ __forceinline__ void fused_chunk(const DinputSmem& sm, int buf, int tx, int ty, float (&acc)[4][4]) {
#pragma unroll
  for (int jj = 0; jj < BK; jj += 4) {
    float4 a[NI], b[4];
#pragma unroll
    for (int i = 0; i < NI; ++i) a[i] = *reinterpret_cast<const float4*>(&sm.As[buf][ty + 16 * i][jj]);
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const float4*>(&sm.Bs[buf][tx + 16 * q][jj]);
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc[i][q] = fmaf(a[i].x, b[q].x, acc[i][q]);
        acc[i][q] = fmaf(a[i].y, b[q].y, acc[i][q]);
        acc[i][q] = fmaf(a[i].z, b[q].z, acc[i][q]);
        acc[i][q] = fmaf(a[i].w, b[q].w, acc[i][q]);
      }
  }
}
// One block.  fetched: `f` holds the block's index triples and first weight chunk (fused_fetch was called before
// the grid barrier) and no thread of the CTA still reads the operand buffers.
// buffers_free() runs once, when the block no longer needs the operand buffers and before its results go out.
template <class FreeFn>
__device__ __forceinline__ void dinput_fused(const BwdParams& p, const FusedItem& it, DinputSmem& sm, int ib, bool fetched,
                                             FusedFetch& f, long long* trace, int lvl, FreeFn buffers_free) {
  (void)trace; (void)lvl;
  if (it.c_lo >= it.chunks) { buffers_free(); return; }   // the same for every thread of the CTA
  const int H = p.H, K = 2 * H;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  if (!fetched) {
    __syncthreads();   // a previous block of this CTA may still be reading the shared arrays
    fused_fetch(p, it, it.c_lo * BK, f);
  }
  fused_deposit(p, it, sm, ib, it.c_lo & 1, it.c_lo * BK, f);
  __syncthreads();
  TL_STAMP(trace, lvl, 8);   // index triples and first weight chunk in shared memory
  float acc[4][4] = {};
  fused_gate_gradients(p, it, sm, ib, it.c_lo & 1, it.c_lo * BK);
  __syncthreads();
  TL_STAMP(trace, lvl, 5);   // gate gradients of the first chunk formed by all warps
  const int ni = (it.rows + 15) / 16;   // 16-row groups of the tile that hold nodes
  for (int cidx = it.c_lo; cidx < it.chunks; ++cidx) {
    const int buf = cidx & 1;
    const bool more = cidx + 1 < it.chunks;
    if (more) fused_weights(p, it, sm, buf ^ 1, (cidx + 1) * BK);
    if (ni == 1) fused_chunk<1>(sm, buf, tx, ty, acc);
    else if (ni == 2) fused_chunk<2>(sm, buf, tx, ty, acc);
    else if (ni == 3) fused_chunk<3>(sm, buf, tx, ty, acc);
    else fused_chunk<4>(sm, buf, tx, ty, acc);
    if (more) {
      fused_gate_gradients(p, it, sm, ib, buf ^ 1, (cidx + 1) * BK);
    }
    __syncthreads();
  }
  TL_STAMP(trace, lvl, 6);   // contraction done
  buffers_free();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = ty + 16 * i;
    if (r >= it.rows) continue;
    const int l = chk(p.st, sm.fleft[ib][r], p.n), rr = chk(p.st, sm.fright[ib][r], p.n);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = it.k0 + tx + 16 * q;
      if (k >= K) continue;
      atomicAdd(&p.dh[(size_t)(k < H ? l : rr) * H + (k < H ? k : k - H)], acc[i][q]);
    }
  }
}

// ---- dW = In^T dZ (contraction over nodes) and db ------------------------------------------- //
// part 0: rows [0,E) from the leaves (In = embedding rows); part 1: rows [E,E+2H) from the
// internal nodes (In = [h_l | h_r]).  Tile 64 (k) x 64 (j); gridDim.y splits the node range.
constexpr int WR = 32;               // nodes per chunk: enough multiply-adds per chunk to cover the fetch of the next one
constexpr int kLdW = WR * BT / 256;  // elements of each operand per thread and chunk

constexpr int kDwRows = 128;         // nodes per block of the dW contraction
struct DweightSmem {
  __align__(16) float As[2][WR][BT];
  __align__(16) float Bs[2][WR][BT];
  int node[kDwRows], ia[kDwRows], ib[kDwRows];   // node id and where its operand row comes from
};
__device__ void dweight_block(const BwdParams& p, int part, int row_begin, int row_end, int rows_per_split,
                              int bx, int by, DweightSmem& sm) {
  float (*As)[WR][BT] = sm.As;
  float (*Bs)[WR][BT] = sm.Bs;
  const int H = p.H, E = p.E, J = 5 * H;
  const int K = part == 0 ? E : 2 * H, koff = part == 0 ? 0 : E;
  const int tiles_j = (J + BT - 1) / BT;
  const int k0 = (bx / tiles_j) * BT, j0 = (bx % tiles_j) * BT;
  const int r_lo = row_begin + by * rows_per_split;
  __syncthreads();   // a previous block of this CTA may still be reading the shared arrays
  const int r_hi = min(row_end, r_lo + min(rows_per_split, kDwRows));
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // the index chain order -> token / children is resolved once per block, not once per fetched element
  for (int i = tid; i < kDwRows; i += 256) {
    int node = 0, ia = 0, ib = 0;
    if (r_lo + i < r_hi) {
      node = chk(p.st, p.order[r_lo + i], p.n);
      if (part == 0) ia = chk(p.st, p.token[node], p.vocab);
      else { ia = chk(p.st, p.left[node], p.n); ib = chk(p.st, p.right[node], p.n); }
    }
    sm.node[i] = node; sm.ia[i] = ia; sm.ib[i] = ib;
  }
  __syncthreads();
  float acc[4][4] = {};
  float ra[kLdW], rb[kLdW];
  // element e of a chunk: node rr = e / 64 of the chunk, column cc = e % 64 of the tile
  auto fetch = [&](int r0) {
#pragma unroll
    for (int q = 0; q < kLdW; ++q) {
      const int e = tid + q * 256, rr = e / BT, cc = e % BT;
      const int row = r0 + rr;
      float va = 0.f, vb = 0.f;
      if (row < r_hi) {
        const int li = row - r_lo;
        const int k = k0 + cc, j = j0 + cc;
        if (k < K) {
          if (part == 0) va = __ldg(p.emb + (size_t)sm.ia[li] * E + k);
          else va = k < H ? p.h[(size_t)sm.ia[li] * H + k] : p.h[(size_t)sm.ib[li] * H + (k - H)];
        }
        if (j < J) vb = p.dz[(size_t)sm.node[li] * J + j];
      }
      ra[q] = va;
      rb[q] = vb;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int q = 0; q < kLdW; ++q) {
      const int e = tid + q * 256;
      As[buf][e / BT][e % BT] = ra[q];
      Bs[buf][e / BT][e % BT] = rb[q];
    }
  };
  if (r_lo < r_hi) {
    fetch(r_lo);
    stash(0);
  }
  __syncthreads();
  int buf = 0;
  for (int r0 = r_lo; r0 < r_hi; r0 += WR, buf ^= 1) {
    if (r0 + WR < r_hi) fetch(r0 + WR);
#pragma unroll
    for (int rr = 0; rr < WR; ++rr) {   // thread (tx, ty): outputs k0 + 4 ty .. + 3  x  j0 + 4 tx .. + 3
      const float4 a4 = *reinterpret_cast<const float4*>(&As[buf][rr][4 * ty]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][rr][4 * tx]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = fmaf(a[i], b[q], acc[i][q]);
    }
    if (r0 + WR < r_hi) stash(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = k0 + 4 * ty + i;
    if (k >= K) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + 4 * tx + q;
      if (j < J) atomicAdd(&p.dW[(size_t)(koff + k) * J + j], acc[i][q]);
    }
  }
}
__global__ void __launch_bounds__(256)
k_bwd_dweight(BwdParams p, int part, int row_begin, int row_end, int rows_per_split) {
  __shared__ DweightSmem sm;
  dweight_block(p, part, row_begin, row_end, rows_per_split, blockIdx.x, blockIdx.y, sm);
}

// column j of db over the nodes [256 by, 256 by + 256)
__device__ __forceinline__ void dbias_piece(const BwdParams& p, int j, int by) {
  const int J = 5 * p.H;
  const int r_lo = by * 256, r_hi = min(p.n, r_lo + 256);
  float acc = 0.f;
  for (int r = r_lo; r < r_hi; ++r) acc += p.dz[(size_t)r * J + j];
  atomicAdd(&p.db[j], acc);
}
__global__ void k_bwd_dbias(BwdParams p) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < 5 * p.H) dbias_piece(p, j, blockIdx.y);
}

// ---- the whole backward pass in one cooperative launch --------------------------------------- //
// Used after a forward that left the level table on the device only (persistent / sub-forest
// modes): no host round trip, no launch per wavefront.  Phases, separated by the bounded grid
// barrier: clear the outputs | mark leaf tokens | token scan (CTA 0) next to the classifier (all
// other CTAs) | per wavefront from the top: gate gradients, then dIn = dz W^T into the children |
// dW, db (they only need every dz).
constexpr int kFusedMaxRows = 128;   // widest wavefront whose gate gradients are formed inside the contraction
#ifdef TREELSTM_TRACE
#define TL_TRACE_ARG trace
#else
#define TL_TRACE_ARG nullptr
#endif
union BwdSmem {
  DinputSmem di;
  DweightSmem dw;
};
template <class T>
__device__ __forceinline__ void zero_range(T* ptr, size_t count, size_t gtid, size_t gthreads) {
  for (size_t i = gtid; i < count; i += gthreads) ptr[i] = T(0);
}
__global__ void __launch_bounds__(256, 2)
k_bwd_persistent(BwdParams p, const int* level_offset, long long wait_limit, int with_dweight, int after_trees) {
  extern __shared__ float4 s_dyn4[];
  BwdSmem& sm = *reinterpret_cast<BwdSmem*>(s_dyn4);
  float* s_cls = reinterpret_cast<float*>(s_dyn4) + (sizeof(BwdSmem) + 3) / 4;
  __shared__ int s_flag;
  if (ld_volatile(&p.st->status) != 0) return;
  // behind k_bwd_begin and the tree kernel: classifier and token table are done, and only forests that the latter leaves
  const bool after_begin = after_trees != 0;
  if (after_begin && p.st->trees_bwd) return;
  const int n_levels = p.st->n_levels;
  const int n = p.n, H = p.H, E = p.E, C = p.C, J = 5 * H;
#ifdef TREELSTM_TRACE
  // first CTA, first thread: row l of the stamp table = wavefront l (slot 0 start, 1 gate gradients done,
  // 2 barrier, 3 input gradients done, 4 barrier); last row = phases of the kernel
  long long* const trace = blockIdx.x == 0 && threadIdx.x == 0 ? p.trace : nullptr;
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  p.n_leaves = n_levels > 0 ? level_offset[1] : 0;
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, gthreads = (size_t)gridDim.x * blockDim.x;
  unsigned int arrivals = 0;
  auto barrier = [&]() {
    arrivals += gridDim.x;
    return grid_barrier(p.st, arrivals, wait_limit, &s_flag, true, after_begin ? &p.st->barrier_levels : &p.st->barrier_bwd);
  };
  if (after_begin) {
    zero_range(p.dc, (size_t)n * H, gtid, gthreads);
  } else {
    if (gtid == 0) { *p.loss = 0.f; *p.n_touched = 0; }
    zero_range(p.dW, (size_t)(E + 2 * H) * J, gtid, gthreads);
    zero_range(p.db, (size_t)J, gtid, gthreads);
    zero_range(p.dWc, (size_t)H * C, gtid, gthreads);
    zero_range(p.dbc, (size_t)C, gtid, gthreads);
    zero_range(p.dc, (size_t)n * H, gtid, gthreads);
    zero_range(p.tok_slot, (size_t)p.vocab + 1, gtid, gthreads);
    zero_range(p.dEmb_rows, (size_t)p.n_leaves * E, gtid, gthreads);
    if (!barrier()) return;
    TL_STAMP(trace, kTraceLevels - 1, 1);   // outputs and scratch cleared
    for (size_t r = gtid; r < (size_t)p.n_leaves; r += gthreads)
      p.tok_slot[chk(p.st, p.token[chk(p.st, p.order[r], p.n)], p.vocab)] = 1;
  }
  for (size_t r = (size_t)p.n_leaves + gtid; r < (size_t)n; r += gthreads) {   // children by ready position
    const int node = chk(p.st, p.order[r], p.n);
    p.pos_left[r] = p.left[node];
    p.pos_right[r] = p.right[node];
  }
  if (!barrier()) return;
  TL_STAMP(trace, kTraceLevels - 1, 2);   // tokens marked
  // (the CTA's operand buffers are idle in this phase: they hold the scan's ballots)
  unsigned int* const s_mask = reinterpret_cast<unsigned int*>(s_dyn4);
  const int mask_cap = (int)(sizeof(BwdSmem) / sizeof(unsigned int));
  int* const group_count = p.tok_slot + p.vocab + 4;   // behind the table and its spare entries
  if (after_begin) {
  } else if (gridDim.x == 1) {
    scan_tokens(p, s_mask, mask_cap);
    classifier_groups(p, 0, 1, s_cls, AlreadyCleared{});
  } else {
    scan_count_groups(p, group_count);
    classifier_groups(p, blockIdx.x, gridDim.x, s_cls, AlreadyCleared{});
  }
  TL_STAMP(trace, kTraceLevels - 1, 3);   // this CTA's part (the first one: the token scan) done
  if (!after_begin && !barrier()) return;
  TL_STAMP(trace, kTraceLevels - 1, 4);   // classifier, loss and token scan done everywhere
  if (!after_begin && gridDim.x > 1) scan_place_groups(p, group_count);   // needs nothing but the counts; its results are read after the kernel
  // the first wavefront boundaries in shared memory: no dependent global load after every barrier
  // (filled here, ordered before its first use by the CTA barriers inside the grid barrier above)
  constexpr int kOffCache = 256;
  __shared__ int s_off[kOffCache];
  for (int i = threadIdx.x; i < kOffCache && i <= n_levels; i += blockDim.x) s_off[i] = level_offset[i];
  __syncthreads();
  auto level_begin = [&](int l) { return l < kOffCache ? s_off[l] : level_offset[l]; };
  auto is_fused = [&](int l) { return l > 0 && level_begin(l + 1) - level_begin(l) <= kFusedMaxRows; };
  // this CTA's first block of every narrow wavefront, worked out once (thread l: wavefront l) - the
  // divisions behind it would otherwise sit between a wavefront's last store and the grid barrier
  auto first_block = [&](int l) {
    FusedItem it{};   // c_lo == chunks == 0: no block
    if (is_fused(l)) {
      const int b = level_begin(l), e = level_begin(l + 1);
      const int ntiles = dinput_tiles(e - b, 2 * H), nsplits = dinput_splits(ntiles, J);
      if ((int)blockIdx.x < ntiles * nsplits) it = fused_item(p, b, e, blockIdx.x % ntiles, blockIdx.x / ntiles, nsplits);
    }
    return it;
  };
  __shared__ FusedItem s_first[kOffCache];
  for (int l = threadIdx.x; l < kOffCache && l < n_levels; l += blockDim.x) s_first[l] = first_block(l);
  __syncthreads();
  bool prepared = false;
  FusedItem pre_item{};
  FusedFetch pre_fetch;
  for (int lvl = n_levels - 1; lvl >= 0; --lvl) {
    const int begin = level_begin(lvl), end = level_begin(lvl + 1), leaf = lvl == 0 ? 1 : 0;
    const long long elems = (long long)(end - begin) * H;
    TL_STAMP(trace, lvl, 0);
    // a narrow internal wavefront forms its gate gradients inside the contraction (dinput_fused)
    const bool fused = is_fused(lvl);
    if (!fused) {
      for (long long idx = (long long)gtid; idx < elems; idx += (long long)gthreads) gates_element(p, begin, idx, leaf);
      TL_STAMP(trace, lvl, 1);
      if (leaf && !with_dweight) break;   // the leaves' input gradients are left to the tensor-core kernel as well
      if (!barrier()) return;
    }
    TL_STAMP(trace, lvl, 2);
    const int tiles = dinput_tiles(end - begin, leaf ? E : 2 * H), splits = dinput_splits(tiles, J);
    // This CTA's first block of the next wavefront: its index triples and first weight chunk are requested
    // as soon as the operand buffers are free - ahead of the atomic adds of this wavefront's results, which
    // would otherwise hold the requests up - and land in shared memory during the grid barrier.
    bool requested = false;
    auto request_next = [&]() {
      TL_STAMP(trace, lvl, 9);
      requested = true;
      prepared = false;
      if (lvl > 1) {
        pre_item = lvl - 1 < kOffCache ? s_first[lvl - 1] : first_block(lvl - 1);
        if (pre_item.c_lo < pre_item.chunks) {
          fused_fetch(p, pre_item, pre_item.c_lo * BK, pre_fetch);
          prepared = true;
        }
      }
      TL_STAMP(trace, lvl, 11);
    };
    if (fused) {
      for (int vb = blockIdx.x; vb < tiles * splits; vb += gridDim.x) {
        const bool ready = prepared && vb == (int)blockIdx.x;
        const bool last = vb + (int)gridDim.x >= tiles * splits;
        const FusedItem item = ready ? pre_item : fused_item(p, begin, end, vb % tiles, vb / tiles, splits);
        if (last) dinput_fused(p, item, sm.di, lvl & 1, ready, pre_fetch, TL_TRACE_ARG, lvl, request_next);
        else dinput_fused(p, item, sm.di, lvl & 1, ready, pre_fetch, TL_TRACE_ARG, lvl, []() {});
      }
      TL_STAMP(trace, lvl, 7);   // own blocks done
    } else {
      for (int vb = blockIdx.x; vb < tiles * splits; vb += gridDim.x)
        dinput_block(p, begin, end, leaf, vb % tiles, vb / tiles, splits, sm.di);
    }
    if (!requested) request_next();
    TL_STAMP(trace, lvl, 3);
    if (lvl > 0 && !barrier()) return;   // the leaves' dIn goes to the embedding rows only
    TL_STAMP(trace, lvl, 4);
  }
  TL_STAMP(trace, kTraceLevels - 1, 5);   // all wavefronts done
  if (!with_dweight) return;              // dW, db and the leaves' dIn are left to the tensor-core kernel that follows on the stream
  const int tiles_j = (J + BT - 1) / BT, rows_per_split = kDwRows;
  for (int part = 0; part < 2; ++part) {
    const int begin = part == 0 ? 0 : p.n_leaves, end = part == 0 ? p.n_leaves : n;
    if (end <= begin) continue;
    const int K = part == 0 ? E : 2 * H;
    const int nbx = ((K + BT - 1) / BT) * tiles_j, nby = (end - begin + rows_per_split - 1) / rows_per_split;
    for (int vb = blockIdx.x; vb < nbx * nby; vb += gridDim.x)
      dweight_block(p, part, begin, end, rows_per_split, vb % nbx, vb / nbx, sm.dw);
    TL_STAMP(trace, kTraceLevels - 1, 6 + part);   // this CTA's blocks of dW from the leaves / the internal nodes done
  }
  const int nby = (n + 255) / 256;
  for (long long idx = (long long)gtid; idx < (long long)J * nby; idx += (long long)gthreads)
    dbias_piece(p, (int)(idx % J), (int)(idx / J));
  TL_STAMP(trace, kTraceLevels - 1, 8);
}

// ---- the wavefronts of a forest that is wide, on the tensor cores ------------------------------ //
// Behind k_bwd_begin, for the forests that the tree kernel leaves.  On fp32 units the contraction dIn = dz W^T of the wide
// wavefronts was 600 of the 880 us of the backward pass of 14.6 k nodes (H = 256).  Here dz is split into bf16 pieces
// (BwdImages, the layout the tensor core reads), and tiles of 128 positions x 128 outputs are multiplied with W split once
// per set of weights: one thread asks for blocks (plain bulk copies of whole tiles), one issues the MMAs, sixteen warps
// add the tile to the children's dh.  The leaves' dIn (their rows of dEmb) is one more such wavefront.  The images stay for the weight
// gradient.  What is left is latency.  Cycles of a wavefront, H = 256, 14.3 k nodes: 15 - 20 k of one of 11 to 83 nodes (4 - 9 k gate gradients, 2.5 k MMAs, 1.2 k read
// back, 4 k adds, 3.2 k grid barrier), 27 - 32 k of 130 to 460, 37 k of 960, 71 k of 2.4 k; 318 us in all (ncu, 19 wavefronts).
constexpr int kWideSmem = 2 * kSpStageBytes + 1024, kWideThreads = 512;
// A wavefront of one tile of nodes forms its gate gradients where the tensor core reads them, which saves the images and a grid barrier; every tile of outputs
// forms them again.  Two tiles of nodes: wide_direct_rows.  Where a CTA has two blocks of them (H > 224) it does not pay: 33 k cycles, through the images 27 k.
constexpr int kWideOffCache = 512;
struct WideArgs {
  const int* level_offset;
  long long wait_limit;
  int after_trees, direct_rows;
  BwdImages img;
};

// How the dIn of a wavefront is cut: tiles of 128 positions (from `base` on) x 128 outputs, each `span` steps long (kbs
// blocks of 64 gate columns, padded to a multiple of `per`); a CTA takes `per` steps after the other.
struct WidePlan {
  int begin, end, base, leaf, direct, to, kbs, span, per, total, skip_first, skip;
};
// The widest wavefront that is formed in place: two tiles of nodes if no CTA has two blocks, loads are of 16 bytes, and rows are whole lines of 128 bytes, so that what is formed
// again reads no parts of more lines, or so short that there is little to it.  Backward passes with 14 wavefronts of 190 to 200 nodes, in place | through the images, us:
// whole lines H = 96 361 | 372, 128 367 | 379, 160 393 | 412, 192 434 | 458, 224 463 | 480 (64, one tile of outputs and few CTAs either way, 334 | 332); short ones
// H = 8 402 | 412, 16 360 | 377, 32 353 | 365; others H = 40 380 | 376, 100 483 | 466, 120 409 | 394, 144 410 | 408, 168 434 | 423, 176 418 | 421, 200 479 | 466,
// 208 474 | 480; loads of 4 bytes H = 30 401 | 394, 150 557 | 468; two blocks a CTA H = 232 575 | 494, 256 518 | 485.  With 130 and 256 nodes the same, 1 to 5 % either way.
inline int wide_direct_rows(int H, int grid, bool vec_h) {
  const int to = (2 * H + 127) / 128;
  return vec_h && (H <= 32 || (H % 32 == 0 && to > 1)) && 2 * to * wsp_kblocks(H) <= grid ? 2 * kSpTile : kSpTile;
}
__device__ __forceinline__ WidePlan wide_plan(int begin, int end, int leaf, int H, int E, int grid, int direct_rows) {
  WidePlan w;
  w.begin = begin; w.end = end; w.leaf = leaf;
  w.direct = !leaf && end - begin <= direct_rows;
  w.base = w.direct ? begin : begin & ~63;
  w.to = ((leaf ? E : 2 * H) + 127) / 128;
  const int tiles = (end - w.base + 127) / 128 * w.to, gp = gate_pitch(H);
  w.kbs = wsp_kblocks(H);
  w.skip_first = w.kbs; w.skip = 0;
  if (leaf) {                                            // a leaf's forget gates are zero: blocks inside them are left out
    w.skip_first = (gp + 63) / 64;
    w.skip = max(0, 3 * gp / 64 - w.skip_first);
    w.kbs -= w.skip;
  }
  if (w.direct) w.per = tiles * w.kbs <= grid ? 1 : 2;
  else if (2 * tiles > grid) w.per = (tiles * w.kbs + grid - 1) / grid;   // equal shares, whatever tile they lie in
  else w.per = (w.kbs + grid / tiles - 1) / (grid / tiles);
  w.span = !w.direct && 2 * tiles > grid ? w.kbs : (w.kbs + w.per - 1) / w.per * w.per;
  w.total = tiles * w.span;
  return w;
}

// units u0 .. u0 + 7 of a row of H; what lies behind the row repeats units of it.  kVec: 16-byte loads (H a multiple of 4)
template <bool kVec>
__device__ __forceinline__ void load8(const float* row, int u0, int H, float (&x)[8]) {
  if (kVec) {
    const float4 a = *reinterpret_cast<const float4*>(row + u0), b = *reinterpret_cast<const float4*>(row + min(u0 + 4, H - 4));
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = row[min(u0 + k, H - 1)];
  }
}
template <bool kVec>
__device__ __forceinline__ void store_units(float* row, int u0, int H, const float (&x)[8]) {
  if (kVec) {
    *reinterpret_cast<float4*>(row + u0) = make_float4(x[0], x[1], x[2], x[3]);
    if (u0 + 4 < H) *reinterpret_cast<float4*>(row + u0 + 4) = make_float4(x[4], x[5], x[6], x[7]);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (u0 + k < H) row[u0 + k] = x[k];
  }
}
__device__ __forceinline__ unsigned char* dz_unit(const BwdImages& img, int pos, int kb, int ju) {
  return img.dz + ((size_t)(pos >> 6) * ju + kb) * kUnitBytes;
}

// This CTA's share of a wavefront's gate gradients -> image, dc of the children.  A thread forms the five gates of eight
// units of one node at a time: all its loads are in flight together and every store is a whole 16-byte piece.
// (One element per thread through shared memory: 12 k cycles for eight nodes per CTA.)
template <bool kVec>
__device__ __forceinline__ void wide_gates(const BwdParams& p, const BwdImages& img, const WidePlan& w) {
  const int H = p.H, gs = row_pitch(H), gp = gate_pitch(H), octs = gp / 8, ju = img_units(5 * gp), tid = threadIdx.x;
  const long long all = (long long)(w.end - w.begin) * octs;
  const int share = (int)((all + gridDim.x - 1) / gridDim.x + 31) / 32 * 32;
  const long long lo = (long long)blockIdx.x * share, hi = min(all, lo + share);
  const int keep_zero = w.leaf ? w.end & ~63 : 0;        // leaves below: nobody reads the blocks of their forget gates
  for (long long e = lo + tid; e < hi; e += kWideThreads) {
    const int i = (int)(e / octs), o = (int)(e - (long long)i * octs), u0 = 8 * o, pos = w.begin + i;
    const int node = chk(p.st, p.order[pos], p.n);
    const int l = w.leaf ? node : chk(p.st, p.pos_left[pos], p.n), r = w.leaf ? node : chk(p.st, p.pos_right[pos], p.n);
    const float* g = p.gates + (size_t)node * 5 * gs;
    float gi[8], go[8], gu[8], c[8], dh[8], dc[8], z[8];
    load8<kVec>(p.c + (size_t)node * H, u0, H, c);
    load8<kVec>(p.dh + (size_t)node * H, u0, H, dh);
    load8<kVec>(p.dc + (size_t)node * H, u0, H, dc);
    load8<true>(g + 3 * gs, u0, gs, go);
    load8<true>(g, u0, gs, gi);
    load8<true>(g + 4 * gs, u0, gs, gu);
    auto put = [&](int gate) {
      const int j = gate * gp + u0;
#pragma unroll
      for (int k = 0; k < 8; ++k) z[k] = u0 + k < H ? z[k] : 0.f;
      split_store8_unit(dz_unit(img, pos, j >> 6, ju), pos & 63, (j >> 3) & 7, z);
    };
    float gf[2][8], cc[2][8];
    if (!w.leaf) {
      load8<true>(g + gs, u0, gs, gf[0]);
      load8<true>(g + 2 * gs, u0, gs, gf[1]);
      load8<kVec>(p.c + (size_t)l * H, u0, H, cc[0]);
      load8<kVec>(p.c + (size_t)r * H, u0, H, cc[1]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float tc = tanhf(c[k]);
      z[k] = dh[k] * tc * go[k] * (1.f - go[k]);
      dc[k] += dh[k] * go[k] * (1.f - tc * tc);
    }
    put(3);
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = dc[k] * gu[k] * gi[k] * (1.f - gi[k]);
    put(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = dc[k] * gi[k] * (1.f - gu[k] * gu[k]);
    put(4);
    if (!w.leaf) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          z[k] = dc[k] * cc[q][k] * gf[q][k] * (1.f - gf[q][k]);
          gf[q][k] *= dc[k];
        }
        put(1 + q);
        store_units<kVec>(p.dc + (size_t)(q ? r : l) * H, u0, H, gf[q]);   // every node has exactly one caller: plain stores
      }
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) z[k] = 0.f;
      for (int q = 1; q < 3; ++q) {
        const int kb = (q * gp + u0) >> 6;
        if (pos >= keep_zero || !forget_tile(kb >> 1, gp)) put(q);
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = 0.f;
    for (int x = 5 * octs + o; x < 8 * ju; x += octs)    // columns behind the last gate
      split_store8_unit(dz_unit(img, pos, x >> 3, ju), pos & 63, x & 7, z);
  }
}

// Block kb of a narrow wavefront's gate gradients, formed where the tensor core reads it: rows 0 .. rows - 1 of the
// tile are the nodes in s_node.  keep: this CTA also stores the block in the image and hands dc to the children.
template <bool kVec>
__device__ __forceinline__ void direct_block(const BwdParams& p, const BwdImages& img, unsigned char* tile, int kb, int pos0, int rows,
                                             bool keep, const int* s_node, const int* s_left, const int* s_right) {
  const int H = p.H, gs = row_pitch(H), gp = gate_pitch(H), ju = img_units(5 * gp), c = threadIdx.x & 7, j = kb * 64 + 8 * c;
  const int gate = j / gp, u0 = j - gate * gp;
  const bool forget = gate == 1 || gate == 2;
  for (int i = threadIdx.x >> 3; i < rows; i += kWideThreads / 8) {
    float z[8];
    if (gate < 5) {
      const int node = s_node[i], child = gate == 2 ? s_right[i] : s_left[i];
      const float* g = p.gates + (size_t)node * 5 * gs;
      float dh[8], dc[8], go[8], cn[8], g1[8], g2[8];
      load8<kVec>(p.dh + (size_t)node * H, u0, H, dh);
      load8<kVec>(p.dc + (size_t)node * H, u0, H, dc);
      load8<true>(g + 3 * gs, u0, gs, go);
      load8<kVec>(p.c + (size_t)node * H, u0, H, cn);
      load8<true>(g + (forget ? gate * gs : 0), u0, gs, g1);                         // f_l / f_r, else i
      if (forget) load8<kVec>(p.c + (size_t)child * H, u0, H, g2);                  // the child's cell state, else u
      else load8<true>(g + 4 * gs, u0, gs, g2);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float tc = tanhf(cn[k]), dcn = dc[k] + dh[k] * go[k] * (1.f - tc * tc);
        const float a = gate == 3 ? dh[k] * tc : dcn * (gate == 4 ? g1[k] : g2[k]);
        const float b = gate == 3 ? go[k] : (gate == 4 ? 1.f : g1[k]);
        const float d = gate == 3 ? go[k] : (gate == 4 ? g2[k] * g2[k] : g1[k]);
        z[k] = u0 + k < H ? a * b * (1.f - d) : 0.f;
        g1[k] *= dcn;
      }
      if (keep && forget) store_units<kVec>(p.dc + (size_t)child * H, u0, H, g1);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) z[k] = 0.f;
    }
    split_store8(tile, i, c, z);
    if (keep) split_store8_unit(dz_unit(img, pos0 + i, kb, ju), (pos0 + i) & 63, c, z);
  }
}

// 64 rows of the inputs' images (leaves first: embedding row and a one; then internal nodes: [h_l | h_r] and a one);
// eight lanes per row, four units in flight
template <bool kVec>
__device__ __forceinline__ void input_rows(const BwdParams& p, const BwdImages& img, int chunk, int rows0) {
  const int H = p.H, E = p.E, n = p.n, c = threadIdx.x & 7;
  const int q = chunk * 64 + (threadIdx.x >> 3), part = q >= rows0;
  const int pos = part ? p.n_leaves / 64 * 64 + q - rows0 : q, feats = part ? 2 * H : E, units = img_units(feats + 1);
  const bool in = part ? pos >= p.n_leaves && pos < n : pos < p.n_leaves;
  const float *s0 = p.h, *s1 = p.h;
  if (in) {
    if (part) {
      s0 = p.h + (size_t)chk(p.st, p.pos_left[pos], p.n) * H;
      s1 = p.h + (size_t)chk(p.st, p.pos_right[pos], p.n) * H - H;
    } else {
      s0 = p.emb + (size_t)chk(p.st, p.token[chk(p.st, p.order[pos], p.n)], p.vocab) * E;
    }
  }
  unsigned char* row = img.x[part] + (size_t)(pos >> 6) * units * kUnitBytes;
  constexpr int kF = 4;
  for (int fb = 0; fb < units; fb += kF) {
    float x[kF][8];
#pragma unroll
    for (int v = 0; v < kF; ++v) {
      const int f = (fb + v) * 64 + c * 8;
      if (kVec) {
#pragma unroll
        for (int q4 = 0; q4 < 2; ++q4) {
          const int fc = min(f + 4 * q4, feats - 4);
          const float4 t = *reinterpret_cast<const float4*>(in ? (part && fc >= H ? s1 : s0) + fc : s0);
          x[v][4 * q4] = t.x; x[v][4 * q4 + 1] = t.y; x[v][4 * q4 + 2] = t.z; x[v][4 * q4 + 3] = t.w;
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int fc = min(f + k, feats - 1);
          x[v][k] = *(in ? (part && fc >= H ? s1 : s0) + fc : s0);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < kF; ++v) {
      if (fb + v >= units) break;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int f = (fb + v) * 64 + c * 8 + k;
        x[v][k] = in ? (f < feats ? x[v][k] : (f == feats ? 1.f : 0.f)) : 0.f;
      }
      split_store8_unit(row + (size_t)(fb + v) * kUnitBytes, pos & 63, c, x[v]);
    }
  }
}

__global__ void __launch_bounds__(kWideThreads, 1) k_bwd_wide(BwdParams p, WideArgs a) {
  extern __shared__ unsigned char wide_dyn[];
  __shared__ __align__(8) uint64_t s_bars[6];            // full, empty (two stages each), accumulator, drain
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort, s_flag;
  __shared__ int s_node[kSpTile], s_da[kSpTile], s_db[kSpTile];
  __shared__ int s_off[kWideOffCache];
  if (ld_volatile(&p.st->status) != 0 || (a.after_trees && p.st->trees_bwd)) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grid = (int)gridDim.x;
  unsigned char* const tiles = wide_dyn + ((1024u - (smem_u32(wide_dyn) & 1023u)) & 1023u);
  const uint32_t tiles_addr = smem_u32(tiles), full0 = smem_u32(&s_bars[0]), empty0 = smem_u32(&s_bars[2]),
                 acc_bar = smem_u32(&s_bars[4]), drain_bar = smem_u32(&s_bars[5]);
  if (tid == 0) {
    for (int s = 0; s < 6; ++s) mbar_init(smem_u32(&s_bars[s]), 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int n_levels = p.st->n_levels, n = p.n, H = p.H, E = p.E, gp = gate_pitch(H), ju = img_units(5 * gp);
  for (int l = tid; l < kWideOffCache && l <= n_levels; l += kWideThreads) s_off[l] = a.level_offset[l];
  if (warp == 0) tmem_alloc(smem_u32(&s_tmem), kSpTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = s_tmem;
  auto level_begin = [&](int l) { return l < kWideOffCache ? s_off[l] : a.level_offset[l]; };
  p.n_leaves = n_levels > 0 ? level_begin(1) : 0;
  const int n_leaves = p.n_leaves, wsp_kb = wsp_kblocks(H);
  // 16-byte accesses to rows of H (and E): whether every row starts on a 16-byte boundary
  const bool vec_h = H % 4 == 0 && ((reinterpret_cast<uintptr_t>(p.h) | reinterpret_cast<uintptr_t>(p.c)) & 15) == 0;
  const bool vec_e = E % 4 == 0 && (reinterpret_cast<uintptr_t>(p.dEmb_rows) & 15) == 0;
  const bool vec_x = vec_h && E % 4 == 0 && (reinterpret_cast<uintptr_t>(p.emb) & 15) == 0;
#ifdef TREELSTM_TRACE
  long long* const trace = blockIdx.x == 0 && tid == 0 ? p.trace : nullptr;
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  unsigned int arrivals = 0;
  bool arrived = false;                                  // at the next barrier already
  auto barrier = [&]() {
    arrivals += gridDim.x;
    const bool arrive = !arrived;
    arrived = false;
    return grid_barrier(p.st, arrivals, a.wait_limit, &s_flag, arrive, &p.st->barrier_levels);
  };
  // The inputs' images are for the kernel behind this one: CTAs without a share of a wavefront write them.  They have nothing to tell the others, and
  // arrive at the wavefront's barrier before: 64 rows take 10 k cycles, about as long as a narrow wavefront, and three of those had
  // taken 21 k and not 11 k (training step, 256 sentences bf16: 605.1 -> 598.3 us).
  const int rows0 = (n_leaves + 63) / 64 * 64, chunks = rows0 / 64 + (n > n_leaves ? (n + 63) / 64 - n_leaves / 64 : 0);
  int chunks_done = 0;
  auto input_chunk = [&](int chunk) {
    if (vec_x) input_rows<true>(p, a.img, chunk, rows0);
    else input_rows<false>(p, a.img, chunk, rows0);
  };
  {                                                      // zeros behind the last position
    const float zero[8] = {};
    for (int q = (int)blockIdx.x * kWideThreads + tid; q < ((n + 63) / 64 * 64 - n) * ju * 8; q += grid * kWideThreads)
      split_store8_unit(dz_unit(a.img, n, q % (ju * 8) >> 3, ju), (n + q / (ju * 8)) & 63, q & 7, zero);
  }
  bool ok = true, fetched = false, tables = false;       // of the next tile: tables read and blocks asked for; tables alone
  uint32_t blk = 0, asked = 0, done = 0;                 // blocks multiplied; asked for (thread 0); tiles
  auto read_tables = [&](const WidePlan& w, int pos0) {  // the nodes of a tile and where its rows go
    if (tid >= kSpTile) return;
    const int pos = pos0 + tid;
    int node = 0, da = -1, db = 0;
    if (pos >= w.begin && pos < w.end) {
      if (w.leaf) {
        da = chk(p.st, p.tok_slot[chk(p.st, p.token[chk(p.st, p.order[pos], p.n)], p.vocab)], p.n_leaves);
      } else {
        if (w.direct) node = chk(p.st, p.order[pos], p.n);
        da = chk(p.st, p.pos_left[pos], p.n);
        db = chk(p.st, p.pos_right[pos], p.n);
      }
    }
    s_node[tid] = node; s_da[tid] = da; s_db[tid] = db;
  };
  // thread 0: blocks k0 .. k0 + nk - 1 of a tile -> the ring; the weights of the first `early` of them have been asked for ahead (ask_weights)
  auto weights_at = [&](const WidePlan& w, int ot, int k) {
    const int kb = k < w.skip_first ? k : k + w.skip;
    return a.img.w + ((size_t)((w.leaf ? 0 : wsp_tiles_x(E)) + ot) * wsp_kb + kb) * kSpOperandBytes;
  };
  auto ask_weights = [&](const WidePlan& w, int ot, int k, uint32_t at) {   // at: the block's number in the ring
    const uint32_t stage = at & 1u, bar = full0 + 8 * stage;
    if (at >= 2 && !mbar_wait(empty0 + 8 * stage, ((at >> 1) - 1) & 1u, &s_abort, a.wait_limit, p.st)) return false;
    mbar_arrive_expect_tx(bar, w.direct ? kSpOperandBytes : kSpStageBytes);
    bulk_load(tiles_addr + stage * kSpStageBytes + kSpOperandBytes, weights_at(w, ot, k), kSpOperandBytes, bar);
    return true;
  };
  auto ask = [&](const WidePlan& w, int pos0, int ot, int k0, int nk, uint32_t early) {
    for (int k = 0; k < nk; ++k) {
      const uint32_t stage = asked & 1u, dst = tiles_addr + stage * kSpStageBytes, bar = full0 + 8 * stage;
      if (k >= (int)early && !ask_weights(w, ot, k0 + k, asked)) return false;
      ++asked;
      if (!w.direct) {
        const int kk = k0 + k, kb = kk < w.skip_first ? kk : kk + w.skip;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < kSpPieces; ++q)
            bulk_load(dst + q * kSpTileBytes + h * kUnitPieceBytes, dz_unit(a.img, pos0 + 64 * h, kb, ju) + q * kUnitPieceBytes,
                      kUnitPieceBytes, bar);
      }
    }
    return true;
  };
  WidePlan w;
  if (n_levels > 0) w = wide_plan(level_begin(n_levels - 1), level_begin(n_levels), n_levels == 1, H, E, grid, a.direct_rows);
  for (int lvl = n_levels - 1; lvl >= 0 && ok; --lvl) {
    TL_STAMP(trace, lvl, 0);
    uint32_t early = 0;                                  // (thread 0)
    if (!w.direct) {
      // What of this CTA's first tile does not depend on the gate gradients: its tables, the weights of two blocks (595 -> 590 us).
      const int lo = blockIdx.x * w.per;
      if (lo < w.total) {
        const int tile = lo / w.span, k0 = lo - tile * w.span, nk = min(min(w.per, w.span - k0), w.kbs - k0);
        if (nk > 0) {
          if (tid == 0)
            while (ok && early < 2u && (int)early < nk) {
              ok = ask_weights(w, tile % w.to, k0 + (int)early, asked + early);
              if (ok) ++early;
            }
          read_tables(w, w.base + tile / w.to * kSpTile);
          tables = true;
        }
      }
      if (vec_h) wide_gates<true>(p, a.img, w);
      else wide_gates<false>(p, a.img, w);
      TL_STAMP(trace, lvl, 1);              // own gate gradients stored
      asm volatile("fence.proxy.async;" ::: "memory");   // the image is read by bulk copies
      if (!(ok = barrier())) {
        asked += early;                                  // (under way)
        break;
      }
      asm volatile("fence.proxy.async;" ::: "memory");
      TL_STAMP(trace, lvl, 2);
    }
    for (int lo = blockIdx.x * w.per; lo < w.total && ok; lo += grid * w.per) {
      for (int at = lo; at < min(lo + w.per, w.total) && ok;) {
        const int tile = at / w.span, k0 = at - tile * w.span, len = min(min(lo + w.per, w.total) - at, w.span - k0);
        const int nk = min(len, w.kbs - k0), ot = tile % w.to, pos0 = w.base + tile / w.to * kSpTile;
        at += len;
        if (nk <= 0) continue;
        if (tid == 0 && !fetched) ok = ask(w, pos0, ot, k0, nk, early);
        if (!fetched && !tables) read_tables(w, pos0);
        tables = false;
        early = 0;
        if (w.direct) {
          if (!fetched) __syncthreads();
          for (int k = 0; k < nk; ++k) {
            unsigned char* dst = tiles + ((blk + k) & 1u) * kSpStageBytes;
            if (vec_h) direct_block<true>(p, a.img, dst, k0 + k, pos0, min(kSpTile, w.end - pos0), ot == 0, s_node, s_da, s_db);
            else direct_block<false>(p, a.img, dst, k0 + k, pos0, min(kSpTile, w.end - pos0), ot == 0, s_node, s_da, s_db);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads these rows
          __syncthreads();
          TL_STAMP(trace, lvl, 7);          // a tile's gate gradients formed
        }
        fetched = false;
        if (warp == 1) {
          const bool issue = elect_one();
          for (int k = 0; k < nk && ok; ++k) {
            const uint32_t b = blk + k, stage = b & 1u, src = tiles_addr + stage * kSpStageBytes;
            ok = __all_sync(kFull, mbar_wait(full0 + 8 * stage, (b >> 1) & 1u, &s_abort, a.wait_limit, p.st));
            if (!ok) break;
            tc_fence_after();
            split_mmas(tmem_base, src, src + kSpOperandBytes, umma_idesc(kSpTile), k == 0, issue);
            if (issue) umma_commit(empty0 + 8 * stage);
            if (issue && k == nk - 1) umma_commit(acc_bar);
          }
        }
        __syncwarp();
        ok = mbar_wait(acc_bar, done & 1u, &s_abort, a.wait_limit, p.st) && ok;
        ++done;
        blk += nk;
        TL_STAMP(trace, lvl, 5);            // a tile accumulated
        if (__syncthreads_or(!ok)) { ok = false; break; }
        tc_fence_after();
        constexpr int kRowStride = kSpTile + 4;
        float* stage_out = reinterpret_cast<float*>(tiles);
        {
          const int quad = warp & 3, quarter = warp >> 2;
          const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(quarter * 32);
          float v[32];
          split_sum(taddr, v);
          tc_fence_before();
          float* dst = stage_out + (size_t)(quad * 32 + lane) * kRowStride + quarter * 32;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<float4*>(dst + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
        __syncthreads();
        TL_STAMP(trace, lvl, 6);            // and read back
        const int K = w.leaf ? E : 2 * H;
        auto out_of = [&](int r, int k) {
          return w.leaf ? p.dEmb_rows + (size_t)s_da[r] * E + k
                        : p.dh + (size_t)(k < H ? s_da[r] : s_db[r]) * H + (k < H ? k : k - H);
        };
        if (w.leaf ? vec_e : vec_h) {
          const int k = ot * 128 + 4 * lane;
          if (k < K)
            for (int r = warp; r < kSpTile; r += kWideThreads / 32)
              if (s_da[r] >= 0)
                atomicAdd(reinterpret_cast<float4*>(out_of(r, k)), *reinterpret_cast<const float4*>(stage_out + (size_t)r * kRowStride + 4 * lane));
        } else {
          for (int r = warp; r < kSpTile; r += kWideThreads / 32) {
            if (s_da[r] < 0) continue;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int c = lane + 32 * i, k = ot * 128 + c;
              if (k < K) atomicAdd(out_of(r, k), stage_out[(size_t)r * kRowStride + c]);
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the next bulk copies overwrite the staging rows
        __syncthreads();
      }
    }
    if (!ok) break;
    const int busy = (w.total + w.per - 1) / w.per;
    if (busy < grid) {
      if ((int)blockIdx.x >= busy && chunks_done + (int)blockIdx.x - busy < chunks) {
        if (lvl > 0) {
          arrived = true;
          __syncthreads();
          if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&p.st->barrier_levels) : "memory");
        }
        input_chunk(chunks_done + blockIdx.x - busy);
      }
      chunks_done += grid - busy;
    }
    if (lvl == 0) break;
    w = wide_plan(level_begin(lvl - 1), level_begin(lvl), lvl == 1, H, E, grid, a.direct_rows);
    if (w.direct) {                                      // what does not depend on the wavefront above, while the barrier is pending
      const int lo = blockIdx.x * w.per;
      if (lo < w.total) {
        const int tile = lo / w.span, k0 = lo - tile * w.span, nk = min(w.per, w.kbs - k0), pos0 = w.base + tile / w.to * kSpTile;
        if (nk > 0) {
          read_tables(w, pos0);
          if (tid == 0) ask(w, pos0, tile % w.to, k0, nk, 0);
          fetched = true;
        }
      }
    }
    TL_STAMP(trace, lvl, 3);
    ok = barrier();
    TL_STAMP(trace, lvl, 4);
  }
  if (ok)
    for (int chunk = chunks_done + (int)blockIdx.x; chunk < chunks; chunk += grid) input_chunk(chunk);
  TL_STAMP(trace, kTraceLevels - 1, 1);
  tc_fence_before();
  if (__syncthreads_or(!ok)) {                           // what was asked for gets a bounded time to land, the MMAs to retire
    if (warp == 1 && elect_one()) { umma_commit(drain_bar); mbar_drain(drain_bar, 0); }
    if (tid == 0)
      for (uint32_t s = 0; s < 2; ++s) {
        const uint32_t times = (asked + 1 - s) / 2;      // how often stage s was filled
        if (times > 0) mbar_drain(full0 + 8 * s, (times - 1) & 1u);
      }
    __syncthreads();
  }
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kSpTmemCols);
  }
}

// What precedes the walk over the trees (trees_fp32.cu), in one cooperative launch: outputs cleared beside the count of every run of
// token ids | classifier, tokens placed; large forests: outputs cleared | leaf tokens marked | tokens counted beside the classifier | tokens
// placed.  Bound by the latency of its grid barriers and of the classifier's chain.  The level table stays on the device.
struct GradSizes { size_t dW, db, dV; };   // floats
constexpr int kBeginMaskWords = 1024;
// Leaf tokens found by the CTA that numbers them rather than flagged in memory: every owner reads the whole forest, two grid barriers and the
// clearing of the flags are saved.  Backward passes, H = 64, 20 000 words, own | flags, us: 106 nodes 105.7 | 110.9, 1.4 k 133.6 | 139.4, 15 k
// 282.5 | 285.5, 30 k 337.8 | 336.8, 60 k 472 | 460; 200 000 words 108 | 117, 136 | 145, 284 | 291, 341 | 345, 475 | 469.
constexpr int kOwnTokensMaxNodes = 20000;
__global__ void __launch_bounds__(256, 2)
k_bwd_begin(BwdParams p, float* dV, GradSizes sizes, const int* level_offset, long long wait_limit, int wide) {
  extern __shared__ float s_cls[];
  __shared__ __align__(16) unsigned int s_mask[kBeginMaskWords];
  __shared__ int s_flag;
  // the kernel behind this one may set itself up: it waits for this grid before it reads dh
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (ld_volatile(&p.st->status) != 0) return;
  const int n_levels = p.st->n_levels, H = p.H, C = p.C;
  p.n_leaves = n_levels > 0 ? level_offset[1] : 0;
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, gthreads = (size_t)gridDim.x * blockDim.x;
  unsigned int arrivals = 0;
  auto barrier = [&]() {
    arrivals += gridDim.x;
    return grid_barrier(p.st, arrivals, wait_limit, &s_flag, true, &p.st->barrier_bwd);
  };
  if (gtid == 0) { *p.loss = 0.f; *p.n_touched = 0; }
  zero_range(p.dW, sizes.dW, gtid, gthreads);
  zero_range(p.db, sizes.db, gtid, gthreads);
  zero_range(dV, sizes.dV, gtid, gthreads);
  zero_range(p.dWc, (size_t)H * C, gtid, gthreads);
  zero_range(p.dbc, (size_t)C, gtid, gthreads);
  const OwnTokens own_tokens(p.vocab);
  const bool own = gridDim.x > 1 && p.n <= kOwnTokensMaxNodes && 4 * (((p.vocab + 127) / 128 + (int)gridDim.x - 1) / (int)gridDim.x) <= kBeginMaskWords;
  if (!own) zero_range(p.tok_slot, (size_t)p.vocab + 1, gtid, gthreads);
  zero_range(p.dEmb_rows, (size_t)p.n_leaves * p.E, gtid, gthreads);
  if (wide) zero_range(p.dc, (size_t)p.n * H, gtid, gthreads);   // k_bwd_wide may follow: dc of the roots
  int* const group_count = p.tok_slot + p.vocab + 4;
  if (own) own_tokens_count(p, own_tokens, s_mask, group_count);
  else if (!barrier()) return;
  for (size_t r = own ? (size_t)p.n_leaves + gtid : gtid; r < (size_t)(wide ? p.n : p.n_leaves); r += gthreads) {
    const int node = chk(p.st, p.order[r], p.n);
    if (r < (size_t)p.n_leaves) {
      p.tok_slot[chk(p.st, p.token[node], p.vocab)] = 1;
    } else {                               // children by position, for k_bwd_wide
      p.pos_left[r] = p.left[node];
      p.pos_right[r] = p.right[node];
    }
  }
  if (own) {                               // the barrier in two halves: by the time the nodes are classified everybody has arrived
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&p.st->barrier_bwd) : "memory");
    if (classifier_groups(p, blockIdx.x, gridDim.x, s_cls, [&]() { return grid_barrier(p.st, gridDim.x, wait_limit, &s_flag, false, &p.st->barrier_bwd); }))
      own_tokens_place(p, own_tokens, s_mask, group_count);
    return;
  }
  if (!barrier()) return;
  if (gridDim.x == 1) {
    scan_tokens(p, s_mask, kBeginMaskWords);
    classifier_groups(p, 0, 1, s_cls, AlreadyCleared{});
  } else {
    scan_count_groups(p, group_count);
    classifier_groups(p, blockIdx.x, gridDim.x, s_cls, AlreadyCleared{});
    if (!barrier()) return;
    scan_place_groups(p, group_count);
  }
}

int launch_bwd_begin(treelstm* ctx, BwdParams& p, float* dV, GradSizes sizes, int wide, cudaStream_t stream) {
  const size_t smem = sizeof(float) * ((size_t)p.H * p.C + p.C + 1);
  if (smem > 160 * 1024 + sizeof(float)) return TREELSTM_ERR_UNSUPPORTED;
  if (smem > 40 * 1024)
    TL_CUDA(ctx, cudaFuncSetAttribute(k_bwd_begin, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TL_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bwd_begin, 256, smem));
  if (per_sm < 1) return TREELSTM_ERR_UNSUPPORTED;
  int grid = ctx->sm_count * (per_sm < 2 ? per_sm : 2);
  if (ctx->opt.max_ctas > 0 && grid > ctx->opt.max_ctas) grid = ctx->opt.max_ctas;
  if (!ctx->bwd_counters_clear)          // (2 us of a training step between its forward and its backward)
    TL_CUDA(ctx, cudaMemsetAsync(&p.st->barrier_bwd, 0, 2 * sizeof(unsigned int), stream));   // and barrier_levels behind it
  ctx->bwd_counters_clear = false;       // until the pass's last kernel is launched
  const int* lvl_off = ctx->last.level_offset;
  long long wait_limit = ctx->opt.wait_limit_kcycles * 1024;
  void* args[] = {&p, &dV, &sizes, &lvl_off, &wait_limit, &wide};
  TL_CUDA(ctx, cudaLaunchCooperativeKernel((void*)k_bwd_begin, dim3(grid), dim3(256), args, smem, stream));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace

static int launch_bwd_persistent(treelstm* ctx, BwdParams& p, size_t cls_smem, int with_dweight, int after_trees, cudaStream_t stream) {
  const size_t smem = ((sizeof(BwdSmem) + 3) / 4) * 4 + cls_smem;
  TL_CUDA(ctx, cudaFuncSetAttribute(k_bwd_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TL_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bwd_persistent, 256, smem));
  if (per_sm < 1) return TREELSTM_ERR_UNSUPPORTED;
  int grid = ctx->sm_count * (per_sm < 2 ? per_sm : 2);
  if (ctx->opt.max_ctas > 0 && grid > ctx->opt.max_ctas) grid = ctx->opt.max_ctas;
  const int* lvl_off = ctx->last.level_offset;
  long long wait_limit = ctx->opt.wait_limit_kcycles * 1024;
  void* args[] = {&p, &lvl_off, &wait_limit, &with_dweight, &after_trees};
  TL_CUDA(ctx, cudaLaunchCooperativeKernel((void*)k_bwd_persistent, dim3(grid), dim3(256), args, smem, stream));
  ctx->launches += 1;
  return TREELSTM_OK;
}

static int launch_bwd_wide(treelstm* ctx, BwdParams& p, const BwdImages& img, int after_trees, cudaStream_t stream) {
  TL_CUDA(ctx, cudaFuncSetAttribute(k_bwd_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSmem));
  int grid = ctx->sm_count;
  if (ctx->opt.max_ctas > 0 && grid > ctx->opt.max_ctas) grid = ctx->opt.max_ctas;
  const bool vec_h = ctx->H % 4 == 0 && ((reinterpret_cast<uintptr_t>(p.h) | reinterpret_cast<uintptr_t>(p.c)) & 15) == 0;
  // (Worked out here, where the sizes and addresses are known; in the kernel it takes the same time.)
  WideArgs a{ctx->last.level_offset, ctx->opt.wait_limit_kcycles * 1024, after_trees, wide_direct_rows(ctx->H, grid, vec_h), img};
  // A grid barrier, so every CTA has to be resident, and the runtime sees to that: a backward pass may run beside other work and
  // other backward passes.  (As a programmatic dependent that comes up while the tree kernel ends it would save 2 us of 200 us,
  // 25 trees in fp32, and of 610, 256 trees in bf16, and end in a timeout where the device is shared.)
  void* args[] = {&p, &a};
  TL_CUDA(ctx, cudaLaunchCooperativeKernel((void*)k_bwd_wide, dim3(grid), dim3(kWideThreads), args, kWideSmem, stream));
  ctx->launches += 1;
  return TREELSTM_OK;
}

int launch_backward(treelstm* ctx, const int32_t* labels, float* loss, float* dW, float* db,
                    float* dWc, float* dbc, int32_t* touched_ids, float* dEmb_rows,
                    int32_t* n_touched, cudaStream_t stream) {
  auto& L = ctx->last;
  L.stream = stream;
  const bool one_launch = !L.host_levels_valid;   // the forward kept the level table on the device
  if (!one_launch) {
    int rc = ensure_host_levels(ctx);
    if (rc != TREELSTM_OK) return rc;
  }
  const int n = L.n, H = ctx->H, E = ctx->E, C = ctx->C, n_levels = one_launch ? 0 : L.n_levels;
  const int32_t* off = ctx->host_level_offset;
  char* base = static_cast<char*>(L.ws);
  BwdParams p;
  p.n = n; p.H = H; p.E = E; p.C = C; p.vocab = ctx->vocab;
  p.n_leaves = n_levels > 0 ? off[1] : 0;
  p.left = L.left; p.right = L.right; p.token = L.token; p.order = L.order; p.labels = labels;
  p.emb = ctx->emb; p.W = ctx->W; p.Wc = ctx->Wc; p.bc = ctx->bc; p.h = L.h; p.c = L.c;
  p.gates = reinterpret_cast<const float*>(base + L.lay.gates);
  p.dh = reinterpret_cast<float*>(base + L.lay.dh);
  p.dc = reinterpret_cast<float*>(base + L.lay.dc);
  p.dz = reinterpret_cast<float*>(base + L.lay.dz);
  p.loss = loss; p.dW = dW; p.db = db; p.dWc = dWc; p.dbc = dbc; p.dEmb_rows = dEmb_rows;
  p.tok_slot = reinterpret_cast<int*>(base + L.lay.tok_slot);
  p.touched_ids = touched_ids; p.n_touched = n_touched;
  p.pos_left = reinterpret_cast<int*>(base + L.lay.parent);      // the scheduler's scratch is free once the forward has run
  p.pos_right = reinterpret_cast<int*>(base + L.lay.order_tmp);
  p.st = reinterpret_cast<DevStatus*>(base + L.lay.status);
  p.trace = nullptr;
#ifdef TREELSTM_TRACE
  p.trace = reinterpret_cast<long long*>(base + L.lay.trace);   // the forward's table: an fp32 forward leaves it unused
  TL_CUDA(ctx, cudaMemsetAsync(p.trace, 0, sizeof(long long) * kTraceSlots * kTraceLevels, stream));
#endif

  const size_t J = 5 * (size_t)H;
  const size_t cls_smem = sizeof(float) * ((size_t)H * C + C + 1);
  if (cls_smem > 160 * 1024 + sizeof(float)) return TREELSTM_ERR_UNSUPPORTED;
  if (one_launch) {
    if (n == 0) {
      TL_CUDA(ctx, cudaMemsetAsync(loss, 0, sizeof(float), stream));
      TL_CUDA(ctx, cudaMemsetAsync(dW, 0, sizeof(float) * (E + 2 * (size_t)H) * J, stream));
      TL_CUDA(ctx, cudaMemsetAsync(db, 0, sizeof(float) * J, stream));
      TL_CUDA(ctx, cudaMemsetAsync(dWc, 0, sizeof(float) * H * C, stream));
      TL_CUDA(ctx, cudaMemsetAsync(dbc, 0, sizeof(float) * C, stream));
      TL_CUDA(ctx, cudaMemsetAsync(n_touched, 0, sizeof(int), stream));
      return TREELSTM_OK;
    }
    const bool trees = trees_take(ctx, n), wide = L.lay.img_dz != L.lay.img_end;
    if (ctx->opt.dw_tensor_cores && (trees || wide)) {
      int rc = launch_bwd_begin(ctx, p, nullptr, {(E + 2 * (size_t)H) * J, J, 0}, wide, stream);
      if (rc == TREELSTM_OK && trees) rc = launch_backward_trees(ctx, stream);
      BwdImages img;
      if (rc == TREELSTM_OK && wide) {
        img.dz = reinterpret_cast<unsigned char*>(base + L.lay.img_dz);
        img.x[0] = reinterpret_cast<unsigned char*>(base + L.lay.img_x0);
        img.x[1] = reinterpret_cast<unsigned char*>(base + L.lay.img_x1);
        img.w = ctx->wsp;
        rc = launch_bwd_wide(ctx, p, img, trees, stream);
      } else if (rc == TREELSTM_OK && !trees_always_pay(0, H, n, true)) {
        rc = launch_bwd_persistent(ctx, p, cls_smem, 0, 1, stream);
      }
      return rc != TREELSTM_OK ? rc : launch_dweight_tc(ctx, n, L.order, L.level_offset, L.token, L.left, L.right, L.h, p.dz, dW, db,
                                                        p.tok_slot, dEmb_rows, p.st, &img, trees, stream);
    }
    TL_CUDA(ctx, cudaMemsetAsync(&p.st->barrier_bwd, 0, sizeof(unsigned int), stream));
    ctx->bwd_counters_clear = false;
    const int with_dweight = ctx->opt.dw_tensor_cores ? 0 : 1;
    const int rc = launch_bwd_persistent(ctx, p, cls_smem, with_dweight, 0, stream);
    if (rc != TREELSTM_OK) return rc;
    if (!with_dweight)
      return launch_dweight_tc(ctx, n, L.order, L.level_offset, L.token, L.left, L.right, L.h, p.dz, dW, db, p.tok_slot,
                               dEmb_rows, p.st, nullptr, false, stream);
    return TREELSTM_OK;
  }
  TL_CUDA(ctx, cudaMemsetAsync(loss, 0, sizeof(float), stream));
  TL_CUDA(ctx, cudaMemsetAsync(dW, 0, sizeof(float) * (E + 2 * (size_t)H) * J, stream));
  TL_CUDA(ctx, cudaMemsetAsync(db, 0, sizeof(float) * J, stream));
  TL_CUDA(ctx, cudaMemsetAsync(dWc, 0, sizeof(float) * H * C, stream));
  TL_CUDA(ctx, cudaMemsetAsync(dbc, 0, sizeof(float) * C, stream));
  TL_CUDA(ctx, cudaMemsetAsync(n_touched, 0, sizeof(int), stream));
  if (n == 0) return TREELSTM_OK;
  TL_CUDA(ctx, cudaMemsetAsync(p.dc, 0, sizeof(float) * (size_t)n * H, stream));
  TL_CUDA(ctx, cudaMemsetAsync(p.tok_slot, 0, sizeof(int) * ((size_t)ctx->vocab + 1), stream));
  TL_CUDA(ctx, cudaMemsetAsync(dEmb_rows, 0, sizeof(float) * (size_t)p.n_leaves * E, stream));

  k_bwd_mark_tokens<<<(p.n_leaves + 255) / 256, 256, 0, stream>>>(p);
  k_bwd_scan_tokens<<<1, 1024, 0, stream>>>(p);
  if (cls_smem > 48 * 1024)
    TL_CUDA(ctx, cudaFuncSetAttribute(k_bwd_classifier, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)cls_smem));
  k_bwd_classifier<<<(n + kClsNodesPerCta - 1) / kClsNodesPerCta, kClsWarps * 32, cls_smem, stream>>>(p);
  ctx->launches += 3;
  for (int lvl = n_levels - 1; lvl >= 0; --lvl) {
    const int begin = off[lvl], end = off[lvl + 1], leaf = lvl == 0 ? 1 : 0;
    const long long elems = (long long)(end - begin) * H;
    k_bwd_gates<<<(unsigned)((elems + 255) / 256), 256, 0, stream>>>(p, begin, end, leaf);
    const int tiles = dinput_tiles(end - begin, leaf ? E : 2 * H), splits = dinput_splits(tiles, (int)J);
    k_bwd_dinput<<<dim3(tiles, splits), 256, 0, stream>>>(p, begin, end, leaf);
    ctx->launches += 2;
  }
  const int tiles_j = (int)((J + BT - 1) / BT);
  for (int part = 0; part < 2; ++part) {
    const int begin = part == 0 ? 0 : p.n_leaves, end = part == 0 ? p.n_leaves : n;
    if (end <= begin) continue;
    const int K = part == 0 ? E : 2 * H;
    const int rows_per_split = kDwRows;
    const int splits = (end - begin + rows_per_split - 1) / rows_per_split;
    dim3 grid(((K + BT - 1) / BT) * tiles_j, splits);
    k_bwd_dweight<<<grid, 256, 0, stream>>>(p, part, begin, end, rows_per_split);
    ctx->launches += 1;
  }
  dim3 gb((unsigned)((J + 127) / 128), (n + 255) / 256);
  k_bwd_dbias<<<gb, 128, 0, stream>>>(p);
  ctx->launches += 1;
  TL_CUDA(ctx, cudaGetLastError());
  return TREELSTM_OK;
}


// ---- TreeRNN / RNTN: backward through structure ------------------------------------------------ //
// Section 4.2.2 for the two other evaluation models of Section 6.1, on the same schedule.  An
// internal node n with x = [h_l ; h_r], p = h_n = tanh(z):
//     dz   = dh_n * (1 - p^2)
//     dW  += x (x) dz,  db += dz,  RNTN: dV_j += dz_j * x (x) x
//     dx   = W dz  (+ RNTN: sum_j dz_j (V_j + V_j^T) x)      -> added to dh of the two children
// a leaf's state is its word vector: dEmb[token] += dh.  Wavefronts in reverse, one launch per phase
// and wavefront; plain fp32, one thread per output element - correct and measured, not tuned.
namespace {

struct RecBwd {
  int n, H, n_leaves, tensor;
  const int *left, *right, *token, *order;
  const float *h, *W, *Vt;     // W [2H][H]; Vt [(a * 2H + b)][j] = V[j][a][b]
  float *dh, *dz;
  float *dW, *db, *dV, *dEmb_rows;
  const int* tok_slot;
  DevStatus* st;
};

__global__ void k_rec_bwd_dz(RecBwd p, int begin, int end) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)(end - begin) * p.H) return;
  const int node = chk(p.st, p.order[begin + (int)(idx / p.H)], p.n), u = (int)(idx % p.H);
  const float hv = p.h[(size_t)node * p.H + u];
  p.dz[(size_t)node * p.H + u] = p.dh[(size_t)node * p.H + u] * (1.f - hv * hv);
}

// one thread per (node of the wavefront, input unit a in [0, 2H)); a child has one caller, so its dh
// is updated without atomics
__global__ void k_rec_bwd_dx(RecBwd p, int begin, int end) {
  const int H = p.H, K = 2 * H;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)(end - begin) * K) return;
  const int node = chk(p.st, p.order[begin + (int)(idx / K)], p.n), a = (int)(idx % K);
  const int l = chk(p.st, p.left[node], p.n), r = chk(p.st, p.right[node], p.n);
  const float* dz = p.dz + (size_t)node * H;
  float acc = 0.f;
  for (int j = 0; j < H; ++j) acc = fmaf(p.W[(size_t)a * H + j], dz[j], acc);
  if (p.tensor) {
    const float* hl = p.h + (size_t)l * H;
    const float* hr = p.h + (size_t)r * H;
    for (int b = 0; b < K; ++b) {
      const float xb = b < H ? hl[b] : hr[b - H];
      const float* vab = p.Vt + ((size_t)a * K + b) * H;
      const float* vba = p.Vt + ((size_t)b * K + a) * H;
      float t = 0.f;
      for (int j = 0; j < H; ++j) t = fmaf(dz[j], vab[j] + vba[j], t);
      acc = fmaf(t, xb, acc);
    }
  }
  const int child = a < H ? l : r;
  p.dh[(size_t)child * H + (a < H ? a : a - H)] += acc;
}

// The wavefronts of a forest that the tree kernel leaves (few large trees), in one cooperative launch behind it and behind
// k_bwd_begin; the gradients are k_rec_grads's either way.  A warp takes one node and kDxUnits of the 2H inputs; its lanes
// share the units of dz and read rows of W (and V) side by side, so that a wavefront is one chain of loads and one grid barrier.
constexpr int kDxUnits = 8, kDxThreads = 256, kDxMaxH = 256;   // (the tree kernels end there)
__global__ void __launch_bounds__(kDxThreads) k_rec_bwd_levels(RecBwd p, const int* level_offset, long long wait_limit) {
  __shared__ int s_flag;
  if (ld_volatile(&p.st->status) != 0 || p.st->trees_bwd) return;
  const int H = p.H, K = 2 * H, lane = threadIdx.x & 31, groups = (K + kDxUnits - 1) / kDxUnits;
  const long long first = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, step = (long long)gridDim.x * (kDxThreads / 32);
  unsigned int arrivals = 0;
  for (int lvl = p.st->n_levels - 1; lvl >= 1; --lvl) {
    const int begin = level_offset[lvl], end = level_offset[lvl + 1];
    for (long long i = first; i < (long long)(end - begin) * groups; i += step) {
      const int node = chk(p.st, p.order[begin + (int)(i / groups)], p.n), a0 = (int)(i % groups) * kDxUnits;
      const int l = chk(p.st, p.left[node], p.n), r = chk(p.st, p.right[node], p.n);
      float dz[kDxMaxH / 32];
#pragma unroll
      for (int t = 0; t < kDxMaxH / 32; ++t) {
        const int j = lane + 32 * t;
        dz[t] = 0.f;
        if (j < H) {
          const float hv = __ldg(p.h + (size_t)node * H + j);
          dz[t] = __ldcg(p.dh + (size_t)node * H + j) * (1.f - hv * hv);
          if (a0 == 0) p.dz[(size_t)node * H + j] = dz[t];
        }
      }
      float acc[kDxUnits];
#pragma unroll
      for (int u = 0; u < kDxUnits; ++u) {
        acc[u] = 0.f;
        const int a = min(a0 + u, K - 1);
#pragma unroll
        for (int t = 0; t < kDxMaxH / 32; ++t)
          if (lane + 32 * t < H) acc[u] = fmaf(__ldg(p.W + (size_t)a * H + lane + 32 * t), dz[t], acc[u]);
        if (p.tensor)
          for (int b = 0; b < K; ++b) {
            const float xb = __ldg(p.h + (size_t)(b < H ? l : r) * H + (b < H ? b : b - H));
#pragma unroll
            for (int t = 0; t < kDxMaxH / 32; ++t) {
              const int j = lane + 32 * t;
              if (j < H) acc[u] = fmaf(xb * dz[t], __ldg(p.Vt + ((size_t)a * K + b) * H + j) + __ldg(p.Vt + ((size_t)b * K + a) * H + j), acc[u]);
            }
          }
      }
#pragma unroll
      for (int u = 0; u < kDxUnits; ++u) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc[u] += __shfl_xor_sync(kFull, acc[u], d);
        const int a = a0 + u;
        if (lane == u && a < K) {                // a child has one caller
          float* at = p.dh + (size_t)(a < H ? l : r) * H + (a < H ? a : a - H);
          *at = __ldcg(at) + acc[u];
        }
      }
    }
    arrivals += gridDim.x;
    if (lvl > 1 && !grid_barrier(p.st, arrivals, wait_limit, &s_flag, true, &p.st->barrier_levels)) return;
  }
}

__global__ void k_rec_bwd_leaves(RecBwd p) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)p.n_leaves * p.H) return;
  const int node = chk(p.st, p.order[(int)(idx / p.H)], p.n), u = (int)(idx % p.H);
  const int row = p.tok_slot[p.token[node]];
  atomicAdd(&p.dEmb_rows[(size_t)row * p.H + u], p.dh[(size_t)node * p.H + u]);
}

// one thread per element of dW [2H][H] (+ db [H] in the threads of row 0): a fixed order of summation
__global__ void k_rec_bwd_dw(RecBwd p) {
  const int H = p.H, K = 2 * H;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= K * H) return;
  const int a = idx / H, j = idx % H;
  float acc = 0.f, accb = 0.f;
  for (int pos = p.n_leaves; pos < p.n; ++pos) {
    const int node = p.order[pos];
    const int child = a < H ? p.left[node] : p.right[node];
    const float dzj = p.dz[(size_t)node * H + j];
    acc = fmaf(p.h[(size_t)child * H + (a < H ? a : a - H)], dzj, acc);
    accb += dzj;
  }
  p.dW[idx] = acc;
  if (a == 0) p.db[j] = accb;
}

// one thread per element of dV [H][2H][2H]
__global__ void k_rec_bwd_dv(RecBwd p) {
  const int H = p.H, K = 2 * H;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)H * K * K) return;
  const int j = (int)(idx / ((long long)K * K)), a = (int)((idx / K) % K), b = (int)(idx % K);
  float acc = 0.f;
  for (int pos = p.n_leaves; pos < p.n; ++pos) {
    const int node = p.order[pos];
    const int l = p.left[node], r = p.right[node];
    const float xa = a < H ? p.h[(size_t)l * H + a] : p.h[(size_t)r * H + a - H];
    const float xb = b < H ? p.h[(size_t)l * H + b] : p.h[(size_t)r * H + b - H];
    acc = fmaf(p.dz[(size_t)node * H + j], xa * xb, acc);
  }
  p.dV[idx] = acc;
}

RecBwd rec_bwd(const treelstm* ctx, const BwdParams& p, float* dW, float* db, float* dV) {
  RecBwd q{};
  const size_t K = 2 * (size_t)p.H;
  q.n = p.n; q.H = p.H; q.n_leaves = p.n_leaves; q.tensor = ctx->cell == TREELSTM_CELL_RNTN ? 1 : 0;
  q.left = p.left; q.right = p.right; q.token = p.token; q.order = p.order;
  q.h = p.h; q.Vt = ctx->Wcat; q.W = ctx->Wcat + (q.tensor ? K * K * p.H : 0);
  q.dh = p.dh; q.dz = p.dz; q.dW = dW; q.db = db; q.dV = dV; q.dEmb_rows = p.dEmb_rows; q.tok_slot = p.tok_slot; q.st = p.st;
  return q;
}

}  // namespace

int launch_backward_rec(treelstm* ctx, const int32_t* labels, float* loss, float* dW, float* db, float* dV,
                        float* dWc, float* dbc, int32_t* touched_ids, float* dEmb_rows, int32_t* n_touched,
                        cudaStream_t stream) {
  auto& L = ctx->last;
  L.stream = stream;
  if (L.n > 0 && !L.host_levels_valid && trees_take(ctx, L.n)) {
    char* base = static_cast<char*>(L.ws);
    BwdParams p{};
    p.n = L.n; p.H = p.E = ctx->H; p.C = ctx->C; p.vocab = ctx->vocab;
    p.left = L.left; p.right = L.right; p.token = L.token; p.order = L.order; p.labels = labels;
    p.Wc = ctx->Wc; p.bc = ctx->bc; p.h = L.h;
    p.dh = reinterpret_cast<float*>(base + L.lay.dh);
    p.dz = reinterpret_cast<float*>(base + L.lay.dz);
    p.loss = loss; p.dW = dW; p.db = db; p.dWc = dWc; p.dbc = dbc; p.dEmb_rows = dEmb_rows;
    p.tok_slot = reinterpret_cast<int*>(base + L.lay.tok_slot);
    p.touched_ids = touched_ids; p.n_touched = n_touched;
    p.st = reinterpret_cast<DevStatus*>(base + L.lay.status);
    const size_t H = ctx->H;
    int rc = launch_bwd_begin(ctx, p, dV, {2 * H * H, H, ctx->cell == TREELSTM_CELL_RNTN ? 4 * H * H * H : 0}, 0, stream);
    if (rc == TREELSTM_OK) rc = launch_backward_trees(ctx, stream);
    if (rc == TREELSTM_OK && !trees_always_pay(ctx->cell, ctx->H, L.n, true)) {
      RecBwd q = rec_bwd(ctx, p, dW, db, dV);
      int per_sm = 0;
      TL_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rec_bwd_levels, kDxThreads, 0));
      if (per_sm < 1) return TREELSTM_ERR_UNSUPPORTED;
      int grid = ctx->sm_count * (per_sm < 2 ? per_sm : 2);
      if (ctx->opt.max_ctas > 0 && grid > ctx->opt.max_ctas) grid = ctx->opt.max_ctas;
      const int* lvl_off = L.level_offset;
      long long wait_limit = ctx->opt.wait_limit_kcycles * 1024;
      void* args[] = {&q, &lvl_off, &wait_limit};
      TL_CUDA(ctx, cudaLaunchCooperativeKernel((void*)k_rec_bwd_levels, dim3(grid), dim3(kDxThreads), args, 0, stream));
      ctx->launches += 1;
    }
    return rc != TREELSTM_OK ? rc : launch_rec_grads(ctx, dW, db, dV, dEmb_rows, p.tok_slot, stream);
  }
  int rc = ensure_host_levels(ctx);      // one read of the level table (a persistent forward left it on the device)
  if (rc != TREELSTM_OK) return rc;
  const int n = L.n, H = ctx->H, C = ctx->C, n_levels = L.n_levels;
  const bool tensor = ctx->cell == TREELSTM_CELL_RNTN;
  const int32_t* off = ctx->host_level_offset;
  const size_t K = 2 * (size_t)H;
  TL_CUDA(ctx, cudaMemsetAsync(loss, 0, sizeof(float), stream));
  TL_CUDA(ctx, cudaMemsetAsync(dW, 0, sizeof(float) * K * H, stream));
  TL_CUDA(ctx, cudaMemsetAsync(db, 0, sizeof(float) * H, stream));
  if (tensor) TL_CUDA(ctx, cudaMemsetAsync(dV, 0, sizeof(float) * H * K * K, stream));
  TL_CUDA(ctx, cudaMemsetAsync(dWc, 0, sizeof(float) * H * C, stream));
  TL_CUDA(ctx, cudaMemsetAsync(dbc, 0, sizeof(float) * C, stream));
  TL_CUDA(ctx, cudaMemsetAsync(n_touched, 0, sizeof(int), stream));
  if (n == 0 || n_levels == 0) return TREELSTM_OK;
  char* base = static_cast<char*>(L.ws);
  const int n_leaves = off[1];
  // the classifier, the loss and the touched-token bookkeeping are the TreeLSTM path's kernels
  BwdParams p{};
  p.n = n; p.H = H; p.E = H; p.C = C; p.vocab = ctx->vocab; p.n_leaves = n_leaves;
  p.left = L.left; p.right = L.right; p.token = L.token; p.order = L.order; p.labels = labels;
  p.Wc = ctx->Wc; p.bc = ctx->bc; p.h = L.h;
  p.dh = reinterpret_cast<float*>(base + L.lay.dh);
  p.dz = reinterpret_cast<float*>(base + L.lay.dz);
  p.loss = loss; p.dWc = dWc; p.dbc = dbc; p.dEmb_rows = dEmb_rows;
  p.tok_slot = reinterpret_cast<int*>(base + L.lay.tok_slot);
  p.touched_ids = touched_ids; p.n_touched = n_touched;
  p.st = reinterpret_cast<DevStatus*>(base + L.lay.status);
  const size_t cls_smem = sizeof(float) * ((size_t)H * C + C + 1);
  if (cls_smem > 160 * 1024 + sizeof(float)) return TREELSTM_ERR_UNSUPPORTED;
  TL_CUDA(ctx, cudaMemsetAsync(p.tok_slot, 0, sizeof(int) * ((size_t)ctx->vocab + 1), stream));
  TL_CUDA(ctx, cudaMemsetAsync(dEmb_rows, 0, sizeof(float) * (size_t)n_leaves * H, stream));
  k_bwd_mark_tokens<<<(n_leaves + 255) / 256, 256, 0, stream>>>(p);
  k_bwd_scan_tokens<<<1, 1024, 0, stream>>>(p);
  if (cls_smem > 48 * 1024)
    TL_CUDA(ctx, cudaFuncSetAttribute(k_bwd_classifier, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cls_smem));
  k_bwd_classifier<<<(n + kClsNodesPerCta - 1) / kClsNodesPerCta, kClsWarps * 32, cls_smem, stream>>>(p);
  ctx->launches += 3;

  const RecBwd q = rec_bwd(ctx, p, dW, db, dV);
  for (int lvl = n_levels - 1; lvl >= 1; --lvl) {
    const int begin = off[lvl], end = off[lvl + 1];
    const long long e1 = (long long)(end - begin) * H, e2 = (long long)(end - begin) * (long long)K;
    k_rec_bwd_dz<<<(unsigned)((e1 + 255) / 256), 256, 0, stream>>>(q, begin, end);
    k_rec_bwd_dx<<<(unsigned)((e2 + 127) / 128), 128, 0, stream>>>(q, begin, end);
    ctx->launches += 2;
  }
  k_rec_bwd_leaves<<<(unsigned)(((long long)n_leaves * H + 255) / 256), 256, 0, stream>>>(q);
  ctx->launches += 1;
  if (n > n_leaves) {
    k_rec_bwd_dw<<<(unsigned)((K * H + 127) / 128), 128, 0, stream>>>(q);
    ctx->launches += 1;
    if (tensor) {
      k_rec_bwd_dv<<<(unsigned)((H * K * K + 127) / 128), 128, 0, stream>>>(q);
      ctx->launches += 1;
    }
  }
  TL_CUDA(ctx, cudaGetLastError());
  return TREELSTM_OK;
}

}  // namespace tl

// TreeRNN and RNTN (Section 6.1), forward and backward through structure, one thread-block cluster per
// group of trees: trees are independent (Section 2.2), so a cluster walks its own trees depth by depth
// with nothing but its own barrier between two depths, and the weights stay in shared memory all the way.
//
// Rows.  A cell is p_j = tanh(sum_r W[r][j] P_r + b_j) over R rows: the K = 2H entries of x = [h_l ; h_r]
// (TreeRNN), behind the K (K + 1) / 2 products x_a x_b, a <= b, of the tensor term (RNTN).  The products
// are symmetric, so the two weights V_j[a][b] and V_j[b][a] are added once at create: half the
// multiply-adds and half the shared memory of the 4H^2-wide form, same sums.
//
// Split.  CTA c of a cluster of cs owns units [c JS, (c + 1) JS) and keeps its R x JS weights resident; cs
// is the smallest power of two up to 8 that makes a slice at most kSliceBytes (a depth of up to NT nodes
// costs one pass over the slice at 128 bytes per cycle, so larger slices would make that pass longer than
// a cluster barrier).  Cluster q takes roots q, q + Q, ... of the forest's ascending list.
//
// Order.  The host-visible schedule (level, order) is the scheduler's; a cluster itself needs only "children
// before parents", and deepest depth first is such an order with the same number of steps.  It finds the
// depths by walking down from its roots over the child arrays in shared memory (one warp, a few dozen
// cycles per depth), so it needs neither sorted sub-forests from the scheduler nor a grid barrier.  All of the
// set-up that does not need the roots (weights, child arrays, the leaves' word vectors) runs while the
// kernel before it on the stream still works.
#include "common.cuh"

namespace tl {
namespace {

constexpr int kT = 512;                   // threads per CTA
constexpr int NT = 4;                     // nodes per pass over the weights
constexpr int kSliceBytes = 100 * 1024;
constexpr int kSmemMax = 225 * 1024;

struct TreeParams {
  int n, H, K, Q, R, JS, SP, vocab;       // Q products, R = Q + K rows, JS units per CTA, SP = JS | 1 words per row
  int* chk_counts;
  const int *left, *right, *token, *roots;
  const float *emb, *W, *b;               // W [R][H]
  float *h, *dh, *dz;
  DevStatus* st;
  long long* trace;                       // cycle stamps of the first CTA (trace builds), else nullptr
};

// Shared memory of a CTA, offsets in 4-byte words.
struct TreeSmem {
  int w, prod, x, red, dz, dx, kids, list, start, words;
};
__host__ __device__ inline TreeSmem tree_smem(int n, int K, int R, int JS, int SP) {
  TreeSmem s{};
  int off = 0;
  auto take = [&](int words) { const int o = off; off += (words + 3) & ~3; return o; };
  s.w = take(R * SP);
  s.prod = take(R * NT);
  s.x = take(K * NT);
  s.red = take(kT * NT);
  s.dz = take(JS * NT);
  s.dx = take(2 * K * NT);
  s.kids = take(n);
  s.list = take(n / 4 + 2);               // uint16 internal nodes of the cluster's trees, root depth first
  s.start = take(n / 4 + 4);              // uint16 first list entry of every depth
  s.words = off;
  return s;
}

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cta_count() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// every thread of the cluster; what any of them wrote before is visible to all of them afterwards
__device__ __forceinline__ void cluster_sync(uint32_t cs) {
  if (cs > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}
__device__ __forceinline__ float ld_peer(uint32_t smem_addr, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// Child table entry of a node: left | right << 16 (ids below 32768), or the top bit and the token of a leaf.
constexpr unsigned kLeafBit = 0x80000000u;
__device__ __forceinline__ bool is_leaf(unsigned kids) { return (kids & kLeafBit) != 0; }

// Weights slice and child table: reads nothing that the kernel ahead on the stream writes.
__device__ __forceinline__ void tree_setup(const TreeParams& p, const TreeSmem& s, float* sm, int j0) {
  const int tid = threadIdx.x;
  const int jn = min(p.JS, p.H - j0);     // units this CTA really has (the last CTA of a cluster may have fewer, or none)
  unsigned* kids = reinterpret_cast<unsigned*>(sm + s.kids);
  for (int k = tid; k < p.n; k += kT) {
    const int l = p.left[k], r = p.right[k], t = p.token[k];
    kids[k] = l < 0 ? kLeafBit | (unsigned)min(max(t, 0), p.vocab - 1) : (unsigned)(l & 0x7FFF) | ((unsigned)(r & 0x7FFF) << 16);
  }
  const int words = p.R * p.SP;
#pragma unroll 8
  for (int e = tid; e < words; e += kT) {
    const int r = e / p.SP, j = e - r * p.SP;
    sm[s.w + e] = j < jn ? __ldg(p.W + (size_t)r * p.H + j0 + j) : 0.f;
  }
}

// The internal nodes of the cluster's trees by depth: list[start[d] .. start[d + 1]).  Returns the number of
// depths.  Warp 0 works (its trees have a few dozen nodes), every thread gets the answer.
__device__ __forceinline__ int tree_depths(const TreeParams& p, const TreeSmem& s, float* sm, int part, int parts, int* s_depths) {
  __syncthreads();                        // the child table is complete
  if (threadIdx.x < 32) {
    const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
    unsigned short* list = reinterpret_cast<unsigned short*>(sm + s.list);
    unsigned short* start = reinterpret_cast<unsigned short*>(sm + s.start);
    const int lane = threadIdx.x, n_roots = p.st->n_roots;
    const unsigned below = (1u << lane) - 1u;
    int count = 0, depth = 0, lo = 0;
    for (int t0 = part; t0 < n_roots; t0 += 32 * parts) {
      const int t = t0 + lane * parts;
      const int node = t < n_roots ? chk(p.st, p.roots[t], p.n) : 0;
      const bool in = t < n_roots && !is_leaf(kids[node]);
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) list[count + __popc(m & below)] = (unsigned short)node;
      count += __popc(m);
    }
    if (lane == 0) start[0] = 0;
    __syncwarp();
    while (lo < count) {
      const int hi = count;
      ++depth;
      if (lane == 0) start[depth] = (unsigned short)hi;
      for (int i0 = lo; i0 < hi; i0 += 32) {
        const bool have = i0 + lane < hi;
        const unsigned kd = have ? kids[list[i0 + lane]] : 0u;
        const int l = (int)(kd & 0xFFFFu), r = (int)(kd >> 16);
        const bool il = have && !is_leaf(kids[l]), ir = have && !is_leaf(kids[r]);
        const unsigned ml = __ballot_sync(0xffffffffu, il), mr = __ballot_sync(0xffffffffu, ir);
        if (il) list[count + __popc(ml & below)] = (unsigned short)l;
        if (ir) list[count + __popc(ml) + __popc(mr & below)] = (unsigned short)r;
        count += __popc(ml) + __popc(mr);
      }
      __syncwarp();
      lo = hi;
    }
    if (lane == 0) *s_depths = depth;
  }
  __syncthreads();
  return *s_depths;
}

// x = [h_l ; h_r] of up to NT nodes, X[k][i] (a leaf's state is its word vector, read from the table itself)
__device__ __forceinline__ void stage_x(const TreeParams& p, const TreeSmem& s, float* sm, int lo, int cnt) {
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
  const unsigned short* list = reinterpret_cast<const unsigned short*>(sm + s.list);
  for (int e = threadIdx.x; e < NT * p.K; e += kT) {
    const int i = e / p.K, k = e - i * p.K;
    float v = 0.f;
    if (i < cnt) {
      const unsigned kd = kids[list[lo + i]];
      const int child = (int)(k < p.H ? kd & 0xFFFFu : kd >> 16), u = k < p.H ? k : k - p.H;
      const unsigned ck = kids[child];
      v = is_leaf(ck) ? __ldg(p.emb + (size_t)(ck & ~kLeafBit) * p.H + u) : __ldcg(p.h + (size_t)child * p.H + u);
    }
    sm[s.x + k * NT + i] = v;
  }
}
// the a and b of product row r (a <= b; row of (a, b) = a K - a (a - 1) / 2 + b - a)
__device__ __forceinline__ int pair_row(int a, int b, int K) { return a * K - ((a * (a - 1)) >> 1) + b - a; }

// ---- forward ------------------------------------------------------------------------------------ //
__global__ void __launch_bounds__(kT, 1) k_rec_trees_forward(TreeParams p) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_depths;
  const uint32_t cs = cta_count(), rank = cta_rank();
  const int tid = threadIdx.x, part = blockIdx.x / cs, parts = gridDim.x / cs, j0 = (int)rank * p.JS;
  const TreeSmem s = tree_smem(p.n, p.K, p.R, p.JS, p.SP);
  const int H = p.H, K = p.K, R = p.R, SP = p.SP;
#ifdef TREELSTM_TRACE
  long long* const trace = blockIdx.x == 0 && threadIdx.x == 0 ? p.trace : nullptr;   // row d: depth d; last row: set-up
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  tree_setup(p, s, sm, j0);
  TL_STAMP(trace, kTraceLevels - 1, 1);
  // the leaves' states, a warp per node (tokens are clamped: nothing has been validated yet)
  {
    const int lane = tid & 31, warps = gridDim.x * (kT / 32);
    for (int k = blockIdx.x * (kT / 32) + (tid >> 5); k < p.n; k += warps)
      if (p.left[k] < 0) {
        const float* src = p.emb + (size_t)min(max(p.token[k], 0), p.vocab - 1) * H;
        for (int u = lane; u < H; u += 32) {
          p.h[(size_t)k * H + u] = __ldg(src + u);
          count_write(p.chk_counts, k, 1);
        }
      }
  }
  TL_STAMP(trace, kTraceLevels - 1, 2);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  TL_STAMP(trace, kTraceLevels - 1, 3);
  if (ld_volatile(&p.st->status) != 0) return;          // the same answer in every CTA
  const int depths = tree_depths(p, s, sm, part, parts, &s_depths);
  TL_STAMP(trace, kTraceLevels - 1, 4);
  const unsigned short* list = reinterpret_cast<const unsigned short*>(sm + s.list);
  const unsigned short* start = reinterpret_cast<const unsigned short*>(sm + s.start);
  const float4* prod = reinterpret_cast<const float4*>(sm + (p.Q ? s.prod : s.x));
  float4* red = reinterpret_cast<float4*>(sm + s.red);
  const int nseg = kT / SP, seg = tid / SP;   // thread: unit tid % SP, rows seg, seg + nseg, ...: consecutive words of W
  for (int d = depths - 1; d >= 0; --d) {
    for (int lo = start[d], hi = start[d + 1]; lo < hi; lo += NT) {
      const int cnt = min(NT, hi - lo);
      TL_STAMP(trace, d, 0);
      stage_x(p, s, sm, lo, cnt);
      __syncthreads();
      TL_STAMP(trace, d, 1);
      if (p.Q) {
        const float4* x = reinterpret_cast<const float4*>(sm + s.x);
        float4* out = reinterpret_cast<float4*>(sm + s.prod);
        // warp w takes a = w, w + 16, ...: the rows of an a lie side by side
        for (int a = tid >> 5; a < K; a += kT / 32) {
          const float4 xa = x[a];
          for (int b = a + (tid & 31); b < K; b += 32) {
            const float4 xb = x[b];
            out[pair_row(a, b, K)] = make_float4(xa.x * xb.x, xa.y * xb.y, xa.z * xb.z, xa.w * xb.w);
          }
        }
        for (int k = tid; k < K; k += kT) out[p.Q + k] = x[k];
        __syncthreads();
      }
      TL_STAMP(trace, d, 2);
      if (seg < nseg) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        const float* w = sm + s.w + tid;
#pragma unroll 8
        for (int r = seg; r < R; r += nseg, w += nseg * SP) {
          const float4 x = prod[r];
          const float wv = *w;
          acc.x = fmaf(x.x, wv, acc.x); acc.y = fmaf(x.y, wv, acc.y);
          acc.z = fmaf(x.z, wv, acc.z); acc.w = fmaf(x.w, wv, acc.w);
        }
        red[tid] = acc;
      }
      __syncthreads();
      TL_STAMP(trace, d, 3);
      for (int o = tid; o < p.JS * NT; o += kT) {
        const int u = o % p.JS, i = o / p.JS;
        if (i < cnt && j0 + u < H) {
          float z = __ldg(p.b + j0 + u);
#pragma unroll 4
          for (int g = 0; g < nseg; ++g) z += sm[s.red + (g * SP + u) * NT + i];
          const int node = list[lo + i];
          p.h[(size_t)node * H + j0 + u] = tanhf(z);
          count_write(p.chk_counts, node, 1);
        }
      }
    }
    TL_STAMP(trace, d, 4);
    cluster_sync(cs);
    TL_STAMP(trace, d, 5);
  }
}

// ---- backward: dz of every internal node, dh of every leaf -------------------------------------- //
// dz = dh (1 - p^2);  M_r = sum_j W[r][j] dz_j over the CTA's own units;  dx_a = M_lin[a] + sum_b M_ab x_b
// (twice that for a = b: V_j[a][a] multiplies a square);  the CTAs' dx are summed by the owner of the unit
// through distributed shared memory and added to dh of the child (which has no other caller).
__global__ void __launch_bounds__(kT, 1) k_rec_trees_backward(TreeParams p) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_depths;
  const uint32_t cs = cta_count(), rank = cta_rank();
  const int tid = threadIdx.x, part = blockIdx.x / cs, parts = gridDim.x / cs, j0 = (int)rank * p.JS;
  const TreeSmem s = tree_smem(p.n, p.K, p.R, p.JS, p.SP);
  const int H = p.H, K = p.K, R = p.R, SP = p.SP, JS = p.JS, jn = max(0, min(JS, H - j0));
#ifdef TREELSTM_TRACE
  long long* const trace = blockIdx.x == 0 && threadIdx.x == 0 ? p.trace : nullptr;   // row d: depth d; last row: set-up
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  tree_setup(p, s, sm, j0);
  TL_STAMP(trace, kTraceLevels - 1, 1);
  // the forward is over (it ended before the kernel ahead of this one began), so its roots can be read already
  const bool bad = ld_volatile(&p.st->status) != 0;
  const int depths = bad ? 0 : tree_depths(p, s, sm, part, parts, &s_depths);
  TL_STAMP(trace, kTraceLevels - 1, 2);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  TL_STAMP(trace, kTraceLevels - 1, 3);
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
  const unsigned short* list = reinterpret_cast<const unsigned short*>(sm + s.list);
  const unsigned short* start = reinterpret_cast<const unsigned short*>(sm + s.start);
  float4* red = reinterpret_cast<float4*>(sm + s.red);
  const float4* dz4 = reinterpret_cast<const float4*>(sm + s.dz);
  int turn = 0;
  for (int d = 0; d < depths; ++d) {
    for (int lo = start[d], hi = start[d + 1]; lo < hi; lo += NT, turn ^= 1) {
      const int cnt = min(NT, hi - lo);
      TL_STAMP(trace, d, 0);
      float* dx = sm + s.dx + turn * K * NT;            // two in turn: peers may still read the last one
      for (int e = tid; e < NT * JS; e += kT) {
        const int i = e / JS, u = e - i * JS;
        float v = 0.f;
        if (i < cnt && u < jn) {
          const size_t at = (size_t)list[lo + i] * H + j0 + u;
          const float hv = __ldcg(p.h + at);
          v = __ldcg(p.dh + at) * (1.f - hv * hv);
          p.dz[at] = v;
        }
        sm[s.dz + u * NT + i] = v;
      }
      if (p.Q) stage_x(p, s, sm, lo, cnt);
      __syncthreads();
      TL_STAMP(trace, d, 1);
      // M: thread per row, all of the CTA's units (fewer rows than threads: the units are split over groups of threads)
      const int groups = R < kT ? kT / R : 1;
      const int g = R < kT ? tid / R : 0;
      for (int r = R < kT ? tid - g * R : tid; r < R && g < groups; r += kT) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        const float* w = sm + s.w + r * SP;
#pragma unroll 8
        for (int u = g; u < jn; u += groups) {
          const float4 x = dz4[u];
          const float wv = w[u];
          acc.x = fmaf(x.x, wv, acc.x); acc.y = fmaf(x.y, wv, acc.y);
          acc.z = fmaf(x.z, wv, acc.z); acc.w = fmaf(x.w, wv, acc.w);
        }
        if (groups > 1) red[g * R + r] = acc;
        else reinterpret_cast<float4*>(sm + s.prod)[r] = acc;
      }
      __syncthreads();
      TL_STAMP(trace, d, 2);
      if (groups > 1 && !p.Q) {                          // TreeRNN: M is dx
        for (int r = tid; r < R; r += kT) {
          float4 v = red[r];
          for (int q = 1; q < groups; ++q) {
            const float4 t = red[q * R + r];
            v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
          }
          reinterpret_cast<float4*>(dx)[r] = v;
        }
      } else if (!p.Q) {
        for (int r = tid; r < R; r += kT) reinterpret_cast<float4*>(dx)[r] = reinterpret_cast<const float4*>(sm + s.prod)[r];
      } else {
        if (groups > 1) {
          for (int r = tid; r < R; r += kT) {
            float4 v = red[r];
            for (int q = 1; q < groups; ++q) {
              const float4 t = red[q * R + r];
              v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
            }
            reinterpret_cast<float4*>(sm + s.prod)[r] = v;
          }
          __syncthreads();
        }
        const float4* m4 = reinterpret_cast<const float4*>(sm + s.prod);
        const float4* x4 = reinterpret_cast<const float4*>(sm + s.x);
        const int nb = kT / K, bs = tid / K, a = tid - bs * K;   // K <= 256: at least two groups of threads share the b
        if (bs < nb) {
          float4 acc = bs == 0 ? m4[p.Q + a] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
          for (int b = bs; b < K; b += nb) {
            const float4 m = m4[a <= b ? pair_row(a, b, K) : pair_row(b, a, K)], x = x4[b];
            const float f = a == b ? 2.f : 1.f;
            acc.x = fmaf(m.x * f, x.x, acc.x); acc.y = fmaf(m.y * f, x.y, acc.y);
            acc.z = fmaf(m.z * f, x.z, acc.z); acc.w = fmaf(m.w * f, x.w, acc.w);
          }
          red[bs * K + a] = acc;
        }
        __syncthreads();
        for (int r = tid; r < K; r += kT) {
          float4 v = red[r];
          for (int q = 1; q < nb; ++q) {
            const float4 t = red[q * K + r];
            v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
          }
          reinterpret_cast<float4*>(dx)[r] = v;
        }
      }
      TL_STAMP(trace, d, 3);
      cluster_sync(cs);
      TL_STAMP(trace, d, 4);
      const uint32_t dx_addr = (uint32_t)__cvta_generic_to_shared(dx);
      for (int e = tid; e < NT * 2 * JS; e += kT) {
        const int i = e / (2 * JS), q = e - i * 2 * JS, side = q / JS, u = q - side * JS;
        if (i < cnt && u < jn) {
          const int a = side * H + j0 + u;
          float v = 0.f;
          if (cs == 1) v = dx[a * NT + i];
          else
            for (uint32_t c = 0; c < cs; ++c) v += ld_peer(dx_addr + (uint32_t)(a * NT + i) * 4u, c);
          const unsigned kd = kids[list[lo + i]];
          float* at = p.dh + (size_t)(side ? kd >> 16 : kd & 0xFFFFu) * H + j0 + u;
          *at = __ldcg(at) + v;
        }
      }
    }
    TL_STAMP(trace, d, 5);
    __syncthreads();                                     // dh of the next depth (this CTA's units) is complete
  }
  cluster_sync(cs);                                      // no CTA leaves while a peer may still read its dx
}

// ---- dW, db, dV and the embedding rows ------------------------------------------------------------ //
// One tile of gradient rows (32 of the R rows) x 32 units per CTA and run of nodes: sum over the internal
// nodes of P_r dz_j.  A product row's sum belongs to V_j[a][b] and V_j[b][a] alike.  The runs are as long
// as two CTAs per SM allow, because every run ends in one atomic add per element.  CTAs behind the tiles
// add dh of the leaves to the rows of their tokens.
constexpr int GR = 32, GU = 32, GN = 64, kGT = 256;
struct GradParams {
  int n, H, K, Q, R, tiles_u, tiles, splits, vocab;
  const int *left, *right, *token, *order, *level_offset, *tok_slot;
  const float *h, *dh, *dz;
  float *dW, *db, *dV, *dEmb_rows;
  DevStatus* st;
};
__global__ void __launch_bounds__(kGT) k_rec_grads(GradParams p) {
  __shared__ float As[GN][GR];
  __shared__ __align__(16) float Ds[GN][GU];
  __shared__ int s_node[GN], s_l[GN], s_r[GN];
  __shared__ int s_a[GR], s_b[GR];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, H = p.H, K = p.K;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (p.st->n_levels < 1 || (ld_volatile(&p.st->status) != 0 && ld_volatile(&p.st->status) != TREELSTM_ERR_LABEL_OUT_OF_RANGE)) return;
  const int n_leaves = p.level_offset[1];
  const int grad_ctas = p.tiles * p.splits;
  if ((int)blockIdx.x >= grad_ctas) {
    const int warps = ((int)gridDim.x - grad_ctas) * (kGT / 32);
    for (int q = ((int)blockIdx.x - grad_ctas) * (kGT / 32) + warp; q < n_leaves; q += warps) {
      const int node = chk(p.st, p.order[q], p.n);
      const int row = p.tok_slot[chk(p.st, p.token[node], p.vocab)];
      for (int u = lane; u < H; u += 32) atomicAdd(p.dEmb_rows + (size_t)row * H + u, __ldg(p.dh + (size_t)node * H + u));
    }
    return;
  }
  const int tile = (int)blockIdx.x % p.tiles, split = (int)blockIdx.x / p.tiles;
  const int r0 = (tile / p.tiles_u) * GR, u0 = (tile % p.tiles_u) * GU;
  const int internal = p.n - n_leaves, per = (internal + p.splits - 1) / p.splits;
  const int q_lo = n_leaves + split * per, q_hi = min(p.n, q_lo + per);
  if (tid < GR) {                          // the two entries of x behind a row (b < 0: a linear row)
    int r = r0 + tid, a = -1, b = -1;
    if (r < p.Q) {
      a = 0;
      while (r >= K - a) { r -= K - a; ++a; }
      b = a + r;
    } else if (r < p.R) {
      a = r - p.Q;
    }
    s_a[tid] = a; s_b[tid] = b;
  }
  float acc[4] = {}, accb[4] = {};
  for (int q0 = q_lo; q0 < q_hi; q0 += GN) {
    __syncthreads();
    if (tid < GN) {
      const int node = chk(p.st, p.order[min(q0 + tid, q_hi - 1)], p.n);
      s_node[tid] = node; s_l[tid] = chk(p.st, p.left[node], p.n); s_r[tid] = chk(p.st, p.right[node], p.n);
    }
    __syncthreads();
    const int a = s_a[lane], b = s_b[lane];
    float va[GN / 8], vb[GN / 8], vd[GN / 8];
#pragma unroll
    for (int e = 0; e < GN / 8; ++e) {     // loads first
      const int i = warp + 8 * e;
      const int aa = max(a, 0), bb = max(b, 0);
      va[e] = __ldg(p.h + (size_t)(aa < H ? s_l[i] : s_r[i]) * H + (aa < H ? aa : aa - H));
      vb[e] = p.Q ? __ldg(p.h + (size_t)(bb < H ? s_l[i] : s_r[i]) * H + (bb < H ? bb : bb - H)) : 1.f;
      vd[e] = __ldg(p.dz + (size_t)s_node[i] * H + min(u0 + lane, H - 1));
    }
#pragma unroll
    for (int e = 0; e < GN / 8; ++e) {
      const int i = warp + 8 * e;
      const bool in = q0 + i < q_hi;
      As[i][lane] = in && a >= 0 ? (b >= 0 ? va[e] * vb[e] : va[e]) : 0.f;
      Ds[i][lane] = in && u0 + lane < H ? vd[e] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int i = 0; i < GN; ++i) {         // thread: row `lane`, units 4 warp .. 4 warp + 3
      const float x = As[i][lane];
      const float4 d = *reinterpret_cast<const float4*>(&Ds[i][4 * warp]);
      acc[0] = fmaf(x, d.x, acc[0]); acc[1] = fmaf(x, d.y, acc[1]);
      acc[2] = fmaf(x, d.z, acc[2]); acc[3] = fmaf(x, d.w, acc[3]);
      accb[0] += d.x; accb[1] += d.y; accb[2] += d.z; accb[3] += d.w;
    }
  }
  if (q_lo >= q_hi) return;
  const int a = s_a[lane], b = s_b[lane];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int u = u0 + 4 * warp + q;
    if (u >= H || a < 0) continue;
    if (b < 0) {
      atomicAdd(p.dW + (size_t)a * H + u, acc[q]);
      if (a == 0) atomicAdd(p.db + u, accb[q]);
    } else {
      float* v = p.dV + (size_t)u * K * K;
      atomicAdd(v + (size_t)a * K + b, acc[q]);
      if (a != b) atomicAdd(v + (size_t)b * K + a, acc[q]);
    }
  }
}

// W of the tree kernels from Wcat (the 4H^2 + 2H rows of the level kernels): symmetric products added up.
__global__ void k_rec_pack_trees(int H, int K, int Q, const float* Wcat, float* out) {
  const int total = (Q + K) * H;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int r = i / H, j = i - r * H;
    float v;
    if (r < Q) {
      int a = 0, q = r;
      while (q >= K - a) { q -= K - a; ++a; }
      const int b = a + q;
      v = Wcat[((size_t)a * K + b) * H + j];
      if (a != b) v += Wcat[((size_t)b * K + a) * H + j];
    } else {
      v = Wcat[((size_t)K * K + r - Q) * H + j];
    }
    out[i] = v;
  }
}

TreeParams tree_params(treelstm* ctx, int n, const int32_t* left, const int32_t* right, const int32_t* token,
                       float* h, void* ws, const WsLayout& lay) {
  char* base = static_cast<char*>(ws);
  const auto& t = ctx->rt;
  TreeParams p{};
  p.n = n; p.H = ctx->H; p.K = 2 * ctx->H; p.Q = t.Q; p.R = t.R; p.JS = t.JS; p.SP = t.SP; p.vocab = ctx->vocab;
  p.chk_counts = check_counters(ws, lay);
  p.left = left; p.right = right; p.token = token;
  p.roots = reinterpret_cast<const int*>(base + lay.roots);
  p.emb = ctx->emb; p.W = t.W ? t.W : ctx->Wcat; p.b = ctx->b;
  p.h = h;
  p.dh = reinterpret_cast<float*>(base + lay.dh);
  p.dz = reinterpret_cast<float*>(base + lay.dz);
  p.st = reinterpret_cast<DevStatus*>(base + lay.status);
  p.trace = nullptr;
#ifdef TREELSTM_TRACE
  p.trace = reinterpret_cast<long long*>(base + lay.trace);   // forward: first table, backward: second
#endif
  return p;
}

// The clusters do not wait for one another: any number may be resident at a time.
int launch_trees(treelstm* ctx, void (*kernel)(TreeParams), const TreeParams& p, bool after_running, cudaStream_t stream) {
  const auto& t = ctx->rt;
  const size_t smem = 4 * (size_t)tree_smem(p.n, p.K, p.R, p.JS, p.SP).words;
  int ctas = after_running ? ctx->sm_count - 1 : ctx->sm_count;   // the single-CTA scheduler keeps its SM
  if (ctx->opt.max_ctas > 0 && ctas > ctx->opt.max_ctas) ctas = ctx->opt.max_ctas;
  int clusters = ctas / t.cs;
  const int most = (p.n + 2) / 3;                        // trees with something to do have three nodes at least
  if (clusters > most) clusters = most;
  if (clusters < 1) clusters = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * t.cs); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = t.cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = after_running ? 1 : 0;
  cfg.attrs = at; cfg.numAttrs = 2;
  TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, kernel, p));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace

int init_rec_trees(treelstm* ctx, cudaStream_t stream) {
  auto& t = ctx->rt;
  const int H = ctx->H, K = 2 * H;
  t.Q = ctx->cell == TREELSTM_CELL_RNTN ? K * (K + 1) / 2 : 0;
  t.R = t.Q + K;
  t.ok = false;
  if (K > kT / (t.Q ? 2 : 1)) return TREELSTM_OK;        // a thread per entry of x (RNTN: at least two)
  for (t.cs = 1; t.cs <= 8; t.cs *= 2) {
    t.JS = (H + t.cs - 1) / t.cs;
    t.SP = t.JS | 1;
    if (4ll * t.R * t.SP <= kSliceBytes) break;
  }
  if (t.cs > 8) return TREELSTM_OK;                      // the level kernels stream the weights instead
  // what is left of shared memory bounds the forest: 4 bytes of child table and 2 of lists per node
  const long long rest = kSmemMax - 4ll * tree_smem(0, K, t.R, t.JS, t.SP).words - 64;
  t.max_nodes = (int)(rest / 6 < 32767 ? rest / 6 : 32767);
  if (rest <= 0 || t.max_nodes < 64) return TREELSTM_OK;
  TL_CUDA(ctx, cudaFuncSetAttribute(k_rec_trees_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
  TL_CUDA(ctx, cudaFuncSetAttribute(k_rec_trees_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
  if (t.Q) {
    TL_CUDA(ctx, cudaMalloc((void**)&t.W, sizeof(float) * (size_t)t.R * H));
    k_rec_pack_trees<<<296, 256, 0, stream>>>(H, K, t.Q, ctx->Wcat, t.W);
    TL_CUDA(ctx, cudaGetLastError());
  }
  t.ok = true;
  return TREELSTM_OK;
}

int launch_forward_rec_trees(treelstm* ctx, int n, const int32_t* left, const int32_t* right, const int32_t* token,
                             float* h, void* ws, const WsLayout& lay, bool after_running, cudaStream_t stream) {
  return launch_trees(ctx, k_rec_trees_forward, tree_params(ctx, n, left, right, token, h, ws, lay), after_running, stream);
}

int launch_backward_rec_trees(treelstm* ctx, float* dW, float* db, float* dV, float* dEmb_rows, const int* tok_slot,
                              cudaStream_t stream) {
  const auto& L = ctx->last;
  const auto& t = ctx->rt;
  TreeParams p = tree_params(ctx, L.n, L.left, L.right, L.token, L.h, L.ws, L.lay);
  if (p.trace) p.trace += kTraceSlots * kTraceLevels;
  int rc = launch_trees(ctx, k_rec_trees_backward, p, true, stream);
  if (rc != TREELSTM_OK) return rc;
  GradParams g{};
  g.n = L.n; g.H = ctx->H; g.K = p.K; g.Q = t.Q; g.R = t.R; g.vocab = ctx->vocab;
  g.left = L.left; g.right = L.right; g.token = L.token; g.order = L.order; g.level_offset = L.level_offset;
  g.tok_slot = tok_slot; g.h = L.h; g.dh = p.dh; g.dz = p.dz;
  g.dW = dW; g.db = db; g.dV = dV; g.dEmb_rows = dEmb_rows; g.st = p.st;
  g.tiles_u = (ctx->H + GU - 1) / GU;
  g.tiles = ((t.R + GR - 1) / GR) * g.tiles_u;
  const int most = (L.n / 2 + GN - 1) / GN;               // runs of at least one chunk
  g.splits = 2 * ctx->sm_count / g.tiles;
  if (g.splits > most) g.splits = most;
  if (g.splits < 1) g.splits = 1;
  const int leaf_ctas = L.n / 16 < 64 ? L.n / 16 + 1 : 64;
  k_rec_grads<<<g.tiles * g.splits + leaf_ctas, kGT, 0, stream>>>(g);
  TL_CUDA(ctx, cudaGetLastError());
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace tl

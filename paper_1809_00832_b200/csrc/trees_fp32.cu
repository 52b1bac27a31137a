// fp32 evaluation and backpropagation of all three cells (TreeLSTM, TreeRNN, RNTN), one thread-block cluster
// per group of trees, with the recurrent weights held in REGISTERS.
//
// Trees are independent (Section 2.2), so a cluster walks its own trees depth by depth and waits for nobody
// else.  A depth is then a handful of matrix-vector products, and its cost is a chain: weights to the
// multipliers, sum over the inputs, activation, state to whoever reads it, barrier.
//   - Weights.  From shared memory the 32 k weights of a TreeRNN with H = 128 take 1 k cycles per pass (2.1 k
//     measured); the register files of the cluster hold them all.
//   - Product.  A thread holds U outputs x a few inputs.  Shared memory gives a thread one word per lane and cycle,
//     broadcast or not, so U decides: with one output per thread a TreeRNN node costs 1.1 k cycles and a TreeLSTM node
//     (H = 150, eight CTAs) 1.65 k, all of it operand reads; the price of a large U is partial sums per output
//     (512 U / outputs).  Four or five outputs balance the two.  (A warp per unit with shuffles instead of partial
//     sums needs no CTA barrier, but every warp then issues the activations of a few values: 2.6 k cycles.)
//   - State.  A node has one caller, so its h is stored straight into the caller's operand row [h_l | h_r] in the
//     shared memory of every CTA of the cluster (distributed shared memory); the cell state stays with the unit's
//     owner.  If the rows of the cluster's trees do not fit, states go through L2.
//
// Split.  CTA r of a cluster of cs owns hidden units [r JS, (r + 1) JS); cs is the smallest power of two whose
// slice fits the registers of one CTA.  Backward is the same product with inputs (the CTA's own gate gradients) and
// outputs (the 2H units of the children) exchanged; partial sums go straight to the unit's owner, who adds them.
//
// Order.  The schedule that callers see (level, order) is the scheduler's.  A cluster needs only "children
// before parents"; deepest depth first is such an order with the same number of steps.  It finds roots and depths
// itself, from the child arrays in shared memory (trees_plan.cuh), so nothing here waits for the scheduler before its end
// (TreeLSTM waits for the leaves' kernel).  Forests that are faster wavefront by wavefront are left to the kernel behind
// (clusters_win).  (A malformed forest is the scheduler's to report; here every index is clamped and every list bounded, so
// that whatever the arrays hold the walk ends.)
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "split_tc.cuh"
#include "trees_plan.cuh"

namespace tl {
namespace {

constexpr int NT = 4;                     // nodes that are multiplied side by side in the forward
// Nodes per pass.  A pass ends with sums, activations, stores to the callers' rows and a barrier, 1.2 k cycles whatever their number; RNTN, whose
// pass has few of them, takes eight (25 sentences, H = 32, training step 163.9 -> 161.4 us; TreeRNN, H = 128, 116.2 -> 121).
__host__ __device__ constexpr int pass_nodes(int cell) { return cell == TREELSTM_CELL_RNTN ? 2 * NT : NT; }
constexpr int kFwdT = 512, kBwdT = 640;   // threads of a CTA (backward: at most)
constexpr int kLstm = 0, kRnn = TREELSTM_CELL_TREERNN, kRntn = TREELSTM_CELL_RNTN;
constexpr int kND = 16;                   // backward: nodes between two cluster barriers at most
constexpr int kRntnBC = 2, kRntnJS = 8, kRntnMaxH = 32, kRntnT = 512;   // RNTN backward: columns and units per thread
constexpr int kRntnBwdWords = 4 * kRntnBC * kRntnJS + kRntnJS;

__device__ __forceinline__ float sigmoid_acc(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// every thread of the cluster; what any of them wrote before its arrival is visible to all of them behind the wait
__device__ __forceinline__ void cluster_arrive(int cs) {
  if (cs > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait(int cs) {
  if (cs > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  else __syncthreads();
}
__device__ __forceinline__ void cluster_sync(int cs) {
  cluster_arrive(cs);
  cluster_wait(cs);
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t smem_addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// A row of n floats to shared memory, by one warp, in pieces of 1, 2 or 4 of them (both ends aligned to a piece, n a multiple); waits for nothing.
__device__ __forceinline__ void copy_row(uint32_t dst, const float* src, int n, int piece, int lane) {
  if (piece == 4)
    for (int k = 4 * lane; k < n; k += 128) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 4u * k), "l"(src + k) : "memory");
  else if (piece == 2)
    for (int k = 2 * lane; k < n; k += 64) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 4u * k), "l"(src + k) : "memory");
  else
    for (int k = lane; k < n; k += 32) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * k), "l"(src + k) : "memory");
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Four sums over each group of LANES lanes: v[0] of a lane becomes the sum of value value_of_lane(lane) - every
// exchange halves the values a lane still carries.
template <int LANES>
__device__ __forceinline__ void lane_sums4(float (&v)[4], int lane) {
  const bool up = (lane & (LANES / 2)) != 0, up2 = (lane & (LANES / 4)) != 0;
  const float s0 = up ? v[0] : v[2], s1 = up ? v[1] : v[3];
  v[0] = (up ? v[2] : v[0]) + __shfl_xor_sync(kFull, s0, LANES / 2);
  v[1] = (up ? v[3] : v[1]) + __shfl_xor_sync(kFull, s1, LANES / 2);
  const float s2 = up2 ? v[0] : v[1];
  v[0] = (up2 ? v[1] : v[0]) + __shfl_xor_sync(kFull, s2, LANES / 4);
#pragma unroll
  for (int d = LANES / 8; d > 0; d /= 2) v[0] += __shfl_xor_sync(kFull, v[0], d);
}
template <int LANES>
__device__ __forceinline__ int value_of_lane(int lane) { return ((lane & (LANES / 2)) ? 2 : 0) + ((lane & (LANES / 4)) ? 1 : 0); }

struct TreesParams : ForestIn {
  int H, E;
  int Hp;                                 // H rounded up to 4: half an operand row in shared memory
  TreesShape s;
  int* chk_counts;
  const float *emb, *W, *b;               // W: register image [rank][word][thread]; b [G H]
  const ushort2* pairs;                   // RNTN: the two operands of every input chunk
  WalkCosts costs;
  int choose;                             // 1: the forest may be left to the kernel behind this one (clusters_win)
  float *h, *c, *gates, *dh, *dc, *dz;
  SavedWalks walks;                       // of the forward pass, for the backward one (at == nullptr: none)
  DevStatus* st;
  long long* trace;                       // cycle stamps of the first CTA (trace builds), else nullptr
};

// ---- which weight a thread holds where (host and device; the register images are packed once) ------- //
struct WeightAt { long long i0, i1; };    // index into the fp32 weights, -1: padding; i1 >= 0: a second one is added
__host__ __device__ inline int real_input(int padded, int H, int Hp) {   // entry of [h_l | h_r] behind a padded one, -1: padding
  const int side = padded >= Hp, k = padded - side * Hp;
  return k < H ? side * H + k : -1;
}
// Forward word (c * 4 + i) * U + u of a thread (lane group t % JL, segment t / JL): input i of the segment's chunk c,
// output u: the unit's gate u (TreeLSTM), unit u JL + lane (the others).
__host__ __device__ inline WeightAt fwd_weight(int cell, int H, int E, const TreesShape& s, int rank, int t, int w, const ushort2* pairs) {
  const WeightAt none{-1, -1};
  const int Hp = (H + 3) & ~3, u = w % s.U, i = (w / s.U) % 4, c = w / (4 * s.U), lane = t % s.JL, seg = t / s.JL;
  // RNTN segments interleave their chunks (the rows of one operand pair lie side by side), the others take runs
  const int ch = cell == kRntn ? seg + s.nseg * c : seg * s.nc + c;
  if (seg >= s.nseg || ch >= s.chunks) return none;
  const int unit = cell == kLstm ? lane : u * s.JL + lane, gate = cell == kLstm ? u : 0;
  const int j = rank * s.JS + unit;
  if (unit >= s.JS || j >= H || gate > 4) return none;
  if (cell != kRntn) {
    const int r = real_input(4 * ch + i, H, Hp);
    if (r < 0) return none;
    return cell == kLstm ? WeightAt{((long long)E + r) * 5 * H + (long long)gate * H + j, -1} : WeightAt{(long long)r * H + j, -1};
  }
  const int K = 2 * H, bp = pairs[ch].y + i, b = real_input(bp, H, Hp);
  if (b < 0) return none;
  if (pairs[ch].x == 0xFFFF) return {((long long)K * K + b) * H + j, -1};      // linear part behind the 4H^2 product rows
  if (bp < pairs[ch].x) return none;                                           // b < a: counted in the other half
  const int a = real_input(pairs[ch].x, H, Hp);
  const long long ab = ((long long)a * K + b) * H + j;
  return {ab, a != b ? ((long long)b * K + a) * H + j : -1};
}
// Backward word (c * 4 + i) * 4 + u: output 4 (t / bseg) + u, input 4 (t % bseg + bseg c) + i of the CTA's gate gradients
// (gate JS + unit).
__host__ __device__ inline WeightAt bwd_weight(int cell, int H, int E, const TreesShape& s, int rank, int t, int w) {
  const WeightAt none{-1, -1};
  if (cell == kRntn) {
    // thread (row a of x, q of TPA): word (c * 4 + i) * 8 + u: entry (a, b) of the symmetric S_u, then the linear part
    const int K = 2 * H, Hp = (H + 3) & ~3, tpa = s.TPA, a = t / tpa, q = t % tpa;
    if (a >= K) return none;
    const int u = w % kRntnJS, j = rank * s.JS + u;
    if (u >= s.JS || j >= H) return none;
    if (w >= 4 * kRntnBC * kRntnJS) return u % tpa == q ? WeightAt{((long long)K * K + a) * H + j, -1} : none;
    const int i = (w / kRntnJS) % 4, c = w / (4 * kRntnJS), bp = 4 * (q + tpa * c) + i;
    const int b = bp < 2 * Hp ? real_input(bp, H, Hp) : -1;
    if (b < 0) return none;
    return {((long long)a * K + b) * H + j, ((long long)b * K + a) * H + j};   // V_ab + V_ba, twice V_aa
  }
  const int out = 4 * (t / s.bseg) + w % 4, c = w / 16, in = 4 * (t % s.bseg + s.bseg * c) + (w / 4) % 4;
  if (out >= 2 * H || c >= s.BC) return none;
  const int gate = in / s.JS, unit = in - gate * s.JS, j = rank * s.JS + unit;
  if (gate >= (cell == kLstm ? 5 : 1) || j >= H) return none;
  return cell == kLstm ? WeightAt{((long long)E + out) * 5 * H + (long long)gate * H + j, -1} : WeightAt{(long long)out * H + j, -1};
}

// forward: partial sums [nseg][pass][outs], gate values [pass][outs], operand rows and cell states of a pass (states in L2)
__host__ __device__ inline int fwd_outs(const TreesShape& s) { return s.U * s.JL; }
__host__ __device__ inline int fwd_parts(int cell, const TreesShape& s) { return ((cell == kRntn ? kFwdT / 32 : s.nseg) + 7) & ~7; }
__host__ __device__ inline int fwd_buf_words(int cell, int H, const TreesShape& s) {
  return (fwd_parts(cell, s) + 1) * pass_nodes(cell) * fwd_outs(s) + pass_nodes(cell) * (2 * ((H + 3) & ~3) + 2 * ((s.JS + 3) & ~3));
}
// backward: gate gradients of a round [kND][in_row], then the sums that came in [2][cs][kND][2 JS] (RNTN: and x)
__host__ __device__ inline int bwd_in_row(int cell, const TreesShape& s) { return cell == kRntn ? kRntnJS : 4 * s.bseg * s.BC; }
__host__ __device__ inline int bwd_buf_words(int cell, int H, const TreesShape& s) {
  return kND * bwd_in_row(cell, s) + 2 * s.cs * kND * 2 * s.JS + (cell == kRntn ? kND * 2 * ((H + 3) & ~3) : 0);
}

// ---- forward -------------------------------------------------------------------------------------- //
// SAVE: a backward pass follows (trees of all cells dealt by size, the cluster's lists kept for it).  An instantiation of its own,
// because what runs once costs as code, run or not: with one for both, TreeRNN H = 128, forward alone, 10 sentences of 2 to 20
// words took 26.7 us and not 24.7, 100 of 2 to 12 words 28.7 and not 26.7; RNTN H = 32, the same 10, 34.2 and not 32.9.
template <int CELL, int U, int RC, bool SAVE>
__global__ void __launch_bounds__(kFwdT, 1) k_trees_forward(const __grid_constant__ TreesParams p) {
  extern __shared__ __align__(16) float sm[];
  __shared__ Walk s_walk;
  __shared__ TreeLoads s_loads;
  constexpr int kPass = pass_nodes(CELL);
  const int cs = p.s.cs, rank = cs > 1 ? (int)cta_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int part = blockIdx.x / cs, parts = gridDim.x / cs;
  const int H = p.H, Hp = p.Hp, JS = p.s.JS, JS4 = (JS + 3) & ~3, JL = p.s.JL, outs = U * JL, j0 = rank * JS, jn = min(JS, H - j0);   // (jn may be below one: a CTA without units)
  const TreesSmem s = trees_smem(p.n, fwd_buf_words(CELL, H, p.s));
#ifdef TREELSTM_TRACE
  long long* const trace = blockIdx.x == 0 && tid == 0 ? p.trace : nullptr;   // row d: depth d; last row: set-up
#else
  long long* const trace = nullptr;
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  float w[RC * 4 * U];
#pragma unroll
  for (int q = 0; q < RC * 4 * U; ++q) w[q] = __ldg(p.W + ((size_t)rank * (RC * 4 * U) + q) * kFwdT + tid);
  float* const red = sm + s.buf;
  if (CELL == kLstm)                                       // (sums beyond the segments stay zero; here beside the leaves' kernel)
    for (int e = tid; e < fwd_parts(CELL, p.s) * kPass * outs; e += kFwdT) red[e] = 0.f;
  // (dealing by size takes 10 k cycles, which TreeLSTM spends beside its leaves and a training step gains twice: 54 chains of 16
  // leaves, TreeRNN H = 79, forward alone 42 us without and 47 with it)
  bool planned = false;
  if constexpr (CELL == kLstm) {
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the leaves' states and the lists come from the kernel ahead, and whose forest it is
    if (p.choose && !ld_volatile(&p.st->trees_fwd)) return;
    planned = load_walk(p.walks, p.costs, p.n, 0, s, sm, part, parts, false, &s_loads, &s_walk);
  }
  if (!planned) {
    deal_trees(p, p.costs, s, sm, part, parts, CELL != kLstm && p.choose, CELL == kLstm || SAVE, &s_loads, &s_walk, trace);
    if (CELL == kLstm && SAVE && tid == 0) s_loads.longer = -1;   // (lists to be kept: below)
  }
#pragma unroll
  for (int q = 0; q < RC * 4 * U; ++q) asm volatile("" : "+f"(w[q]));   // held in registers: not to be loaded again where it is used
  TL_STAMP(trace, kTraceLevels - 1, 2);
  const Walk walk = s_walk;
  if (CELL != kLstm && SAVE && rank == 0) save_walk(p.walks, s, sm, part, parts, walk);
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
  const unsigned short* list = reinterpret_cast<const unsigned short*>(sm + s.list);
  const unsigned short* start = reinterpret_cast<const unsigned short*>(sm + s.start);
  const unsigned short* par = reinterpret_cast<const unsigned short*>(sm + s.par);
  const unsigned short* leaf = reinterpret_cast<const unsigned short*>(sm + s.leaf);
  const unsigned short* leaf_par = reinterpret_cast<const unsigned short*>(sm + s.leaf_par);
  // operand rows [h_l | h_r] of the internal nodes, padded to whole segments; then (TreeLSTM) the children's c of the
  // CTA's own units
  const int row = CELL == kRntn ? 2 * Hp : 4 * p.s.nseg * RC, crow = CELL == kLstm ? 2 * JS4 : 0;
  const bool resident = (long long)walk.internal * (row + crow) <= s.state_words;
  float* const act = red + fwd_parts(CELL, p.s) * kPass * outs;
  float* const xrow = act + kPass * outs;                   // states in L2: operand rows and cell states of a pass
  float* const state = resident ? sm + s.state : xrow;
  float* const cstate = state + (resident ? walk.internal * row : kPass * 2 * Hp);
  const uint32_t state_addr = smem_u32(state);
  const int xstride = resident ? row : 2 * Hp;           // (the padding behind an L2 row is the next row: finite, times zero)
  for (int e = tid; e < (resident ? walk.internal * (row - 2 * H) : kPass * (2 * Hp + 2 * JS4)); e += kFwdT) {
    if (resident) {
      const int q = e / (row - 2 * H), k = e - q * (row - 2 * H);
      state[q * row + (k < Hp - H ? H + k : H + k + H)] = 0.f;
    } else {
      xrow[e] = 0.f;
    }
  }
  if (CELL != kLstm)
    for (int e = tid; e < fwd_parts(CELL, p.s) * kPass * outs; e += kFwdT) red[e] = 0.f;
  const int depths = walk.depths, leaves = walk.leaves;
  // A leaf per warp and turn, as copies that need no registers, so that all of a warp's leaves are under way at once (one leaf
  // after the other through registers took 10 k cycles for the 60 of two sentences, pairs of leaves 8 k, this way 4 k).
  const float* const leaf_rows = CELL == kLstm ? p.h : p.emb;
  const int piece = H % 4 == 0 && (reinterpret_cast<uintptr_t>(leaf_rows) & 15) == 0 ? 4 : (H % 2 == 0 && (reinterpret_cast<uintptr_t>(leaf_rows) & 7) == 0 ? 2 : 1);
  const uint32_t cstate_addr = smem_u32(cstate);
#pragma unroll 1
  for (int q = warp; q < leaves && resident; q += kFwdT / 32) {
    const int node = leaf[q];
    const unsigned code = leaf_par[q];
    if (code == kNoCaller) continue;
    copy_row(state_addr + 4u * ((code >> 1) * row + (code & 1) * Hp), leaf_rows + (size_t)(CELL == kLstm ? node : (int)(kids[node] & ~kLeafBit)) * H, H, piece, lane);
    if (CELL == kLstm && jn > 0)
      copy_row(cstate_addr + 4u * ((code >> 1) * crow + (code & 1) * JS4), p.c + (size_t)node * H + j0, jn, 1, lane);
  }
  if (CELL != kLstm)                                     // a leaf's state is its word vector
    for (int q = rank + cs * warp; q < leaves; q += cs * (kFwdT / 32)) {
      const int node = leaf[q];
      const float* const src = p.emb + (size_t)(kids[node] & ~kLeafBit) * H;
      for (int k = lane; k < H; k += 32) {
        p.h[(size_t)node * H + k] = __ldg(src + k);
        count_write(p.chk_counts, node, 1);
      }
    }
  asm volatile("cp.async.wait_all;" ::: "memory");
  // the thread's first chunk, or (RNTN) its chunks' operands: b in bits 8.., a below, 255: the linear part
  const int lane_out = tid % JL, seg = tid / JL;
  const bool works = seg < p.s.nseg;
  int ops[CELL == kRntn ? RC : 1];
  if constexpr (CELL == kRntn) {
#pragma unroll
    for (int c = 0; c < RC; ++c) {
      const ushort2 ab = p.pairs[min(seg + p.s.nseg * c, p.s.chunks - 1)];
      ops[c] = ((int)ab.y << 8) | (ab.x & 255);
    }
  } else {
    ops[0] = 4 * min(seg, p.s.nseg - 1) * RC;
  }
  // what this thread adds up (node red_i of a pass, output red_o; further ones kFwdT entries on) and updates
  const int step_i = kFwdT / outs, step_o = kFwdT - step_i * outs;
  const int red_i = tid / outs, red_o = tid - red_i * outs;
  const float red_bias = __ldg(p.b + (CELL == kLstm ? min(red_o / JS, 4) * H + min(j0 + red_o % JS, H - 1) : min(j0 + red_o, H - 1)));
  const int red_g = CELL == kLstm ? red_o / JS : 0, red_u = CELL == kLstm ? red_o - red_g * JS : red_o;
  const int sets = max(1, kFwdT / (NT * JS)), cell_set = tid / (NT * JS), cell_q = tid - cell_set * NT * JS;
  const int cell_i = cell_q / JS, cell_u = cell_q - cell_i * JS;
  (void)cell_i; (void)cell_u; (void)sets;
  const int parts_sum = fwd_parts(CELL, p.s);
  cluster_sync(cs);                                      // the leaves' states are in place; every CTA of the cluster runs: its shared memory may be written
  TL_STAMP(trace, kTraceLevels - 1, 3);
  for (int d = depths - 1; d >= 0; --d) {
    for (int lo = start[d], hi = start[d + 1]; lo < hi; lo += kPass) {
      const int cnt = min(kPass, hi - lo);
      TL_STAMP(trace, d, 0);
      if (!resident) {
        // the children's states from L2 (a leaf of TreeRNN / RNTN: from the table itself)
        __syncthreads();
        for (int i = warp; i < 2 * cnt; i += kFwdT / 32) {
          const unsigned kd = kids[list[lo + (i >> 1)]];
          const int child = (int)((i & 1) ? kd >> 16 : kd & 0xFFFFu);
          const unsigned ck = kids[child];
          const bool table = CELL != kLstm && is_leaf(ck);
          const float* src = table ? p.emb + (size_t)(ck & ~kLeafBit) * H : p.h + (size_t)child * H;
          for (int k = lane; k < H; k += 32) xrow[i * Hp + k] = table ? __ldg(src + k) : __ldcg(src + k);
          if (CELL == kLstm)
            for (int u = lane; u < JS && j0 + u < H; u += 32) cstate[i * JS4 + u] = __ldcg(p.c + (size_t)child * H + j0 + u);
        }
        __syncthreads();
      }
      const float* const x0 = state + (resident ? lo * row : 0);
      auto multiply = [&](auto n_const, int first) {       // nodes `first` .. of the pass
        constexpr int N = decltype(n_const)::value;
        float acc[N][U];
        const float* xb[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          xb[i] = x0 + min(first + i, cnt - 1) * xstride + (CELL == kRntn ? 0 : ops[0]);
#pragma unroll
          for (int u = 0; u < U; ++u) acc[i][u] = 0.f;
        }
#pragma unroll
        for (int c = 0; c < RC; ++c) {
          float4 x[N];
#pragma unroll
          for (int i = 0; i < N; ++i) {
            if constexpr (CELL == kRntn) {
              x[i] = *reinterpret_cast<const float4*>(xb[i] + (ops[c] >> 8));
              const int a = ops[c] & 255;
              const float f = a == 255 ? 1.f : xb[i][a];
              x[i].x *= f; x[i].y *= f; x[i].z *= f; x[i].w *= f;
            } else {
              x[i] = *reinterpret_cast<const float4*>(xb[i] + 4 * c);
            }
          }
#pragma unroll
          for (int i = 0; i < N; ++i)
#pragma unroll
            for (int u = 0; u < U; ++u) {
              acc[i][u] = fmaf(x[i].x, w[(c * 4 + 0) * U + u], acc[i][u]);
              acc[i][u] = fmaf(x[i].y, w[(c * 4 + 1) * U + u], acc[i][u]);
              acc[i][u] = fmaf(x[i].z, w[(c * 4 + 2) * U + u], acc[i][u]);
              acc[i][u] = fmaf(x[i].w, w[(c * 4 + 3) * U + u], acc[i][u]);
            }
        }
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
          for (int u = 0; u < U; ++u) {
            if constexpr (CELL == kRntn) {               // JL is a power of two: a warp adds its own segments first
              float v = acc[i][u];
              for (int dd = JL; dd < 32; dd <<= 1) v += __shfl_xor_sync(kFull, v, dd);
              if (lane < JL) red[(warp * kPass + first + i) * outs + u * JL + lane_out] = v;
            } else if (works) {
              red[(seg * kPass + first + i) * outs + u * JL + lane_out] = acc[i][u];
            }
          }
      };
#pragma unroll 1
      for (int first = 0; first < (kPass > NT ? cnt : 1); first += NT) {
        if (cnt - first == 1) multiply(std::integral_constant<int, 1>{}, first);
        else if (cnt - first == 2) multiply(std::integral_constant<int, 2>{}, first);
        else multiply(std::integral_constant<int, NT>{}, first);
      }
      __syncthreads();
      TL_STAMP(trace, d, 1);
      auto put_h = [&](int q, int unit, float hv, int first, int by) {   // into the caller's row, in every CTA (or every by-th)
        const unsigned code = par[q];
        if (!resident || code == kNoCaller) return;
        const int at = (int)(code >> 1) * row + (int)(code & 1) * Hp + unit;
        if (cs == 1) state[at] = hv;
        else
          for (int c = first; c < cs; c += by) st_cluster(peer_addr(state_addr + 4u * (uint32_t)at, (uint32_t)c), hv);
      };
      // States of the last nodes of a depth go to global memory behind the arrival at the cluster's barrier, which otherwise
      // waits until L2 has them (a release covers them too; nobody in the cluster reads them there if the rows are resident):
      // 25 sentences, TreeLSTM H = 150, forward 73.6 -> 71.3 us; training step TreeRNN H = 128 118.3 -> 115.9, RNTN H = 32 162.3 -> 160.4
      const bool early = resident && lo + kPass >= hi;
      float* h_to = nullptr;
      float h_kept = 0.f;
      for (int i = red_i, o = red_o; i < cnt;) {
        const bool own = o == red_o;                     // else: a second output of this thread (JS > 128 / gates)
        const int g = CELL == kLstm ? (own ? red_g : o / JS) : 0, u = CELL == kLstm ? (own ? red_u : o - g * JS) : o;
        float z = own ? red_bias : __ldg(p.b + min(g, 4) * H + min(j0 + u, H - 1));
        const float* r = red + i * outs + o;
        for (int q = 0; q < parts_sum; q += 8, r += 8 * kPass * outs) {   // eight reads in flight (the sums are padded to eights)
          float v[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = r[k * kPass * outs];
          z += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
        if constexpr (CELL == kLstm) {
          const float a = g == 4 ? tanhf(z) : sigmoid_acc(z);
          act[i * outs + o] = a;
          if (p.gates && j0 + u < H) p.gates[((size_t)list[lo + i] * 5 + g) * row_pitch(H) + j0 + u] = a;
        } else if (u < JS && j0 + u < H) {
          const float hv = tanhf(z);
          const int node = list[lo + i];
          put_h(lo + i, j0 + u, hv, 0, 1);
          if (h_to) *h_to = h_kept;
          h_to = p.h + (size_t)node * H + j0 + u;
          h_kept = hv;
          count_write(p.chk_counts, node, 1);
        }
        i += step_i;
        o += step_o;
        if (o >= outs) { o -= outs; ++i; }
      }
      if (CELL != kLstm) {
        if (early) cluster_arrive(cs);
        if (h_to) *h_to = h_kept;
      }
      TL_STAMP(trace, d, 2);
      if constexpr (CELL == kLstm) {
        __syncthreads();
        // cell update; several sets of threads repeat the same few operations and share the stores to the CTAs
        float c_kept = 0.f;
        if (cell_i < cnt && j0 + cell_u < H && cell_set < sets) {
          const int q = lo + cell_i;
          const float* a = act + cell_i * outs + cell_u;
          const float* cc = cstate + (resident ? q : cell_i) * crow + cell_u;
          const float cv = a[0] * a[4 * JS] + a[JS] * cc[0] + a[2 * JS] * cc[JS4];
          const float hv = a[3 * JS] * tanhf(cv);
          put_h(q, j0 + cell_u, hv, cell_set, sets);
          if (cell_set == 0) {
            const unsigned code = par[q];
            if (resident && code != kNoCaller) cstate[(code >> 1) * crow + (code & 1) * JS4 + cell_u] = cv;
            h_to = p.h + (size_t)list[q] * H + j0 + cell_u;
            h_kept = hv;
            c_kept = cv;
            count_write(p.chk_counts, list[q], 1);
          }
        }
        if (early) cluster_arrive(cs);
        if (h_to) {
          *h_to = h_kept;
          p.c[h_to - p.h] = c_kept;
        }
      }
      if (CELL != kLstm && lo + kPass < hi) __syncthreads();   // the next pass's partial sums overwrite these
      TL_STAMP(trace, d, 3);
    }
    if (!resident) cluster_arrive(cs);
    cluster_wait(cs);                                    // the depth's states are in place (and no CTA leaves while a peer still writes to it)
    TL_STAMP(trace, d, 4);
  }
  // (TreeLSTM: not before all CTAs of the cluster have looked at the header, which says that there is nothing; and behind the walk, which the weights in
  // registers leave no room for it beside: spilled, 25 sentences, training step 185 -> 187 us.)
  if (CELL == kLstm && SAVE && rank == 0 && s_loads.longer < 0) save_walk(p.walks, trees_smem(p.n, fwd_buf_words(CELL, p.H, p.s)), sm, part, parts, s_walk);
  // what follows on the stream waits for this grid only: it must not end before the scheduler ahead of it has
  if (CELL != kLstm && blockIdx.x == 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid == 0) p.st->trees_fwd = s_loads.win;         // (TreeLSTM: the leaves' kernel has said so)
  }
}

// ---- TreeLSTM leaves ------------------------------------------------------------------------------ //
// Their states need no schedule, so this kernel runs beside the scheduler, over the whole GPU.  A CTA takes 32 to 64 consecutive node
// ids (as few as give every SM some), the leaves among them (about half), and 32 hidden units x the three gates a leaf has.  All operands of
// kLeafK contraction indices are asked for at once - the weights as one bulk copy out of an image kept for it, the
// embedding rows through registers - because the kernel is bound by the latency of its loads: in chunks of 32 indices,
// each a round trip behind the one before, 25 trees (H = 150, E = 300) took 43 us with cold caches, this way 17.
// A warp takes a quarter of the rows (4, 5, 7, 8, 10, 12 or 16) and a quarter of the contraction: rows read as broadcasts, weights one
// word per lane, 96 multiply-adds per 20 reads.  (Half of the rows and twice the quarters of the contraction, 48 per 16 reads,
// was bound by shared memory: 15 k cycles for 32 leaves.)  The quarters meet in shared memory, every warp finishes some rows.
constexpr int kLeafT = 512, kLeafU = 32, kLeafIds = 64, kLeafK = 320;
constexpr int kLeafSmem = 4 * kLeafK * (3 * kLeafU + kLeafIds);
static_assert(4 * kLeafIds <= kLeafK, "the sums of the quarters fit where the weights were");
struct LeafParams {
  int n, H, E, vocab;
  int* chk_counts;
  const int *left, *token;
  const float *emb, *Wx, *b;
  float *h, *c, *gates;
  DevStatus* st;
  long long wait_limit;
  int choose, parts;                       // 1: the first CTA says whether the clusters (so many) take the forest (clusters_win)
  const int* right;
  WalkCosts costs;
  SavedWalks walks;                        // where it leaves what each of them walks
  int ids;                                 // consecutive node ids of a CTA
};
// image of the input weights: [slice of 32 units][input unit][gate i, o, u][unit], zeros behind the last unit
__host__ __device__ inline size_t leaf_image_words(int H, int E) { return (size_t)((H + kLeafU - 1) / kLeafU) * E * 3 * kLeafU; }
__device__ __forceinline__ float leaf_weight(int H, int E, const float* W, int i) {
  const int uu = i % kLeafU, g = i / kLeafU % 3, k = i / (3 * kLeafU) % E, u = i / (3 * kLeafU) / E * kLeafU + uu;
  return u < H ? W[(size_t)k * 5 * H + (g ? g + 2 : 0) * H + u] : 0.f;
}
// RPT rows from `rows` on and a quarter of nk contraction indices
template <int RPT>
__device__ __forceinline__ void leaf_rows(const float* As, const float* Ws, int pitch, int nk, int rows, int quarter, int lane,
                                          float (&acc)[16][3]) {
  const int per = (nk + 15) / 16 * 4, lo = quarter * per, hi = min(lo + per, (nk + 3) & ~3);
#pragma unroll 1
  for (int k = lo; k < hi; k += 4) {
    float w[4][3];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int g = 0; g < 3; ++g) w[q][g] = Ws[(k + q) * 3 * kLeafU + g * kLeafU + lane];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const float4 x = *reinterpret_cast<const float4*>(As + (rows + i) * pitch + k);
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        acc[i][g] = fmaf(x.x, w[0][g], acc[i][g]);
        acc[i][g] = fmaf(x.y, w[1][g], acc[i][g]);
        acc[i][g] = fmaf(x.z, w[2][g], acc[i][g]);
        acc[i][g] = fmaf(x.w, w[3][g], acc[i][g]);
      }
    }
  }
}
// The first CTA plans for the clusters' kernel, which waits for the leaves anyhow: whether it takes the forest, and what each cluster walks.  The
// leaves' kernel is no longer for it (14.5 us, 25 sentences), and the clusters' kernel reads its lists in 2 k cycles where it made them in 23 k (H = 150, with
// the leaves' copies there: forward 71 -> 60 us, training step 199 -> 184).
constexpr int kLeafTableWords = kLeafSmem / 4;
__host__ __device__ inline int leaves_tables_at(int n) { return (n + n / 32 + 4) / 4 * 4; }   // (16-byte boundary)
__host__ __device__ inline bool leaves_hold_tables(int n) { return leaves_tables_at(n) + deal_words(n) <= kLeafTableWords; }
__device__ __forceinline__ void leaves_plan(const LeafParams& p, float* sm) {
  __shared__ TreeLoads s_loads;
  const ForestIn q{p.n, p.vocab, p.left, p.right, p.token};
  TreesSmem s{};
  s.child = p.n;
  const int tables = leaves_tables_at(p.n), used = tables + deal_words(p.n);
  const TreeLinks links = tree_links(sm + tables, p.n);
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm);
  const unsigned* child = reinterpret_cast<const unsigned*>(sm + s.child);
  if (threadIdx.x == 0) { s_loads.win = 1; s_loads.internal = 0; }
  const bool forest = !load_kids(q, s, sm, links.up, &s_loads.internal);   // (else the scheduler reports it)
  const bool dealt = forest && deals_by_size(p.n, s_loads.internal, p.parts);
  const bool climbed = p.n <= kLeafT * kClimbs && used + p.n <= kLeafTableWords;
  if (forest)
    deal_by_size(p.n, kids, child, links, p.costs, p.parts, dealt, p.choose != 0, 0, &s_loads, climbed ? reinterpret_cast<unsigned*>(sm + used) : nullptr);
  __syncthreads();
  const int win = s_loads.win;
  plan_walks(p.n, kids, child, links, win != 0, forest, dealt, climbed, p.parts, reinterpret_cast<int*>(sm + used), kLeafTableWords - used, p.walks, &s_loads);
  asm volatile("griddepcontrol.wait;" ::: "memory");     // the scheduler clears the control block at its start
  if (threadIdx.x == 0) p.st->trees_fwd = win;
}
__global__ void __launch_bounds__(kLeafT) k_leaves_fp32(const __grid_constant__ LeafParams p) {
  extern __shared__ __align__(16) float leaf_smem[];
  float* const Ws = leaf_smem;                           // [kLeafK][3 gates][32 units]; then the quarters' sums
  float* const As = leaf_smem + kLeafK * 3 * kLeafU;     // [rows][pitch]
  __shared__ int s_node[kLeafIds], s_tok[kLeafIds], s_count, s_abort;
  __shared__ __align__(8) uint64_t s_bar;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, H = p.H, E = p.E;
  const int tiles_u = (H + kLeafU - 1) / kLeafU, block = (int)blockIdx.x - 1, slice = block % tiles_u;
  const int id0 = block / tiles_u * p.ids, u0 = slice * kLeafU;
  const uint32_t bar = smem_u32(&s_bar);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x == 0) { leaves_plan(p, leaf_smem); return; }
  auto ask = [&](int k0) {                               // one thread: the weights of the next kLeafK indices
    const uint32_t bytes = (uint32_t)min(kLeafK, E - k0) * 3 * kLeafU * 4;
    mbar_arrive_expect_tx(bar, bytes);
    bulk_load(smem_u32(Ws), p.Wx + ((size_t)slice * E + k0) * 3 * kLeafU, bytes, bar);
  };
  if (tid == 32) {
    mbar_init(bar, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    ask(0);
  }
  if (tid < 32) {                                        // the leaves among the CTA's node ids, ascending
    int count = 0;
#pragma unroll
    for (int q = 0; q < kLeafIds / 32; ++q) {
      const int k = id0 + 32 * q + tid;
      const bool lf = k < min(p.n, id0 + p.ids) && p.left[min(k, p.n - 1)] < 0;
      const unsigned m = __ballot_sync(0xffffffffu, lf);
      if (lf) {
        const int at = count + __popc(m & ((1u << tid) - 1u));
        s_node[at] = k;
        s_tok[at] = min(max(p.token[k], 0), p.vocab - 1);   // nothing has been validated yet
      }
      count += __popc(m);
    }
    if (tid == 0) s_count = count;
  }
  __syncthreads();
  const int count = s_count, quarter = warp >> 2;
  // Rows of a warp.  32 ids, what a CTA takes of a small forest, hold 16 leaves and a few more or less.  A size is code of its own that each SM fetches once: with one for 24
  // leaves as well, 25 sentences, H = 150, took 57.1 us and not 56.4; without the one for 20, one sentence 36.5 and not 35.4, five 50.5 and not 49.5.
  const int rpt = count <= 16 ? 4 : (count <= 20 ? 5 : (count <= 28 ? 7 : (count <= 32 ? 8 : (count <= 40 ? 10 : (count <= 48 ? 12 : 16))))), row0 = (warp & 3) * rpt;
  const int u = min(u0 + lane, H - 1);
  const float bi = __ldg(p.b + u), bo = __ldg(p.b + 3 * H + u), bu = __ldg(p.b + 4 * H + u);
  float acc[16][3] = {};
  bool ok = true;
  for (int k0 = 0, turn = 0; k0 < E; k0 += kLeafK, ++turn) {
    const int nk = min(kLeafK, E - k0), pitch = (nk + 3) & ~3;
    if (turn > 0) {
      __syncthreads();                                   // the previous indices' readers are done
      if (tid == 32) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        ask(k0);
      }
    }
    // rows: a warp takes every 16th; lanes along the row, ten loads in flight; zeros up to the pitch
    for (int i = warp; i < count; i += kLeafT / 32) {
      const float* src = p.emb + (size_t)s_tok[i] * E + k0;
      float v[kLeafK / 32];
#pragma unroll
      for (int j = 0; j < kLeafK / 32; ++j) v[j] = __ldg(src + min(lane + 32 * j, nk - 1));
#pragma unroll
      for (int j = 0; j < kLeafK / 32; ++j)
        if (lane + 32 * j < pitch) As[i * pitch + lane + 32 * j] = lane + 32 * j < nk ? v[j] : 0.f;
    }
    ok = mbar_wait(bar, turn & 1, &s_abort, p.wait_limit, p.st) && ok;
    // behind the last index, up to a multiple of four: zeros, like the rows' (shared memory may hold anything)
    if (nk & 3)
      for (int e = tid; e < (pitch - nk) * 3 * kLeafU; e += kLeafT) Ws[nk * 3 * kLeafU + e] = 0.f;
    if (__syncthreads_or(!ok)) { ok = false; break; }
    if (row0 < count) {
      if (rpt == 4) leaf_rows<4>(As, Ws, pitch, nk, row0, quarter, lane, acc);
      else if (rpt == 5) leaf_rows<5>(As, Ws, pitch, nk, row0, quarter, lane, acc);
      else if (rpt == 7) leaf_rows<7>(As, Ws, pitch, nk, row0, quarter, lane, acc);
      else if (rpt == 8) leaf_rows<8>(As, Ws, pitch, nk, row0, quarter, lane, acc);
      else if (rpt == 10) leaf_rows<10>(As, Ws, pitch, nk, row0, quarter, lane, acc);
      else if (rpt == 12) leaf_rows<12>(As, Ws, pitch, nk, row0, quarter, lane, acc);
      else leaf_rows<16>(As, Ws, pitch, nk, row0, quarter, lane, acc);
    }
  }
  if (__syncthreads_or(!ok)) {                           // a wait expired: what was asked for gets a bounded time to land
    if (tid == 32) { mbar_drain(bar, 0); mbar_drain(bar, 1); }
    __syncthreads();
    return;
  }
  float* const red = Ws;                                 // [quarter][row][gate][unit]
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (i < rpt)
#pragma unroll
      for (int g = 0; g < 3; ++g) red[((quarter * kLeafIds + row0 + i) * 3 + g) * kLeafU + lane] = acc[i][g];
  __syncthreads();
  if (u0 + lane < H) {
    for (int at = warp; at < count; at += kLeafT / 32) {
      const int node = s_node[at];
      float z[3];
#pragma unroll
      for (int g = 0; g < 3; ++g) {
        const float* r = red + (at * 3 + g) * kLeafU + lane;
        constexpr int kq = kLeafIds * 3 * kLeafU;
        z[g] = (r[0] + r[kq]) + (r[2 * kq] + r[3 * kq]);
      }
      const float gi = sigmoid_acc(z[0] + bi), go = sigmoid_acc(z[1] + bo), gu = tanhf(z[2] + bu);
      const float cv = gi * gu;
      p.c[(size_t)node * H + u] = cv;
      p.h[(size_t)node * H + u] = go * tanhf(cv);
      count_write(p.chk_counts, node, 1);
      if (p.gates) {
        const int gs = row_pitch(H);
        float* g = p.gates + (size_t)node * 5 * gs + u;
        g[0] = gi; g[3 * gs] = go; g[4 * gs] = gu;
      }
    }
  }
  // (The kernel behind this one waits for this grid only, which must not end before the scheduler ahead of it has: the first CTA waits
  // for that, the others make room for that kernel.)
}


// ---- backward: dz of every node (TreeRNN / RNTN: dh of the leaves) from the classifier's dh --------- //
// TreeLSTM   dc += dh o (1 - tanh^2 c);  dz_o = dh tanh(c) o (1 - o),  dz_i = dc u i (1 - i),  dz_u = dc i (1 - u^2),
//            dz_f = dc c_child f (1 - f),  dc_child = dc f;  dh_children += W_h dz
// TreeRNN    dz = dh (1 - h^2);  dh_children += W dz
// RNTN       the same dz;  dh_children += W dz + sum_b x_b sum_j dz_j (V_j[a][b] + V_j[b][a])
// A round is up to kND nodes of one depth: gate gradients of the CTA's own units (a thread each) | products, SEG lanes
// per four outputs, sums sent to the owners of the units | cluster barrier | the owner adds what came to dh.
// What a round needs from global memory and no ancestor changes is fetched a round ahead.
template <int CELL, int SEG, int BC, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_trees_backward(const __grid_constant__ TreesParams p) {
  constexpr int G = CELL == kLstm ? 5 : 1;
  constexpr int kWords = CELL == kRntn ? kRntnBwdWords : BC * 16;
  extern __shared__ __align__(16) float sm[];
  __shared__ Walk s_walk;
  __shared__ TreeLoads s_loads;
  const int cs = p.s.cs, rank = cs > 1 ? (int)cta_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
  const int part = blockIdx.x / cs, parts = gridDim.x / cs;
  const int H = p.H, Hp = p.Hp, JS = p.s.JS, j0 = rank * JS, jn = max(0, min(JS, H - j0));
  const int in_row = bwd_in_row(CELL, p.s), nd = min(kND, nt / JS);
  const TreesSmem s = trees_smem(p.n, bwd_buf_words(CELL, H, p.s));
#ifdef TREELSTM_TRACE
  long long* const trace = blockIdx.x == 0 && tid == 0 ? p.trace : nullptr;
#else
  long long* const trace = nullptr;
#endif
  TL_STAMP(trace, kTraceLevels - 1, 0);
  if (p.choose) {
    // the schedule is the forward's: where even an equal deal and a chain of the forest's depth would take too long, no
    // table is set up
    const int roots = p.st->n_roots, internal = (p.n - roots) / 2, waves = p.st->n_levels - 1, busy = max(1, min(roots, parts));
    const float least = fmaxf(tree_cost(p.costs, (float)internal / (float)busy, 1.f, (float)internal),
                              tree_cost(p.costs, (float)waves, (float)waves, (float)internal));
    if (least >= grid_cost(p.costs, (float)waves, (float)internal)) {
      if (blockIdx.x == 0) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (tid == 0) p.st->trees_bwd = 0;
      }
      return;
    }
  }
  float* const in = sm + s.buf;                          // [kND][in_row]
  float* const dx = in + kND * in_row;                   // [2][cs][kND][2 JS]
  float* const xs = dx + 2 * cs * kND * 2 * JS;          // RNTN: [kND][2 Hp]
  for (int e = tid; e < kND * in_row; e += nt) in[e] = 0.f;
  if (CELL == kRntn)
    for (int e = tid; e < kND * 2 * Hp; e += nt) xs[e] = 0.f;
  TL_STAMP(trace, kTraceLevels - 1, 1);
  if (!(p.walks.at && p.st->trees_fwd && load_walk(p.walks, p.costs, p.n, p.st->n_roots, s, sm, part, parts, p.choose != 0, &s_loads, &s_walk)))
    deal_trees(p, p.costs, s, sm, part, parts, p.choose != 0, true, &s_loads, &s_walk, trace);
  // The weights behind the lists: asked for before them, some were spilled, and read again in every round (25 sentences, H = 150,
  // training step 224 us, this way 216).
  const float* image = p.W + (size_t)rank * kWords * nt + tid;
  asm volatile("" : "+l"(image));
  float w[kWords];
#pragma unroll
  for (int q = 0; q < kWords; ++q) w[q] = __ldg(image + (size_t)q * nt);
#pragma unroll
  for (int q = 0; q < kWords; ++q) asm volatile("" : "+f"(w[q]));       // held in registers: not to be loaded again where it is used
  TL_STAMP(trace, kTraceLevels - 1, 2);
  const Walk walk = s_walk;
  const unsigned* kids = reinterpret_cast<const unsigned*>(sm + s.kids);
  const unsigned short* list = reinterpret_cast<const unsigned short*>(sm + s.list);
  const unsigned short* start = reinterpret_cast<const unsigned short*>(sm + s.start);
  const unsigned short* par = reinterpret_cast<const unsigned short*>(sm + s.par);
  const unsigned short* leaf = reinterpret_cast<const unsigned short*>(sm + s.leaf);
  const unsigned short* leaf_par = reinterpret_cast<const unsigned short*>(sm + s.leaf_par);
  // by caller: dh (and behind it dc) of its two children, the CTA's own units: in shared memory if they fit
  const int row = CELL == kLstm ? 4 * JS : 2 * JS;
  const bool resident = (long long)walk.internal * row <= s.state_words;
  float* const state = sm + s.state;
  const int my_i = tid / JS, my_u = tid - my_i * JS;     // the thread's node of a round and unit
  const bool mine = my_i < nd && my_u < jn;
  float g[G] = {}, cn = 0.f, cl = 0.f, cr = 0.f, xv[2] = {0.f, 0.f};    // of the next round: gates and cell states, or h; x
  auto fetch = [&](int lo) {
    if (lo >= walk.internal) return;
    if (mine) {
      const int node = list[min(lo + my_i, walk.internal - 1)];
      const size_t at = (size_t)node * H + j0 + my_u;
      if constexpr (CELL == kLstm) {
        const unsigned kd = kids[node];
        const float* gp = p.gates + (size_t)node * 5 * row_pitch(H) + j0 + my_u;
#pragma unroll
        for (int q = 0; q < G; ++q) g[q] = __ldg(gp + q * row_pitch(H));
        cn = __ldg(p.c + at);
        cl = __ldg(p.c + (size_t)(kd & 0xFFFFu) * H + j0 + my_u);
        cr = __ldg(p.c + (size_t)(kd >> 16) * H + j0 + my_u);
      } else {
        cn = __ldg(p.h + at);
      }
    }
    if constexpr (CELL == kRntn) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int e = tid + q * nt, i = e / (2 * H), k = e - i * 2 * H;
        const unsigned kd = kids[list[min(lo + i, walk.internal - 1)]];
        xv[q] = __ldg(p.h + (size_t)(k >= H ? kd >> 16 : kd & 0xFFFFu) * H + (k >= H ? k - H : k));
      }
    }
  };
  fetch(0);
  // where this thread's output goes: the owner of unit k of a child, [rank][0][side JS + u] of its buffer
  const int out = CELL == kRntn ? tid / p.s.TPA : 4 * (tid / SEG) + value_of_lane<SEG>(lane);
  const bool sends = out < 2 * H && (CELL == kRntn ? tid % p.s.TPA == 0 : (lane & (SEG / 4 - 1)) == 0);
  uint32_t send_addr = 0;
  if (sends) {
    const int side = out >= H, k = out - side * H, owner = k / JS;
    const uint32_t local = smem_u32(dx) + 4u * (uint32_t)(rank * kND * 2 * JS + side * JS + k - owner * JS);
    send_addr = cs > 1 ? peer_addr(local, (uint32_t)owner) : local;
  }
  const uint32_t send_turn = 4u * (uint32_t)(cs * kND * 2 * JS), send_node = 4u * (uint32_t)(2 * JS);
  const int sum_i0 = tid / (2 * JS), sum_k0 = tid - sum_i0 * 2 * JS, sum_di = nt / (2 * JS), sum_dk = nt - sum_di * 2 * JS;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // All that is ahead of this grid has ended: the weight gradient's kernel may read it while it sets itself up.  (k_rec_grads, whose CTAs are small, would
  // come up eight to an SM on the few SMs without a cluster and stay there: RNTN step 160 -> 174 us.)
  if (CELL == kLstm) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  TL_STAMP(trace, kTraceLevels - 1, 3);
  if (resident)
    for (int e = tid; e < walk.internal * 2 * JS; e += nt) {
      const int q = e / (2 * JS), k = e - q * 2 * JS, side = k >= JS, u = k - side * JS;
      const unsigned kd = kids[list[q]];
      state[q * row + k] = u < jn ? __ldcg(p.dh + (size_t)(side ? kd >> 16 : kd & 0xFFFFu) * H + j0 + u) : 0.f;
    }
  // generic pointers: shared or global memory, written by this CTA only.  A root's dh is the classifier's.
  auto dh_at = [&](unsigned code, int node, int u) -> float* {
    return resident && code != kNoCaller ? state + (code >> 1) * row + (code & 1) * JS + u : p.dh + (size_t)node * H + j0 + u;
  };
  auto dc_at = [&](unsigned code, int node, int u) -> float* {
    return resident ? state + (code >> 1) * row + 2 * JS + (code & 1) * JS + u : p.dc + (size_t)node * H + j0 + u;
  };
  cluster_sync(cs);                                      // every CTA of the cluster runs: its shared memory may be written
  TL_STAMP(trace, kTraceLevels - 1, 4);
  int turn = 0;
  for (int d = 0; d < walk.depths; ++d) {
    const int hi = start[d + 1];
    for (int lo = start[d]; lo < hi; lo += nd, turn ^= 1) {
      const int cnt = min(nd, hi - lo);
      TL_STAMP(trace, d, 0);
      if (mine && my_i < cnt) {
        const int q = lo + my_i, node = list[q];
        const unsigned code = par[q];
        const float dhn = *dh_at(code, node, my_u);
        float* z = in + my_i * in_row + my_u;
        if constexpr (CELL == kLstm) {
          const float gi = g[0], gl = g[1], gr = g[2], go = g[3], gu = g[4];
          const float tc = tanhf(cn);
          const float dcn = (d == 0 ? 0.f : *dc_at(code, node, my_u)) + dhn * go * (1.f - tc * tc);
          const float v[5] = {dcn * gu * gi * (1.f - gi), dcn * cl * gl * (1.f - gl), dcn * cr * gr * (1.f - gr),
                              dhn * tc * go * (1.f - go), dcn * gi * (1.f - gu * gu)};
#pragma unroll
          for (int k = 0; k < 5; ++k) z[k * JS] = v[k];
          const unsigned kd = kids[node];
          *dc_at(2u * q, (int)(kd & 0xFFFFu), my_u) = dcn * gl;          // every node has exactly one caller: plain stores
          *dc_at(2u * q + 1u, (int)(kd >> 16), my_u) = dcn * gr;
        } else {
          z[0] = dhn * (1.f - cn * cn);
        }
      }
      if constexpr (CELL == kRntn) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int e = tid + q * nt, i = e / (2 * H), k = e - i * 2 * H;
          if (i < kND) xs[i * 2 * Hp + (k >= H ? Hp + k - H : k)] = xv[q];
        }
      }
      __syncthreads();
      TL_STAMP(trace, d, 1);
      // What the products do not wait for: dz to memory, the next round's values.  (Ahead of the barrier the gates of 16 nodes took 2.5 k cycles, this way
      // 1.1 k and the products 0.6 k more: 25 sentences, H = 150, training step 183.4 -> 180.2 us.)
      if (mine && my_i < cnt) {
        float* dz = p.dz + (size_t)list[lo + my_i] * G * H + j0 + my_u;
#pragma unroll
        for (int k = 0; k < G; ++k) dz[k * H] = in[my_i * in_row + my_u + k * JS];
      }
      fetch(lo + cnt);
      const uint32_t to = send_addr + (uint32_t)turn * send_turn;
      auto send = [&](int i, float v) {
        if (!sends) return;
        if (cs > 1) st_cluster(to + (uint32_t)i * send_node, v);
        else asm volatile("st.shared.f32 [%0], %1;" ::"r"(to + (uint32_t)i * send_node), "f"(v) : "memory");
      };
      if constexpr (CELL == kRntn) {
        // thread (row a of x, every TPA-th chunk of columns): M_ab = sum_u S_u[a][b] dz_u, then sum_b M_ab x_b
        const int tpa = p.s.TPA, q = tid % tpa;
        for (int i = 0; i < cnt; ++i) {
          const float4 z0 = *reinterpret_cast<const float4*>(in + i * in_row), z1 = *reinterpret_cast<const float4*>(in + i * in_row + 4);
          const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
          float v = 0.f;
#pragma unroll
          for (int c = 0; c < kRntnBC; ++c) {
            const float4 x4 = *reinterpret_cast<const float4*>(xs + i * 2 * Hp + min(4 * (q + tpa * c), 2 * Hp - 4));
            const float x[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              float m = 0.f;
#pragma unroll
              for (int u = 0; u < kRntnJS; ++u) m = fmaf(w[(c * 4 + k) * kRntnJS + u], z[u], m);
              v = fmaf(m, x[k], v);
            }
          }
#pragma unroll
          for (int u = 0; u < kRntnJS; ++u) v = fmaf(w[4 * kRntnBC * kRntnJS + u], z[u], v);
          for (int dd = tpa / 2; dd > 0; dd >>= 1) v += __shfl_xor_sync(kFull, v, dd);
          send(i, v);
        }
      } else {
        const float* const zin = in + 4 * (tid % SEG);
        auto nodes = [&](auto n_const, int i0) {
          constexpr int N = decltype(n_const)::value;
          float acc[N][4];
#pragma unroll
          for (int i = 0; i < N; ++i)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[i][u] = 0.f;
#pragma unroll
          for (int c = 0; c < BC; ++c) {
            if (c >= p.s.BC) break;                      // the same for every thread
#pragma unroll
            for (int i = 0; i < N; ++i) {
              const float4 x = *reinterpret_cast<const float4*>(zin + (i0 + i) * in_row + 4 * SEG * c);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                acc[i][u] = fmaf(x.x, w[16 * c + u], acc[i][u]); acc[i][u] = fmaf(x.y, w[16 * c + 4 + u], acc[i][u]);
                acc[i][u] = fmaf(x.z, w[16 * c + 8 + u], acc[i][u]); acc[i][u] = fmaf(x.w, w[16 * c + 12 + u], acc[i][u]);
              }
            }
          }
#pragma unroll
          for (int i = 0; i < N; ++i) {
            lane_sums4<SEG>(acc[i], lane);
            send(i0 + i, acc[i][0]);
          }
        };
        int i = 0;
        for (; i + 1 < cnt; i += 2) nodes(std::integral_constant<int, 2>{}, i);
        if (i < cnt) nodes(std::integral_constant<int, 1>{}, i);
      }
      TL_STAMP(trace, d, 2);
      cluster_sync(cs);
      TL_STAMP(trace, d, 3);
      const float* got = dx + turn * cs * kND * 2 * JS;
      for (int i = sum_i0, k = sum_k0; i < cnt;) {
        const int side = k >= JS, u = k - side * JS;
        float v = 0.f;
#pragma unroll 8
        for (int c = 0; c < cs; ++c) v += got[(c * kND + i) * 2 * JS + k];
        const unsigned kd = resident ? 0u : kids[list[lo + i]];
        float* at = dh_at((unsigned)(2 * (lo + i) + side), (int)(side ? kd >> 16 : kd & 0xFFFFu), u);
        if (u < jn) *at = *at + v;
        i += sum_di;
        k += sum_dk;
        if (k >= 2 * JS) { k -= 2 * JS; ++i; }
      }
      TL_STAMP(trace, d, 4);
    }
    __syncthreads();                                     // the next depth's dh (this CTA's units) is complete
    TL_STAMP(trace, d, 5);
  }
  // leaves: their own gate gradients (no forget gates), or for the other cells dh where the gradient kernel reads it
  for (int e = tid; e < walk.leaves * JS; e += nt) {
    const int q = e / JS, u = e - q * JS;
    if (u >= jn) continue;
    const unsigned code = leaf_par[q];
    const int node = leaf[q];
    const size_t at = (size_t)node * H + j0 + u;
    if constexpr (CELL == kLstm) {
      const int gs = row_pitch(H);
      const float* gp = p.gates + (size_t)node * 5 * gs + j0 + u;
      const float gi = __ldg(gp), go = __ldg(gp + 3 * gs), gu = __ldg(gp + 4 * gs), tc = tanhf(__ldg(p.c + at));
      const float dhn = *dh_at(code, node, u);
      const float dcn = (code == kNoCaller ? 0.f : *dc_at(code, node, u)) + dhn * go * (1.f - tc * tc);
      float* dz = p.dz + (size_t)node * 5 * H + j0 + u;
      dz[0] = dcn * gu * gi * (1.f - gi);
      dz[H] = 0.f;
      dz[2 * H] = 0.f;
      dz[3 * H] = dhn * tc * go * (1.f - go);
      dz[4 * H] = dcn * gi * (1.f - gu * gu);
    } else if (resident) {
      p.dh[at] = *dh_at(code, node, u);
    }
  }
  if (blockIdx.x == 0 && tid == 0) p.st->trees_bwd = s_loads.win;
  cluster_sync(cs);                                      // no CTA leaves while a peer may still write to it
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
  StatusOut out;
};
__device__ __forceinline__ void rec_grads(const GradParams& p) {
  __shared__ float As[GN][GR];
  __shared__ __align__(16) float Ds[GN][GU];
  __shared__ int s_node[GN], s_l[GN], s_r[GN];
  __shared__ int s_a[GR], s_b[GR];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, H = p.H, K = p.K;
  // On any error the kernels ahead may have stopped half way: with a label out of range some CTAs of k_bwd_begin give up at
  // their last barrier, and the tokens they would have placed still hold the mark 1, which is no row of dEmb_rows.
  if (__syncthreads_or(ld_volatile(&p.st->status) != 0 || p.st->n_levels < 1)) return;
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
__global__ void __launch_bounds__(kGT) k_rec_grads(const __grid_constant__ GradParams p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  rec_grads(p);
  publish_status(p.st, p.out);
}


// ---- register images and launches ------------------------------------------------------------------ //
// The images that are wanted (out != nullptr), one after the other in one launch: it belongs to every change of the weights.
struct PackParams {
  int cell, H, E, fwd_words, bwd_words;
  TreesShape s;
  const ushort2* pairs;
  const float* src;
  float *fwd, *bwd, *leaves;
};
__global__ void k_trees_pack(const __grid_constant__ PackParams p) {
  const int n_fwd = p.fwd ? p.s.cs * p.fwd_words * kFwdT : 0, n_bwd = p.bwd ? p.s.cs * p.bwd_words * p.s.bthreads : 0;
  const int total = n_fwd + n_bwd + (p.leaves ? (int)leaf_image_words(p.H, p.E) : 0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    if (i >= n_fwd + n_bwd) {
      p.leaves[i - n_fwd - n_bwd] = leaf_weight(p.H, p.E, p.src, i - n_fwd - n_bwd);
      continue;
    }
    const bool backward = i >= n_fwd;
    const int at_i = backward ? i - n_fwd : i, threads = backward ? p.s.bthreads : kFwdT, words = backward ? p.bwd_words : p.fwd_words;
    const int t = at_i % threads, w = (at_i / threads) % words, rank = at_i / threads / words;
    const WeightAt at = backward ? bwd_weight(p.cell, p.H, p.E, p.s, rank, t, w) : fwd_weight(p.cell, p.H, p.E, p.s, rank, t, w, p.pairs);
    float v = 0.f;
    if (at.i0 >= 0) v = p.src[at.i0];
    if (at.i1 >= 0) v += p.src[at.i1];
    (backward ? p.bwd : p.fwd)[at_i] = v;
  }
}

constexpr int kLstmRC = 4, kRnnRC = 4, kRntnRC = 3;       // forward chunks per thread (U = 5, 4, 4)
int fwd_words(int cell) { return cell == kLstm ? 20 * kLstmRC : (cell == kRnn ? 16 * kRnnRC : 16 * kRntnRC); }
int bwd_chunks(int cell, const TreesShape& s) { return cell == kLstm && s.bseg == 4 ? 5 : 4; }
int bwd_words(int cell, const TreesShape& s) { return cell == kRntn ? kRntnBwdWords : 16 * bwd_chunks(cell, s); }

// One cluster size: does the slice fit the registers?
bool shape_fits(int cell, int H, int cs, TreesShape& s) {
  const int Hp = round_up(H, 4), G = cell == kLstm ? 5 : 1;
  s.cs = cs;
  s.JS = (H + cs - 1) / cs;
  s.U = cell == kLstm ? 5 : 4;
  if (NT * s.JS > kFwdT) return false;
  if (cell == kRntn) {
    for (s.JL = 1; 4 * s.JL < s.JS; s.JL *= 2) {}
    s.nc = kRntnRC;
    s.nseg = (s.chunks + s.nc - 1) / s.nc;
    if (s.nseg * s.JL > kFwdT) return false;
    s.bthreads = kRntnT; s.bseg = 1; s.BC = kRntnBC;
    for (s.TPA = 32; s.TPA * 2 * H > kRntnT; s.TPA /= 2) {}
    return s.JS <= kRntnJS;
  }
  s.chunks = 2 * Hp / 4;
  s.JL = cell == kLstm ? s.JS : (s.JS + 3) / 4;
  s.nc = cell == kLstm ? kLstmRC : kRnnRC;                // whole segments: as few partial sums as the registers allow
  s.nseg = (s.chunks + s.nc - 1) / s.nc;
  if (s.nseg * s.JL > kFwdT) return false;
  // backward: eight lanes per four outputs where the threads allow it
  const int groups = (2 * H + 3) / 4;
  s.bseg = groups * 8 <= kBwdT ? 8 : 4;
  if (groups * s.bseg > kBwdT) return false;
  s.bthreads = round_up(groups * s.bseg, 32);
  if (s.bthreads < s.JS) s.bthreads = round_up(s.JS, 32);
  s.BC = ((G * s.JS + 3) / 4 + s.bseg - 1) / s.bseg;
  return s.BC <= bwd_chunks(cell, s);
}

using TreesKernel = void (*)(const TreesParams);
template <bool SAVE>
TreesKernel forward_kernel_of(int cell) {
  return cell == kRntn ? k_trees_forward<kRntn, 4, kRntnRC, SAVE> : (cell == kRnn ? k_trees_forward<kRnn, 4, kRnnRC, SAVE> : k_trees_forward<kLstm, 5, kLstmRC, SAVE>);
}
TreesKernel forward_kernel(int cell, bool save) { return save ? forward_kernel_of<true>(cell) : forward_kernel_of<false>(cell); }
TreesKernel backward_kernel(int cell, const TreesShape& s) {
  if (cell == kRntn) return k_trees_backward<kRntn, 8, 1, kRntnT>;
  if (cell == kRnn) return s.bseg == 8 ? k_trees_backward<kRnn, 8, 4, kBwdT> : k_trees_backward<kRnn, 4, 4, 512>;
  return s.bseg == 8 ? k_trees_backward<kLstm, 8, 4, kBwdT> : k_trees_backward<kLstm, 4, 5, 512>;
}

// RNTN chunks of row a of x: products x_a x_b, b >= a, four b at a time; a = 2 Hp stands for x itself
__host__ __device__ inline int pair_chunks(int a, int H, int Hp) { return a == 2 * Hp ? Hp / 2 : (a % Hp < H ? Hp / 2 - a / 4 : 0); }
__global__ void k_trees_pairs(int H, ushort2* pairs) {   // a thread per row
  const int Hp = (H + 3) & ~3, a = threadIdx.x;
  if (a > 2 * Hp) return;
  int at = 0;
  for (int b = 0; b < a; ++b) at += pair_chunks(b, H, Hp);
  for (int c = 0, n = pair_chunks(a, H, Hp); c < n; ++c)
    pairs[at + c] = a == 2 * Hp ? make_ushort2(0xFFFF, (unsigned short)(4 * c)) : make_ushort2((unsigned short)a, (unsigned short)(4 * (a / 4 + c)));
}
constexpr int kPairsT = 128;
static_assert(2 * kRntnMaxH + 1 <= kPairsT, "a thread for every row of x, and one for x itself");
size_t images_bytes(const treelstm* ctx, int what) {     // forward image, backward image, chunk operands, leaves' weights
  const auto& s = ctx->trees.s;
  const size_t cta = sizeof(float) * (size_t)s.cs;
  return round_up_sz(what == 0 ? cta * kFwdT * fwd_words(ctx->cell) : (what == 1 ? cta * s.bthreads * bwd_words(ctx->cell, s)
                                                                               : what == 2 ? sizeof(ushort2) * (ctx->cell == kRntn ? s.chunks : 0)
                                                                                           : ctx->cell == kLstm ? 4 * leaf_image_words(ctx->H, ctx->E) : 0), 256);
}

TreesParams trees_params(treelstm* ctx, int n, const int32_t* left, const int32_t* right, const int32_t* token, float* h,
                         float* c, void* ws, const WsLayout& lay) {
  char* base = static_cast<char*>(ws);
  TreesParams p{};
  p.n = n; p.H = ctx->H; p.E = ctx->E; p.vocab = ctx->vocab; p.Hp = round_up(ctx->H, 4); p.s = ctx->trees.s;
  p.chk_counts = check_counters(ws, lay);
  p.left = left; p.right = right; p.token = token;
  p.emb = ctx->emb; p.b = ctx->b; p.pairs = ctx->trees.pairs;
  p.h = h; p.c = c;
  p.dh = reinterpret_cast<float*>(base + lay.dh);
  p.dc = reinterpret_cast<float*>(base + lay.dc);
  p.dz = reinterpret_cast<float*>(base + lay.dz);
  p.st = reinterpret_cast<DevStatus*>(base + lay.status);
  p.trace = nullptr;
#ifdef TREELSTM_TRACE
  p.trace = reinterpret_cast<long long*>(base + lay.trace);   // forward: first table, backward: second
#endif
  return p;
}

// As many clusters as the device holds at once (they do not wait for one another, but trees dealt to a cluster that
// starts late end late).  `after_running`: the kernel may start while the one ahead of it on the stream still runs (it
// waits on the device for its end).
int launch_trees(treelstm* ctx, TreesKernel kernel, const TreesParams& p, int threads, int clusters, bool after_running, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * p.s.cs); cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = kSmemMax; cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = p.s.cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = after_running ? 1 : 0;
  cfg.attrs = at; cfg.numAttrs = 2;
  TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, kernel, p));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace

// Fitted to whole calls, each way forced (caches cold; 1, 4, 25, 100 and 250 trees, balanced, chains and sentences, one large tree
// among 24 sentences; TreeLSTM H = 64 to 256, TreeRNN 64 to 256, RNTN 16 and 32).  Forward / backward in us, clusters against
// whole GPU: TreeLSTM H = 150, 25 sentences 100 / 163 against 170 / 298, chain of 1024 leaves 3 410 / 3 870 against 7 450 / 8 530,
// balanced tree of 1024 leaves 945 / 848 against 166 / 240; TreeRNN H = 128, 25 sentences 51 / 112 against 351 / 361, balanced
// tree of 8192 leaves 3 080 / 3 320 against 590 / 1 330.  Both ways have become faster since (TreeLSTM H = 150, 25 sentences 69 / 127 against 138 / 252, chain 3 220 / 3 820
// against 7 340 / 8 890, balanced tree 908 / 768 against 151 / 212) and the constants are those of the fit: of 420 calls (TreeLSTM H = 64 to 256, TreeRNN 128, RNTN 32,
// both directions, many of them near the border) 27 take more than 5 % longer than the better way, at most 24 %.
WalkCosts walk_costs(int cell, int H, bool backward) {
  const float h = (float)H;
  if (cell == kLstm) {
    // a wavefront over the whole GPU: with the weights' slice resident in shared memory, or streamed (from H = 165 on)
    if (!backward)
      return {10.f, 0.35f + 0.0025f * fminf(h, 200.f), 1.9f, 1.5e-4f * h, 40.f, H <= 164 ? 3.2f + 0.0265f * h : 0.1f * h, fmaxf(0.f, 2.9e-4f * h - 0.0075f)};
    return {66.f, 0.65f, 2.9f, 2e-4f * h, H % 4 ? 150.f : 105.f, 8.f, 1.5e-4f * h};   // (rows that are no whole 16 bytes)
  }
  if (cell == kRnn) {
    const float unit = 0.3f + 0.0011f * h;
    if (!backward) return {15.f, unit, 1.2f, 0.f, 45.f, 1.5f + 0.157f * h, 2.5e-4f * h};
    return {56.f, unit, 1.7f, 0.f, 85.f, 12.5f, 1.2e-3f * h};
  }
  if (!backward) return {18.f, 0.87f, 1.05f, 0.f, 50.f, 0.27f * h * h, 1.1e-4f * h * h};
  return {56.f, 0.55f, 2.f, 0.f, 85.f, 3.9f * h, 4.2e-4f * h * h};
}
// Forests whose calls launch the tree kernels only.  A forest of n nodes gains most from the whole GPU as one balanced tree: it
// is small if the clusters are the better way even then.  For TreeRNN and RNTN, where a second kernel that only looks and exits
// would be 3 to 5 us of a call of 50 to 90, they may lose a quarter of the forward (25 sentences of 2 to 56 words have 1 450
// nodes; TreeRNN, H = 128: up to 1 640), and the backward follows the forward.  TreeLSTM decides for the backward by itself,
// since the size of its workspace hangs on it.
bool trees_always_pay(int cell, int H, int n, bool backward) {
  const WalkCosts c = walk_costs(cell, H, backward && cell == kLstm);
  const float internal = (float)((n - 1) / 2), depth = ceilf(log2f(internal + 1.f));
  return tree_cost(c, internal, depth, internal) <= (cell == kLstm ? 1.f : 1.25f) * grid_cost(c, depth, internal);
}

// Chooses the shapes and says how much device memory the register images take (0: the level kernels stream the
// weights instead).
size_t plan_trees(treelstm* ctx) {
  auto& t = ctx->trees;
  auto& s = t.s;
  const int H = ctx->H, cell = ctx->cell;
  if (H > (cell == kRntn ? kRntnMaxH : 256)) return 0;
  if (cell == kRntn)
    for (int a = 0, Hp = round_up(H, 4); a <= 2 * Hp; ++a) s.chunks += pair_chunks(a, H, Hp);
  // (TreeRNN: four CTAs at least from H = 64 on: 25 trees, H = 128, forward / backward on clusters of 1, 2, 4, 8 CTAs:
  // 58.6 / 142, 60.6 / 133, 56.0 / 124, 67.2 / 122 us)
  for (int cs = cell == kRnn && H >= 64 ? 4 : 1; cs <= 16 && !t.ok; cs *= 2) t.ok = shape_fits(cell, H, cs, s);
  const bool forward = ctx->precision == TREELSTM_FP32;     // (the bf16 forward has kernels of its own)
  for (int kind = forward ? 0 : 2; kind < 3 && t.ok; ++kind) {   // forward, the same with lists kept for the backward, backward
    const bool back = kind == 2;
    TreesKernel k = back ? backward_kernel(cell, s) : forward_kernel(cell, kind == 1);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = s.cs; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(s.cs); cfg.blockDim = dim3(back ? s.bthreads : kFwdT); cfg.dynamicSmemBytes = kSmemMax;
    cfg.attrs = &at; cfg.numAttrs = 1;
    int clusters = 0;
    t.ok = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) == cudaSuccess &&
           (s.cs <= 8 || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
           cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) == cudaSuccess && clusters >= 1;
    if (back) t.clusters_bwd = clusters;
    else t.clusters = kind == 0 ? clusters : std::min(t.clusters, clusters);
  }
  if (!t.ok) { cudaGetLastError(); return 0; }
  if (forward && cell == kLstm && cudaFuncSetAttribute(k_leaves_fp32, cudaFuncAttributeMaxDynamicSharedMemorySize, kLeafSmem) != cudaSuccess) {
    cudaGetLastError();
    t.ok = false;
    return 0;
  }
  return forward ? images_bytes(ctx, 0) + images_bytes(ctx, 2) + images_bytes(ctx, 3) : 0;
}
size_t tree_backward_bytes(const treelstm* ctx) { return ctx->trees.ok ? images_bytes(ctx, 1) : 0; }

int init_trees(treelstm* ctx, unsigned char* memory, cudaStream_t stream) {
  auto& t = ctx->trees;
  if (!t.ok || ctx->precision != TREELSTM_FP32) return TREELSTM_OK;
  t.Wf = reinterpret_cast<float*>(memory);
  t.pairs = reinterpret_cast<ushort2*>(memory + images_bytes(ctx, 0));
  t.Wx = reinterpret_cast<float*>(memory + images_bytes(ctx, 0) + images_bytes(ctx, 2));
  if (ctx->cell == kRntn) k_trees_pairs<<<1, kPairsT, 0, stream>>>(ctx->H, t.pairs);
  TL_CUDA(ctx, cudaGetLastError());
  return TREELSTM_OK;
}

int pack_trees(treelstm* ctx, bool forward, bool backward, cudaStream_t stream) {
  const auto& t = ctx->trees;
  if (!t.ok) return TREELSTM_OK;
  PackParams p{};
  p.cell = ctx->cell; p.H = ctx->H; p.E = ctx->E; p.s = t.s; p.pairs = t.pairs;
  p.fwd_words = fwd_words(ctx->cell); p.bwd_words = bwd_words(ctx->cell, t.s);
  p.src = ctx->cell == kLstm ? ctx->W : ctx->Wcat;
  p.fwd = forward ? t.Wf : nullptr;
  p.leaves = forward && ctx->cell == kLstm ? t.Wx : nullptr;
  p.bwd = backward ? t.Wb : nullptr;
  if (!p.fwd && !p.bwd) return TREELSTM_OK;
  k_trees_pack<<<592, 256, 0, stream>>>(p);
  TL_CUDA(ctx, cudaGetLastError());
  return TREELSTM_OK;
}

// Forests whose tables fit shared memory; beyond that the level kernels are used.
bool trees_take(const treelstm* ctx, int n) {
  const auto& s = ctx->trees.s;
  return ctx->trees.ok && n >= 1 && n <= 32767 && leaves_hold_tables(n) && trees_smem(n, fwd_buf_words(ctx->cell, ctx->H, s)).state_words >= 0 &&
         trees_smem(n, bwd_buf_words(ctx->cell, ctx->H, s)).state_words >= 0;
}

// Clusters that a launch takes: the same number in both directions, so that the backward pass can walk what the forward pass has.
static int most_parts(const treelstm* ctx) {
  const auto& t = ctx->trees;
  int clusters = t.clusters_bwd;
  if (ctx->precision == TREELSTM_FP32) {
    if (t.clusters < clusters) clusters = t.clusters;
    if ((ctx->sm_count - 1) / t.s.cs < clusters) clusters = (ctx->sm_count - 1) / t.s.cs;   // a single scheduling CTA keeps its SM
  }
  return clusters < 1 ? 1 : (clusters > kMaxTreeClusters ? kMaxTreeClusters : clusters);
}
static int trees_parts(const treelstm* ctx, int n) {
  int clusters = most_parts(ctx);
  if (ctx->opt.max_ctas > 0 && ctx->opt.max_ctas / ctx->trees.s.cs < clusters) clusters = ctx->opt.max_ctas / ctx->trees.s.cs;
  if (clusters > n) clusters = n;                        // (a tree is a node at least)
  return clusters < 1 ? 1 : clusters;
}
// For any number of clusters, since TREELSTM_OPT_MAX_CTAS may change it, and no less for more nodes.
size_t saved_walks_bytes(const treelstm* ctx, int n) {
  if (ctx->precision != TREELSTM_FP32 || !ctx->trees.ok) return 0;
  size_t most = 0;
  n = std::min(n, 32767);
  for (int parts = most_parts(ctx); parts >= 1; --parts) most = std::max(most, parts * saved_block(saved_cap(n, parts)) + (ctx->cell == kLstm ? longer_bytes(n, parts) : 0));
  return most;
}

int launch_forward_trees(treelstm* ctx, int n, const int32_t* left, const int32_t* right, const int32_t* token, float* h,
                         float* c, bool save, void* ws, const WsLayout& lay, bool after_running, cudaStream_t stream) {
  TreesParams p = trees_params(ctx, n, left, right, token, h, c, ws, lay);
  p.W = ctx->trees.Wf;
  p.costs = walk_costs(ctx->cell, ctx->H, false);
  p.choose = !trees_always_pay(ctx->cell, ctx->H, n, false);
  const int parts = trees_parts(ctx, n);
  p.gates = save && ctx->cell == kLstm ? reinterpret_cast<float*>(static_cast<char*>(ws) + lay.gates) : nullptr;
  if (save || ctx->cell == kLstm) p.walks = {reinterpret_cast<unsigned char*>(ws) + lay.walks, saved_cap(n, parts)};
  if (ctx->cell == kLstm) {
    // As many CTAs as there are SMs, if that leaves each of them 32 ids or more: 25 sentences, H = 150, on 145 and not 115 of them 28 leaves and not 40 at most
    // (with the planning CTA's shorter climbs: forward 58.7 -> 57.8 us).
    const int slices = (ctx->H + kLeafU - 1) / kLeafU, blocks = std::max(1, (ctx->sm_count - 1) / slices);
    const int ids = std::min(kLeafIds, std::max(32, (n + blocks - 1) / blocks));
    LeafParams q{n, ctx->H, ctx->E, ctx->vocab, p.chk_counts, left, token, ctx->emb, ctx->trees.Wx, ctx->b, h, c, p.gates,
                 p.st, ctx->opt.wait_limit_kcycles * 1024, p.choose, parts, right, p.costs, p.walks, ids};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((n + ids - 1) / ids * slices + 1);
    cfg.blockDim = dim3(kLeafT); cfg.dynamicSmemBytes = kLeafSmem; cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = after_running ? 1 : 0;
    cfg.attrs = &at; cfg.numAttrs = 1;
    TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_leaves_fp32, q));
    ctx->launches += 1;
  }
  return launch_trees(ctx, forward_kernel(ctx->cell, save), p, kFwdT, parts, after_running, stream);
}

int launch_backward_trees(treelstm* ctx, cudaStream_t stream) {
  const auto& L = ctx->last;
  TreesParams p = trees_params(ctx, L.n, L.left, L.right, L.token, L.h, L.c, L.ws, L.lay);
  p.W = ctx->trees.Wb;
  p.costs = walk_costs(ctx->cell, ctx->H, true);
  p.choose = !trees_always_pay(ctx->cell, ctx->H, L.n, true);
  p.gates = reinterpret_cast<float*>(static_cast<char*>(L.ws) + L.lay.gates);
  const int parts = trees_parts(ctx, L.n);
  if (ctx->precision == TREELSTM_FP32 && L.mode == TREELSTM_PERSISTENT)
    p.walks = {reinterpret_cast<unsigned char*>(L.ws) + L.lay.walks, saved_cap(L.n, parts)};
  if (p.trace) p.trace += kTraceSlots * kTraceLevels;
  return launch_trees(ctx, backward_kernel(ctx->cell, p.s), p, p.s.bthreads, parts, true, stream);
}

int launch_rec_grads(treelstm* ctx, float* dW, float* db, float* dV, float* dEmb_rows, const int* tok_slot, cudaStream_t stream) {
  const auto& L = ctx->last;
  char* base = static_cast<char*>(L.ws);
  GradParams g{};
  g.n = L.n; g.H = ctx->H; g.K = 2 * ctx->H; g.Q = ctx->cell == kRntn ? g.K * (g.K + 1) / 2 : 0; g.R = g.Q + g.K; g.vocab = ctx->vocab;
  g.left = L.left; g.right = L.right; g.token = L.token; g.order = L.order; g.level_offset = L.level_offset;
  g.tok_slot = tok_slot; g.h = L.h;
  g.dh = reinterpret_cast<const float*>(base + L.lay.dh); g.dz = reinterpret_cast<const float*>(base + L.lay.dz);
  g.dW = dW; g.db = db; g.dV = dV; g.dEmb_rows = dEmb_rows;
  g.st = reinterpret_cast<DevStatus*>(base + L.lay.status);
  g.tiles_u = (ctx->H + GU - 1) / GU;
  g.tiles = ((g.R + GR - 1) / GR) * g.tiles_u;
  const int most = (L.n / 2 + GN - 1) / GN;               // runs of at least one chunk
  g.splits = 2 * ctx->sm_count / g.tiles;
  if (g.splits > most) g.splits = most;
  if (g.splits < 1) g.splits = 1;
  const int leaf_ctas = L.n / 16 < 64 ? L.n / 16 + 1 : 64;
  g.out = {ctx->bwd_status, expect_status(ctx, stream)};
  cudaLaunchConfig_t cfg = {};                            // (the programmatic dependent of whatever is ahead: it comes up while that ends)
  cfg.gridDim = dim3(g.tiles * g.splits + leaf_ctas); cfg.blockDim = dim3(kGT); cfg.stream = stream;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization; at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at; cfg.numAttrs = 1;
  TL_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_rec_grads, g));
  ctx->launches += 1;
  return TREELSTM_OK;
}

}  // namespace tl

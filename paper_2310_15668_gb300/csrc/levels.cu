// Exact counting of closed instances by levels of overlap.
//
// An instance is closed when its three hyperedges overlap pairwise.  Call a
// pair of hyperedges "heavy" when it shares two nodes or more.  On real and
// synthetic hypergraphs most closed instances have no heavy pair at all: they
// share one popular node.  Enumerating them one by one (the triangle kernels
// of count_split.cu) is most of the work of Algorithm "exact_motif_counting"
// (Section 3.2).  Here instances are counted as if their unread overlaps were
// 1, from sums over nodes, node pairs, heavy pairs and centres of heavy
// pairs, and only instances whose three pairs are all heavy are enumerated;
// each of them takes back what the sums counted for it.
//
// F(A, B, C, x, y, z, t) is the contribution of one closed instance {a, b, k}
// with sizes A, B, C, overlaps x = |a&b|, y = |b&k|, z = |k&a| and
// t = |a&b&k|: its motif, minus its "as if open" term at each centre (as in
// count_split.cu, whose open pairs are counted here too).  The levels:
//   0  every node v and triple of hyperedges that contain v:
//        Fs = F(A, B, C, 1, 1, 1, 1);
//      every node triple u, v, w and distinct hyperedges a > {u, w},
//      b > {u, v}, k > {v, w}:  Ft = F(A, B, C, 1, 1, 1, 0).
//      An instance is met t times in the first sum and
//      xyz - t (x + y + z) + 2 t times in the second.
//   1  every heavy pair (a, b) and hyperedge k that holds a node of a & b:
//        G1 = F(A, B, C, x, 1, 1, 1) - Fs;
//      or that holds u in a \ b and w in b \ a, once per (u, w):
//        G0 = F(A, B, C, x, 1, 1, 0) - x Ft.
//      An instance is met t and (z - t)(y - t) times.
//   2  every centre a with two heavy pairs (a, b), (a, k) and node v of
//      b & k: if v is in a,
//        K1 = F(A, B, C, x, 1, z, 1) - G1(a, b) - G1(a, k) - Fs
//             - (x - 1)(z - 1) Ft,
//      else
//        K0 = F(A, B, C, x, 1, z, 0) - z G0(a, b) - x G0(a, k) - x z Ft.
//      An instance is met t and y - t times.
//   3  every instance with three heavy pairs: F minus all the above.
// An instance with no, one or two heavy pairs is thus counted exactly by the
// levels 0 to 0, 1 and 2, and one with three by level 3.  All sums are exact
// 64-bit integers.
//
// None of the kernels of levels 0 to 2 goes over instances: they collect
// integer tables keyed by what F depends on (sizes only up to the point where
// every region state stays the same), and one last kernel turns the tables
// into motif counts.  On the Zipf hypergraphs of the benchmark 1.5 to 4 % of
// the closed instances have three heavy pairs.
//
// Measured (Zipf(1.0) members, sizes s^-2.5 on [2, 25]), 10,000 / 60,000
// hyperedges, each kernel alone, and what bounds it:
//   k_lv_fill         0.12 /  2.1 ms  reads the line graph once (HBM at 60,000)
//   k_lv_triples      0.54 / 23   ms  L1 sectors of the overlap matrix, latency
//   k_lv_many         0.56 /  8.9 ms  shared-memory multiply-adds of class pairs
//   k_lv_light        0.30 /  4.6 ms  gathers of hyperedges at unpopular nodes
//   k_lv_open         0.15 /  1.0 ms  shared atomics
//   k_lv_tri          0.21 /  0.95 ms gathers of node-pair counts
//   k_lv_few          0.12 /  0.25 ms hash probes
//   k_lv_light_pairs  0.10 /  0.28 ms the same
// They run side by side on four streams: a whole count 1.3 / 31 ms, against
// 21 / 890 ms for the triangle kernels of count_split.cu.
#include <cmath>
#include <cstring>

#include "classify.cuh"
#include "phases.cuh"

namespace mochy {
namespace {

constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;

// ---------------------------------------------------------------------------
// Arguments
// ---------------------------------------------------------------------------

// one hypergraph of a batch (a lone hypergraph is unit 0)
struct LevelUnit {
  int64_t dbase;    // first dense index (hyperedges with two heavy pairs or more)
  int64_t moff;     // first word of its overlap matrix
  int64_t mstride;  // words a row
  int64_t n_dense;
  int64_t hbase;    // first hub index
  int64_t n_hubs;   // at most kMaxHubs, those of highest degree
  int64_t hmoff;    // first entry of its hub matrix
};

// Level 2: centres of at most this many heavy pairs go pair by pair (8 and 32:
// within 5 % of 16 at 2,000 to 60,000 hyperedges).
constexpr int kFewHeavy = 16;

constexpr int kMaxHubs = 4096;   // hubs of one unit (their pair counts are a matrix)

constexpr int kTripleT = 5;   // triple intersections 0..4 kept in the table of tuples

// table of level 3: entry (t, p, q, r, a1, b1, c1) for an instance with
// x = t + p, y = t + q, z = t + r and own regions a1, b1, c1 (capped at
// t + theta + 1, from where no state changes)
struct TripleTable {
  int off[kTripleT];   // first entry for each t
  int lo[kTripleT];    // smallest p, q, r (each overlap is at least 2)
  int n[kTripleT];     // how many values of p, q, r
  int total;
};

struct LevelArgs {
  int64_t n_edges, n_nodes;
  const int64_t* eoff;
  const int32_t* enode;
  const uint8_t* esize;
  const int64_t* voff;
  const int32_t* vedge;
  const int64_t* noff;
  const uint2* nadj;
  int theta, Q, S;           // Q = theta + 3 size classes, S = largest hyperedge
  int n_units;
  const int64_t* nseg;       // [U+1] node ranges (null: one unit)
  const int64_t* eseg;       // [U+1] hyperedge ranges
  const LevelUnit* unit;     // [U]
  const int64_t* hoff;       // [E+1] heavy rows
  const int32_t* hplus;      // [E] leading entries of a row: partners after it
  const uint2* hadj;         // heavy entries (line-graph layout)
  const int32_t* many;       // rows of more than kFewHeavy heavy pairs
  const int32_t* n_many;
  const int32_t* tlist;      // rows of two later partners or more, by size class
  const int64_t* tfirst;     // [units x classes + 1] first of each class
  const int64_t* dscan;      // [E+1] dense index of a row (if it is dense)
  uint32_t* mat;             // overlaps of dense rows, 4 bits each, row < column
  const uint32_t* ncls;      // [N][Q] hyperedges of each size class holding v
  const uint16_t* ehub;      // [n_inc] hub index within the unit, 0xffff: none
  const uint64_t* hkey;      // node pairs: open addressing, 0 free
  const uint32_t* hcnt;      // [slots][CP] hyperedges of size class 2.. holding it
  uint64_t hmask;
  int CP;
  const uint32_t* hubm;      // hub x hub pair counts (CP each)
  // tables (one block per unit)
  int64_t* tab;
  int64_t tab_stride;
  int64_t o_star, o_tri, o_in1, o_out1, o_in2, o_out2, o_trip;
  int64_t n_tab;
  TripleTable tt;
  unsigned long long* okey;  // level 3 tuples outside the table
  unsigned long long* ocnt;
  uint64_t omask;
  int32_t* queue;
};

__device__ __forceinline__ int unit_of(const int64_t* seg, int n, int64_t i) {
  return n > 1 ? seg_of(seg, n, i) : 0;
}

// a pair {a, b}: is b after a in the order (heavy degree, id)?
__device__ __forceinline__ bool after(int64_t hb, int64_t b, int64_t ha, int64_t a) {
  return hb != ha ? hb > ha : b > a;
}

// first entry of the table of centres of size A (level 2): rows and columns
// are classes (x, min(B - x, theta + 2)), x = 2..A
__host__ __device__ __forceinline__ int64_t level2_at(int A, int Q) {
  // sum over s = 2..A-1 of ((s - 1) Q)^2
  const int64_t m = A - 2;
  return (int64_t)Q * Q * (m * (m + 1) * (2 * m + 1) / 6);
}

__device__ __forceinline__ int class2(int x, int B, int Q) {
  return (x - 2) * Q + min(B - x, Q - 1);
}

__device__ __forceinline__ void gadd(int64_t* p, int64_t v) {
  atomicAdd((unsigned long long*)p, (unsigned long long)v);
}

__device__ __forceinline__ bool in_sorted(const int32_t* s, int n, int32_t u) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (s[m] < u) lo = m + 1; else hi = m;
  }
  return lo < n && s[lo] == u;
}

// slot of node pair u < w, or -1
__device__ __forceinline__ int64_t find_pair(const LevelArgs& g, int32_t u, int32_t w) {
  const uint64_t key = ((uint64_t)(uint32_t)min(u, w) << 32) | (uint32_t)max(u, w);
  uint64_t s = mix64(key) & g.hmask;
  for (uint64_t probe = 0; probe <= g.hmask; ++probe) {
    const uint64_t k = __ldg(&g.hkey[s]);
    if (k == key) return (int64_t)s;
    if (k == 0ull) return -1;
    s = (s + 1) & g.hmask;
  }
  return -1;
}

// slots used for a threshold: omega_bk - 1 = 0 .. 5 - theta
__host__ __device__ inline int trip_slots(int theta) { return 6 - theta; }
// size classes of rows: 2 .. theta + 9 (from where the own region of a is at
// its cap for every x + z <= 8), and rows without node masks
__host__ __device__ inline int trip_classes(int theta) { return theta + 9; }
__host__ __device__ inline int trip_class(int A, int theta) {
  return A > kMaskedMax ? theta + 8 : min(A, theta + 9) - 2;
}

// ---------------------------------------------------------------------------
// Preparation
// ---------------------------------------------------------------------------

// What the ways of counting have to go over (see levels_pay): the sum of the
// squared line degrees, and what light nodes cost the levels, in units of 1,024.
// overlaps: the overlaps of all pairs of hyperedges together (to see how large
// they are on average).
struct Work {
  unsigned long long deg2, light_pairs, light_rows, overlaps;
};

// adds up n, one value a thread, over a block of kRowThreads
__device__ __forceinline__ void block_add(unsigned long long n, unsigned long long* out) {
  __shared__ unsigned long long part[kRowWarps];
  for (int d = 16; d; d >>= 1) n += __shfl_xor_sync(0xffffffffu, n, d);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0ull;
    for (int w = 0; w < kRowWarps; ++w) s += part[w];
    if (s) atomicAdd(out, s);
  }
  __syncthreads();   // the next call's sums
}

// heavy degrees, which rows can be in a triangle of heavy pairs, and node
// pairs of each hyperedge
__global__ void __launch_bounds__(kRowThreads)
k_lv_rows(int64_t n_edges, const int64_t* __restrict__ noff, const int32_t* __restrict__ heavy,
          const uint8_t* __restrict__ esize, int64_t* __restrict__ seg_h,
          int64_t* __restrict__ seg_d, int64_t* __restrict__ seg_p, Work* __restrict__ work) {
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t deg = 0;
  if (a < n_edges) {
    const int64_t h = heavy[a], A = esize[a];
    deg = noff[a + 1] - noff[a];
    seg_h[a] = h;
    seg_d[a] = h >= 2 ? 1 : 0;
    seg_p[a] = A * (A - 1) / 2;
  }
  block_add((unsigned long long)(deg * deg), &work->deg2);
}

// The light work of a node in d hyperedges, with `others` other members in all
// and `many` heavy pairs at those of its hyperedges that have more than
// kFewHeavy: d d' summed over the nodes d' that it shares a hyperedge with (as
// if they were alike), and d / 2 for each of the heavy pairs.
struct LightWork {
  unsigned long long pairs = 0ull, rows = 0ull, overlaps = 0ull;
  __device__ __forceinline__ void add(int64_t d, int64_t others, int64_t many) {
    pairs += ((unsigned long long)d * d * (others + d) / 2 + 512) >> 10;
    rows += ((unsigned long long)d * many / 2 + 512) >> 10;
  }
};

// warp per node: hyperedges of each size class that hold it, whether it is a
// hub, and a bound on its neighbours in the node graph
__global__ void __launch_bounds__(kRowThreads)
k_lv_nodes(LevelArgs g, int hub_deg, const int32_t* __restrict__ heavy,
           uint32_t* __restrict__ ncls, int64_t* __restrict__ seg_b, int64_t* __restrict__ seg_n,
           Work* __restrict__ work) {
  LightWork light;   // of lane 0
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t v = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5); v < g.n_nodes; v += nw) {
    const int64_t b = g.voff[v], e = g.voff[v + 1];
    const bool hub = e - b >= hub_deg;
    int64_t others = 0, many = 0;
    uint32_t mine = 0;   // count of class `lane` (Q <= 32)
    for (int64_t p0 = b; p0 < e; p0 += 32) {
      const int64_t p = p0 + lane;
      const int32_t k = p < e ? g.vedge[p] : 0;
      const int s = p < e ? g.esize[k] : 0;
      others += s > 0 ? s - 1 : 0;
      if (!hub && p < e) {
        const int32_t h = heavy[k];
        many += h > kFewHeavy ? h : 0;
      }
      const int c = s > 0 ? min(s, g.Q) - 1 : -1;
      for (int q = 0; q < g.Q; ++q) {
        const int n = __popc(__ballot_sync(0xffffffffu, c == q));
        if (lane == q) mine += n;
      }
    }
    for (int d = 16; d; d >>= 1) others += __shfl_xor_sync(0xffffffffu, others, d);
    if (!hub)
      for (int d = 16; d; d >>= 1) many += __shfl_xor_sync(0xffffffffu, many, d);
    if (lane < g.Q) ncls[v * g.Q + lane] = mine;
    if (lane == 0) {
      seg_b[v] = hub ? 1 : 0;
      seg_n[v] = others;
      if (!hub) light.add(e - b, others, many);
      light.overlaps += (unsigned long long)(e - b) * (unsigned long long)(e - b - 1) / 2;
    }
  }
  // the sums of the warps, three neighbouring counters
  __shared__ unsigned long long part[3][kRowWarps];
  if (lane == 0) {
    part[0][threadIdx.x >> 5] = light.pairs;
    part[1][threadIdx.x >> 5] = light.rows;
    part[2][threadIdx.x >> 5] = light.overlaps;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    unsigned long long s = 0ull;
    for (int w = 0; w < kRowWarps; ++w) s += part[threadIdx.x][w];
    if (s) atomicAdd(&work->light_pairs + threadIdx.x, s);
  }
}

// Units of more hubs than kMaxHubs keep those of highest degree, the lower id
// first among equals: with ids in another order than by popularity, the first
// kMaxHubs by id would leave popular nodes among the light ones, whose node
// pairs cost the product of their degrees (k_lv_light_pairs).  The nodes are
// sorted by degree, then (a batch) stably by unit.
__global__ void k_lv_degree_keys(LevelArgs g, uint32_t* __restrict__ key,
                                 uint32_t* __restrict__ val) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= g.n_nodes) return;
  key[v] = ~(uint32_t)(g.voff[v + 1] - g.voff[v]);
  val[v] = (uint32_t)v;
}

__global__ void k_lv_unit_keys(LevelArgs g, const uint32_t* __restrict__ val,
                               uint32_t* __restrict__ key) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < g.n_nodes) key[i] = (uint32_t)unit_of(g.nseg, g.n_units, val[i]);
}

__global__ void k_lv_pick_hubs(LevelArgs g, const uint32_t* __restrict__ val, int hub_deg,
                               int64_t* __restrict__ seg_b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.n_nodes) return;
  const int64_t v = val[i];
  const int64_t rank = i - (g.n_units > 1 ? g.nseg[unit_of(g.nseg, g.n_units, v)] : 0);
  seg_b[v] = rank < kMaxHubs && g.voff[v + 1] - g.voff[v] >= hub_deg ? 1 : 0;
}

// is node v a hub?  bscan: the scan of the hubs' flags (one entry follows the
// last node's)
__device__ __forceinline__ bool is_hub(const int64_t* __restrict__ bscan, int64_t v) {
  return bscan[v + 1] != bscan[v];
}

// The light work again, when the hubs are not all nodes of that degree (thread
// per hyperedge): with l the degrees of its light nodes together, l^2 / 2 pairs
// of hyperedges, and h l / 2 around its heavy pairs h.
__global__ void __launch_bounds__(kRowThreads)
k_lv_light_work(LevelArgs g, const int32_t* __restrict__ heavy, const int64_t* __restrict__ bscan,
                Work* __restrict__ work) {
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long l = 0ull, h = 0ull;
  if (a < g.n_edges) {
    for (int64_t q = g.eoff[a]; q < g.eoff[a + 1]; ++q) {
      const int32_t v = g.enode[q];
      if (!is_hub(bscan, v)) l += (unsigned long long)(g.voff[v + 1] - g.voff[v]);
    }
    h = (unsigned long long)heavy[a];
  }
  block_add((l * l / 2 + 512) >> 10, &work->light_pairs);
  block_add(h > kFewHeavy ? (h * l / 2 + 512) >> 10 : 0ull, &work->light_rows);
}

// totals the host needs: [h, pairs, neighbours] then per unit the first dense
// index and the first hub index (U + 1 each), then the work
__global__ void k_lv_totals(LevelArgs g, const int64_t* __restrict__ S, int64_t o_d, int64_t o_p,
                            int64_t o_b, int64_t o_n, int64_t end, const Work* __restrict__ work,
                            int64_t* __restrict__ out) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u == 0) {
    out[0] = S[o_d] - S[0];
    out[1] = S[o_b] - S[o_p];
    out[2] = S[end] - S[o_n];
    int64_t* w = out + 3 + 2 * (g.n_units + 1);
    w[0] = (int64_t)work->deg2;
    w[1] = (int64_t)work->light_pairs;
    w[2] = (int64_t)work->light_rows;
    w[3] = (int64_t)work->overlaps;
  }
  if (u > g.n_units) return;
  const int64_t e = g.n_units > 1 ? g.eseg[u] : (u ? g.n_edges : 0);
  const int64_t n = g.n_units > 1 ? g.nseg[u] : (u ? g.n_nodes : 0);
  out[3 + u] = S[o_d + e] - S[o_d];
  out[3 + g.n_units + 1 + u] = S[o_b + n] - S[o_b];
}

// warp per row: heavy entries, partners after the row (in the order of heavy
// degree, then id) first, ascending by id, the others from the end
__global__ void __launch_bounds__(kRowThreads)
k_lv_fill(LevelArgs g, uint2* __restrict__ hadj, int32_t* __restrict__ hplus,
          int32_t* __restrict__ many, int32_t* __restrict__ n_many, int32_t* __restrict__ tlist,
          uint32_t* __restrict__ tcount) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t a = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5); a < g.n_edges; a += nw) {
    const int64_t hb = g.hoff[a], he = g.hoff[a + 1];
    int64_t front = hb, back = he;
    if (he > hb) {
      const int64_t rb = g.noff[a], re = g.noff[a + 1];
      const int A = (int)(g.eoff[a + 1] - g.eoff[a]);
      for (int64_t p0 = rb; p0 < re; p0 += 128) {
        uint2 e[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int64_t p = p0 + 32 * r + lane;
          e[r] = p < re ? g.nadj[p] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const bool heavy = entry_omega(e[r].y, A) >= 2;
          if (!__any_sync(0xffffffffu, heavy)) continue;
          bool plus = false;
          if (heavy) {
            const int64_t b = ent_id(e[r]);
            plus = after(g.hoff[b + 1] - g.hoff[b], b, he - hb, a);
          }
          const unsigned mp = __ballot_sync(0xffffffffu, heavy && plus);
          const unsigned mm = __ballot_sync(0xffffffffu, heavy && !plus);
          if (heavy && plus) hadj[front + __popc(mp & lt)] = e[r];
          if (heavy && !plus) hadj[back - 1 - __popc(mm & lt)] = e[r];
          front += __popc(mp);
          back -= __popc(mm);
        }
      }
    }
    if (lane == 0) {
      hplus[a] = (int32_t)(front - hb);
      if (he - hb > kFewHeavy) many[atomicAdd(n_many, 1)] = (int32_t)a;
      if (front - hb >= 2) {
        // the rows of level 3 by size class
        const int u = unit_of(g.eseg, g.n_units, a);
        const int cls = trip_class((int)(g.eoff[a + 1] - g.eoff[a]), g.theta);
        const uint32_t at = atomicAdd(&tcount[u * trip_classes(g.theta) + cls], 1u);
        tlist[(int64_t)cls * g.n_edges + (g.n_units > 1 ? g.eseg[u] : 0) + at] = (int32_t)a;
      }
    }
  }
}

// warp per row: overlaps of its heavy pairs into the matrix of its unit, at
// (smaller id, larger id): min(omega - 1, 15), 0 for pairs that are not heavy
__global__ void __launch_bounds__(kRowThreads) k_lv_matrix(LevelArgs g) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t a = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5); a < g.n_edges; a += nw) {
    const int64_t hb = g.hoff[a];
    if (g.hoff[a + 1] - hb < 2) continue;
    const int n = g.hplus[a];
    if (n == 0) continue;
    const LevelUnit un = g.unit[unit_of(g.eseg, g.n_units, a)];
    const int A = (int)(g.eoff[a + 1] - g.eoff[a]);
    const int64_t ia = g.dscan[a] - un.dbase;
    for (int q = lane; q < n; q += 32) {
      const uint2 e = g.hadj[hb + q];
      const int64_t b = ent_id(e);
      const int64_t ib = g.dscan[b] - un.dbase;   // dense: its heavy degree is at least a's
      const uint32_t om = min(entry_omega(e.y, A) - 1, 15);
      const int64_t r = b > a ? ia : ib, c = b > a ? ib : ia;
      atomicOr(&g.mat[un.moff + r * un.mstride + (c >> 3)], om << (4 * (int)(c & 7)));
    }
  }
}

// warp per hyperedge: its node pairs into the pair table, hub indices of its
// nodes
__global__ void __launch_bounds__(kRowThreads)
k_lv_pairs(LevelArgs g, const int64_t* __restrict__ bscan, uint64_t* __restrict__ hkey,
           uint32_t* __restrict__ hcnt, uint16_t* __restrict__ ehub) {
  __shared__ int32_t nodes[kRowWarps][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t a = (int64_t)blockIdx.x * kRowWarps + warp; a < g.n_edges; a += nw) {
    const int64_t eb = g.eoff[a];
    const int A = (int)(g.eoff[a + 1] - eb);
    const int64_t hbase = g.n_units > 1 ? g.unit[unit_of(g.eseg, g.n_units, a)].hbase : 0;
    for (int q = lane; q < A; q += 32) {
      const int32_t v = g.enode[eb + q];
      nodes[warp][q] = v;
      ehub[eb + q] = is_hub(bscan, v) ? (uint16_t)(bscan[v] - bscan[0] - hbase) : (uint16_t)0xffff;
    }
    __syncwarp();
    const int c = min(A, g.Q) - 2;
    // pair index n of (i, j), i < j: column j holds j pairs
    const int np = A * (A - 1) / 2;
    for (int n = lane; n < np; n += 32) {
      int j = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)n)) * 0.5f);
      while (j * (j - 1) / 2 > n) --j;
      while ((j + 1) * j / 2 <= n) ++j;
      const int i = n - j * (j - 1) / 2;
      const uint64_t key = ((uint64_t)(uint32_t)nodes[warp][i] << 32) | (uint32_t)nodes[warp][j];
      uint64_t s = mix64(key) & g.hmask;
      for (uint64_t probe = 0; probe <= g.hmask; ++probe) {
        unsigned long long k = hkey[s];
        if (k == 0ull) k = atomicCAS((unsigned long long*)&hkey[s], 0ull, (unsigned long long)key);
        if (k == 0ull || k == key) {
          atomicAdd(&hcnt[s * g.CP + c], 1u);
          break;
        }
        s = (s + 1) & g.hmask;
      }
    }
    __syncwarp();
  }
}

// node graph, each pair kept at its node of lower (degree, id)
__global__ void k_lv_orient(LevelArgs g, const int64_t* __restrict__ nscan,
                            uint32_t* __restrict__ cursor, uint2* __restrict__ adj) {
  const int64_t n = (int64_t)g.hmask + 1;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = g.hkey[s];
    if (!k) continue;
    const int32_t u = (int32_t)(k >> 32), w = (int32_t)(k & 0xffffffffu);
    const bool up = after(g.voff[w + 1] - g.voff[w], w, g.voff[u + 1] - g.voff[u], u);
    const int32_t low = up ? u : w, high = up ? w : u;
    const uint32_t at = atomicAdd(&cursor[low], 1u);
    adj[nscan[low] - nscan[0] + at] = make_uint2((uint32_t)high, (uint32_t)s);
  }
}

// ---------------------------------------------------------------------------
// Level 0
// ---------------------------------------------------------------------------

__device__ __forceinline__ int sorted3(int a, int b, int c, int Q) {
  const int lo = min(a, min(b, c)), hi = max(a, max(b, c));
  return (lo * Q + (a + b + c - lo - hi)) * Q + hi;
}

// triples of the hyperedges of each node, by size classes
__global__ void __launch_bounds__(kRowThreads) k_lv_star(LevelArgs g) {
  extern __shared__ unsigned long long acc[];
  const int Q = g.Q, n3 = Q * Q * Q;
  for (int q = threadIdx.x; q < n3; q += blockDim.x) acc[q] = 0ull;
  __syncthreads();
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < g.n_nodes;
       v += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t* n = g.ncls + v * Q;
    int64_t* out = g.n_units > 1 ? g.tab + unit_of(g.nseg, g.n_units, v) * g.tab_stride + g.o_star
                                 : nullptr;
    for (int i = 0; i < Q; ++i) {
      const long long a = n[i];
      if (!a) continue;
      for (int j = i; j < Q; ++j) {
        const long long b = n[j];
        if (!b) continue;
        for (int k = j; k < Q; ++k) {
          const long long c = n[k];
          if (!c) continue;
          unsigned long long m;
          if (i == j && j == k) {
            // a (a - 1) (a - 2) / 6, dividing before the product grows
            const unsigned long long p = (unsigned long long)(a * (a - 1) / 2);
            const unsigned long long r = (unsigned long long)(a >= 2 ? a - 2 : 0);
            m = p % 3 == 0 ? p / 3 * r : p * (r / 3) + p * (r % 3) / 3;
          } else if (i == j) {
            m = (unsigned long long)(a * (a - 1) / 2) * c;
          } else if (j == k) {
            m = (unsigned long long)(b * (b - 1) / 2) * a;
          } else {
            m = (unsigned long long)(a * b) * c;
          }
          if (!m) continue;
          if (out) gadd(out + (i * Q + j) * Q + k, (int64_t)m);
          else shared_bin_add(acc, (i * Q + j) * Q + k, (long long)m);
        }
      }
    }
  }
  __syncthreads();
  if (g.n_units == 1)
    for (int q = threadIdx.x; q < n3; q += blockDim.x)
      if (acc[q]) gadd(g.tab + g.o_star + q, (int64_t)acc[q]);
}

// node triples with a hyperedge for each of their pairs: warp per node u,
// lanes over the pairs of its later neighbours; then, for the choices that
// are not three distinct hyperedges, warp per hyperedge a and node pair p of
// it: (|a| - 2) hyperedges of p meet a taken twice, and a taken three times
// is counted 3 - 1 times too often among those
__global__ void __launch_bounds__(kRowThreads)
k_lv_tri(LevelArgs g, const int64_t* __restrict__ nscan, const uint32_t* __restrict__ cursor,
         const uint2* __restrict__ adj) {
  extern __shared__ unsigned long long acc[];
  __shared__ int32_t nodes[kRowWarps][64];
  const int Q = g.Q, n3 = Q * Q * Q, nc = Q - 1;   // size classes 2..Q
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = threadIdx.x; q < n3; q += blockDim.x) acc[q] = 0ull;
  __syncthreads();
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  const int64_t w0 = (int64_t)blockIdx.x * kRowWarps + warp;
  auto add = [&](int64_t* out, int i, int j, int k, long long m) {
    const int at = sorted3(i + 1, j + 1, k + 1, Q);
    if (out) gadd(out + at, m);
    else shared_bin_add(acc, at, m);
  };
  for (int64_t u = w0; u < g.n_nodes; u += nw) {
    const int n = (int)cursor[u];
    if (n < 2) continue;
    const uint2* L = adj + (nscan[u] - nscan[0]);
    int64_t* out = g.n_units > 1 ? g.tab + unit_of(g.nseg, g.n_units, u) * g.tab_stride + g.o_tri
                                 : nullptr;
    for (int i0 = 0; i0 + 1 < n; i0 += 32) {
      // pairs (i, j), i in [i0, i0 + 32), j > i, lanes over all of them
      const int ni = min(32, n - 1 - i0), w = n - 1 - i0;   // i = i0 has w partners
      const int np = ni * w - ni * (ni - 1) / 2;
      for (int m = lane; m < np; m += 32) {
        int i = (int)((2.0f * w + 1.0f - sqrtf((2.0f * w + 1.0f) * (2.0f * w + 1.0f) - 8.0f * m)) *
                      0.5f);
        i = max(min(i, ni - 1), 0);
        while (i > 0 && i * w - i * (i - 1) / 2 > m) --i;
        while (i + 1 < ni && (i + 1) * w - (i + 1) * i / 2 <= m) ++i;
        const int j = i + 1 + (m - (i * w - i * (i - 1) / 2));
        const uint2 ei = L[i0 + i], ej = L[i0 + j];
        const int64_t s = find_pair(g, (int32_t)ei.x, (int32_t)ej.x);
        if (s < 0) continue;
        const uint32_t* mi = g.hcnt + (uint64_t)ei.y * g.CP;
        const uint32_t* mj = g.hcnt + (uint64_t)ej.y * g.CP;
        const uint32_t* mk = g.hcnt + (uint64_t)s * g.CP;
        for (int a = 0; a < nc; ++a) {
          const long long na = mi[a];
          if (!na) continue;
          for (int b = 0; b < nc; ++b) {
            const long long nb = mj[b];
            if (!nb) continue;
            for (int c = 0; c < nc; ++c) {
              const long long k = mk[c];
              if (k) add(out, a, b, c, na * nb * k);
            }
          }
        }
      }
    }
  }
  for (int64_t a = w0; a < g.n_edges; a += nw) {
    const int64_t eb = g.eoff[a];
    const int A = (int)(g.eoff[a + 1] - eb);
    if (A < 3) continue;
    for (int q = lane; q < A; q += 32) nodes[warp][q] = g.enode[eb + q];
    __syncwarp();
    int64_t* out = g.n_units > 1 ? g.tab + unit_of(g.eseg, g.n_units, a) * g.tab_stride + g.o_tri
                                 : nullptr;
    const int ca = min(A, Q) - 2;
    long long sum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = 0; i + 1 < A; ++i)
      for (int j = i + 1 + lane; j < A; j += 32) {
        const int64_t s = find_pair(g, nodes[warp][i], nodes[warp][j]);
        if (s < 0) continue;
        const uint32_t* m = g.hcnt + (uint64_t)s * g.CP;
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (c < nc) sum[c] += m[c];
      }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (c >= nc) break;
      long long v = sum[c];
      for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
      if (lane == 0) {
        v = -v * (A - 2);
        if (c == ca) v += 2ll * A * (A - 1) * (A - 2) / 6;
        if (v) add(out, ca, ca, c, v);
      }
    }
  }
  __syncthreads();
  if (g.n_units == 1)
    for (int q = threadIdx.x; q < n3; q += blockDim.x)
      if (acc[q]) gadd(g.tab + g.o_tri + q, (int64_t)acc[q]);
}

// ---------------------------------------------------------------------------
// Levels 1 and 2.
//
// Level 1 needs, per heavy pair (a, b) with T = a & b, the size classes of
// the hyperedges of T's nodes (less a and b), and
//   out(a, b) = sum of M_uw over u in a \ b, w in b \ a,
// M_uw the hyperedges that hold u and w.  Over all u in a, w in b, u != w,
// take off those with u in T (rs_b(T)) or w in T (rs_a(T)) and add those with
// both (MT(T)) back, where rs_a(T) = sum over i in T, j in a of M_ij.  Nodes of
// high degree ("hubs") and the others ("light") are summed apart: from row a
//   D(a, b) = sum over hubs w of b of R_a[w] - 2 rs_a(T) + MT(T),
//   R_a[w] = sum over hubs u of a of M_uw + 2 sum over light u of a of M_uw,
// and D(a, b) + D(b, a) + 2 (light-light part) = 2 out(a, b).  So a row only
// looks its partners' hubs up in a table of its own, R_a, and the light-light
// part, whose M_uw are few, is found from the node pairs (k_lv_light_pairs).
// The level 1 tables hold both directions and are halved at the end.
//
// Rows of many heavy pairs (k_lv_many) need the partners one by one only to
// count them by (node, class); both levels are then sums over these counts.
// ---------------------------------------------------------------------------
constexpr int kL1Rows = 8;   // overlaps 2..9 have their table rows in shared memory

// level 1 table entry of a heavy pair with overlap x (class index to be added)
__device__ __forceinline__ int level1_at(int x, int A, int B, int Q) {
  const int da = min(A - x, Q - 1), db = min(B - x, Q - 1);
  return (((x - 2) * Q + min(da, db)) * Q + max(da, db)) * Q;
}

constexpr int kMatMax = 16;   // stands for 16 or more

// overlap of dense rows b and k (ids) from the matrix, 0 when not heavy
__device__ __forceinline__ int mat_omega(const LevelArgs& g, const LevelUnit& un, int64_t b,
                                         int64_t k) {
  const int64_t ib = g.dscan[min(b, k)] - un.dbase, ik = g.dscan[max(b, k)] - un.dbase;
  const int v = (int)(__ldg(&g.mat[un.moff + ib * un.mstride + (ik >> 3)]) >> (4 * (int)(ik & 7))) & 15;
  return v ? v + 1 : 0;
}

// overlap of rows b and k (ids) with hb and hk heavy pairs: 0 when not heavy
__device__ __forceinline__ int heavy_omega(const LevelArgs& g, const LevelUnit& un, int64_t b,
                                           int64_t hb, int64_t k, int64_t hk) {
  int om = 0;
  if (hb >= 2 && hk >= 2) {
    om = mat_omega(g, un, b, k);
  } else if (hb >= 1 && hk >= 1) {
    // the row of one heavy pair: is the other its partner?
    const int64_t one = hb == 1 ? b : k, other = hb == 1 ? k : b;
    const uint2 e = g.hadj[g.hoff[one]];
    if ((int64_t)ent_id(e) == other)
      om = min(entry_omega(e.y, (int)(g.eoff[one + 1] - g.eoff[one])), kMatMax);
  }
  if (om == kMatMax)
    om = sorted_overlap(g.enode + g.eoff[b], (int)(g.eoff[b + 1] - g.eoff[b]),
                        g.enode + g.eoff[k], (int)(g.eoff[k + 1] - g.eoff[k]));
  return om;
}

// i < j of the n-th pair in the order (0,1), (0,2), (1,2), (0,3), ...
__device__ __forceinline__ void nth_pair(int n, int& i, int& j) {
  j = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)n)) * 0.5f);
  while (j * (j - 1) / 2 > n) --j;
  while ((j + 1) * j / 2 <= n) ++j;
  i = n - j * (j - 1) / 2;
}

// hubs x hubs: M_uw, four counts a pair (size classes from 2), per unit
__global__ void k_lv_hub_matrix(LevelArgs g, const int64_t* __restrict__ bscan,
                                uint32_t* __restrict__ hubm) {
  const int64_t n = (int64_t)g.hmask + 1;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = g.hkey[s];
    if (!k) continue;
    const int32_t u = (int32_t)(k >> 32), w = (int32_t)(k & 0xffffffffu);
    if (!is_hub(bscan, u) || !is_hub(bscan, w)) continue;
    const LevelUnit un = g.unit[unit_of(g.nseg, g.n_units, u)];
    const int64_t hu = bscan[u] - bscan[0] - un.hbase, hw = bscan[w] - bscan[0] - un.hbase;
    for (int c = 0; c < g.CP; ++c) {
      const uint32_t m = g.hcnt[(uint64_t)s * g.CP + c];
      hubm[(un.hmoff + hu * un.n_hubs + hw) * g.CP + c] = m;
      hubm[(un.hmoff + hw * un.n_hubs + hu) * g.CP + c] = m;
    }
  }
}

// Rows of few heavy pairs, warp per row.  Level 1: eight lanes per partner,
// over the node pairs (u, w) that D(a, b) sums; level 2: lanes over the pairs
// of partners.
template <int kQ>
__global__ void __launch_bounds__(kRowThreads) k_lv_few(LevelArgs g) {
  constexpr int nc = kQ - 1;
  constexpr int kCell = kQ * kQ * kQ;   // (dmin, dmax, class) of one overlap
  extern __shared__ unsigned long long acc[];   // in, then out: [kL1Rows][kCell]
  __shared__ uint2 ent[kRowWarps][kFewHeavy];
  __shared__ int32_t anodes[kRowWarps][64];
  __shared__ uint8_t aflag[kRowWarps][64];      // 1: hub
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = lane >> 3, gl = lane & 7;
  const unsigned gmask = 0xffu << (8 * grp);
  const int n_sh = min(kL1Rows, g.S - 1) * kCell;
  for (int q = threadIdx.x; q < 2 * n_sh; q += blockDim.x) acc[q] = 0ull;
  __syncthreads();
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t a = (int64_t)blockIdx.x * kRowWarps + warp; a < g.n_edges; a += nw) {
    const int64_t hb = g.hoff[a];
    const int n = (int)min(g.hoff[a + 1] - hb, (int64_t)kFewHeavy + 1);
    if (n < 1 || n > kFewHeavy) continue;
    const int64_t eb = g.eoff[a];
    const int A = (int)(g.eoff[a + 1] - eb);
    const int32_t* an = anodes[warp];
    for (int q = lane; q < n; q += 32) ent[warp][q] = g.hadj[hb + q];
    for (int q = lane; q < A; q += 32) {
      anodes[warp][q] = g.enode[eb + q];
      aflag[warp][q] = g.ehub[eb + q] != 0xffff ? 1 : 0;
    }
    __syncwarp();
    int64_t* tab = g.tab + unit_of(g.eseg, g.n_units, a) * g.tab_stride;
    for (int e0 = grp; e0 < n; e0 += 4) {
      const uint2 e = ent[warp][e0];
      const int B = ent_size(e), x = entry_omega(e.y, A);
      const int64_t bb = g.eoff[ent_id(e)];
      unsigned long long in[kQ], out[nc];
#pragma unroll
      for (int c = 0; c < kQ; ++c) in[c] = 0ull;
#pragma unroll
      for (int c = 0; c < nc; ++c) out[c] = 0ull;
      // (u, w) = nodes of a and b, flattened
      const uint32_t recip = ((1u << 20) + A - 1) / A;   // exact for indices below 63 x 63
      for (int i = gl; i < A * B; i += 8) {
        const int qb = (int)(((uint32_t)i * recip) >> 20), qa = i - qb * A;
        const int32_t w = g.enode[bb + qb], u = an[qa];
        if (u == w) {
#pragma unroll
          for (int c = 0; c < kQ; ++c) in[c] += g.ncls[(int64_t)u * kQ + c];
          continue;
        }
        const bool w_in = in_sorted(an, A, w);
        const bool w_hub = g.ehub[bb + qb] != 0xffff;
        int coef = w_hub ? 2 - aflag[warp][qa] : 0;
        if (w_in) {
          const bool u_in = A <= kMaskedMax ? ((e.y >> qa) & 1u) != 0u
                                            : in_sorted(g.enode + bb, B, u);
          coef += u_in ? -1 : -2;
        }
        if (!coef) continue;
        const int64_t s = find_pair(g, u, w);
        if (s < 0) continue;
#pragma unroll
        for (int c = 0; c < nc; ++c)
          out[c] += (long long)coef * (long long)g.hcnt[(uint64_t)s * g.CP + c];
      }
      // sums of the group; a and b themselves hold each node of a & b
#pragma unroll
      for (int c = 0; c < kQ; ++c) {
#pragma unroll
        for (int d = 4; d; d >>= 1) in[c] += __shfl_xor_sync(gmask, in[c], d);
        if (c == min(A, kQ) - 1) in[c] -= x;
        if (c == min(B, kQ) - 1) in[c] -= x;
      }
#pragma unroll
      for (int c = 0; c < nc; ++c)
#pragma unroll
        for (int d = 4; d; d >>= 1) out[c] += __shfl_xor_sync(gmask, out[c], d);
      const int cell = level1_at(x, A, B, kQ);
      const bool sh = g.n_units == 1 && x - 2 < kL1Rows;
#pragma unroll
      for (int c = 0; c < kQ; ++c) {
        if (gl == c && in[c]) {
          if (sh) shared_bin_add(acc, cell + c, in[c]);
          else gadd(tab + g.o_in1 + cell + c, in[c]);
        }
        if (c < nc && gl == c && out[c < nc ? c : 0]) {
          const unsigned long long o = out[c < nc ? c : 0];
          if (sh) shared_bin_add(acc + n_sh, cell + c + 1, o);
          else gadd(tab + g.o_out1 + cell + c + 1, o);
        }
      }
      __syncwarp(gmask);
    }
    __syncwarp();
    const int ncl = (A - 1) * kQ;
    int64_t* t_in = tab + g.o_in2 + level2_at(A, kQ);
    int64_t* t_out = tab + g.o_out2 + level2_at(A, kQ);
    const int np = n * (n - 1) / 2;
    for (int m = lane; m < np; m += 32) {
      int i, j;
      nth_pair(m, i, j);
      const uint2 eb2 = ent[warp][i], ek = ent[warp][j];
      const int64_t b = ent_id(eb2), k = ent_id(ek);
      const int B = ent_size(eb2), C = ent_size(ek);
      const int32_t* bn = g.enode + g.eoff[b];
      const int32_t* kn = g.enode + g.eoff[k];
      const int t = A <= kMaskedMax ? __popc(eb2.y & ek.y) : sorted_overlap3(an, A, bn, B, kn, C);
      const int y = sorted_overlap(bn, B, kn, C);
      const int at = class2(entry_omega(eb2.y, A), B, kQ) * ncl + class2(entry_omega(ek.y, A), C, kQ);
      if (t) gadd(t_in + at, t);
      if (y > t) gadd(t_out + at, y - t);
    }
    __syncwarp();
  }
  __syncthreads();
  if (g.n_units == 1)
    for (int q = threadIdx.x; q < n_sh; q += blockDim.x) {
      if (acc[q]) gadd(g.tab + g.o_in1 + q, (int64_t)acc[q]);
      if (acc[n_sh + q]) gadd(g.tab + g.o_out1 + q, (int64_t)acc[n_sh + q]);
    }
}

// Rows of many heavy pairs, CTA per row a.  For each node v (the nodes of a
// first, then the hubs of the unit outside a, as many at a time as fit) the
// partners of a that hold v are counted by class in shared memory: n_v[class].
// Level 2 sums n_v[i] n_v[j] over the nodes, level 1 n_v[class] times R_a[v],
// rs_a and the size classes of v.
constexpr int kManyThreads = 256;
constexpr int kManyBytes = 100 * 1024;
constexpr int kPairBytes = 40 * 1024;   // shared sums of class pairs, when they fit this

__global__ void __launch_bounds__(kManyThreads) k_lv_many(LevelArgs g) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int32_t anodes[64];
  __shared__ uint16_t ahub[64];
  __shared__ int64_t row_s;
  const int Q = g.Q, nc = Q - 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) row_s = atomicAdd(g.queue, 1);
    __syncthreads();
    if (row_s >= *g.n_many) break;
    const int64_t a = g.many[row_s];
    const int64_t hb = g.hoff[a], n = g.hoff[a + 1] - hb;
    const int64_t eb = g.eoff[a];
    const int A = (int)(g.eoff[a + 1] - eb);
    const int u = unit_of(g.eseg, g.n_units, a);
    const LevelUnit un = g.unit[u];
    const int n_hubs = (int)un.n_hubs;
    int64_t* tab = g.tab + u * g.tab_stride;
    const int ncl = (A - 1) * Q, npairs = ncl * (ncl + 1) / 2;
    // shared layout: sums of level 1 [ncl][Q] in, [ncl][nc] out; class-pair
    // sums; M_ij of a's node pairs; rs and own R of a's nodes; cells
    unsigned long long* l_in = (unsigned long long*)smem;
    unsigned long long* l_out = l_in + ncl * Q;
    unsigned long long* pacc = l_out + ncl * nc;
    const bool psh = npairs * 8 <= kPairBytes;
    uint32_t* mp = (uint32_t*)(pacc + (psh ? npairs : 0));
    int32_t* coef = (int32_t*)(mp + A * (A - 1) / 2 * nc);   // [A][nc]: R_a - 2 rs_a
    uint32_t* cell = (uint32_t*)(coef + A * nc);
    const int words = (int)((smem + kManyBytes - (unsigned char*)cell) / 4);
    for (int q = threadIdx.x; q < ncl * (Q + nc) + (psh ? npairs : 0); q += kManyThreads)
      l_in[q] = 0ull;
    if (threadIdx.x < A) {
      anodes[threadIdx.x] = g.enode[eb + threadIdx.x];
      ahub[threadIdx.x] = g.ehub[eb + threadIdx.x];
    }
    for (int q = threadIdx.x; q < A * nc; q += kManyThreads) coef[q] = 0;
    __syncthreads();
    for (int m = threadIdx.x; m < A * (A - 1) / 2; m += kManyThreads) {
      int i, j;
      nth_pair(m, i, j);
      const int64_t s = find_pair(g, anodes[i], anodes[j]);
      const bool hi = ahub[i] != 0xffff, hj = ahub[j] != 0xffff;
      for (int c = 0; c < nc; ++c) {
        const uint32_t v = s >= 0 ? g.hcnt[(uint64_t)s * g.CP + c] : 0u;
        mp[m * nc + c] = v;
        if (v) {
          // node i: R_a[i] (if a hub) takes j once or twice, rs_a[i] takes it
          atomicAdd(&coef[i * nc + c], (int)v * ((hi ? (hj ? 1 : 2) : 0) - 2));
          atomicAdd(&coef[j * nc + c], (int)v * ((hj ? (hi ? 1 : 2) : 0) - 2));
        }
      }
    }
    __syncthreads();
    int h0 = -A;   // rows -A..-1: the nodes of a; from 0 on: the hubs
    while (h0 < n_hubs) {
      const bool inside = h0 < 0;
      const int fit = words / (ncl + nc);
      const int rows = inside ? min(-h0, fit) : min(n_hubs - h0, fit);
      const int first = inside ? A + h0 : h0;
      uint32_t* R = cell + rows * ncl;   // [rows][nc] of the hubs
      for (int q = threadIdx.x; q < rows * ncl; q += kManyThreads) cell[q] = 0u;
      if (!inside) {
        // R_a of the hubs of this pass: a's hubs from the hub matrix ...
        for (int r = threadIdx.x; r < rows; r += kManyThreads)
          for (int c = 0; c < nc; ++c) R[r * nc + c] = 0u;
        __syncthreads();
        for (int w = threadIdx.x; w < rows; w += kManyThreads) {
          for (int i = 0; i < A; ++i) {
            if (ahub[i] == 0xffff) continue;
            const uint32_t* m =
                g.hubm + (un.hmoff + (int64_t)ahub[i] * n_hubs + first + w) * g.CP;
            for (int c = 0; c < nc; ++c) R[w * nc + c] += m[c];
          }
        }
        __syncthreads();
        // ... and its light nodes from their hyperedges
        for (int i = 0; i < A; ++i) {
          if (ahub[i] != 0xffff) continue;
          const int64_t vb = g.voff[anodes[i]], ve = g.voff[anodes[i] + 1];
          for (int64_t p = vb + (threadIdx.x >> 3); p < ve; p += kManyThreads / 8) {
            const int64_t k = g.vedge[p];
            const int64_t kb = g.eoff[k];
            const int C = (int)(g.eoff[k + 1] - kb);
            if (C < 2) continue;
            for (int q = threadIdx.x & 7; q < C; q += 8) {
              const int w = (int)g.ehub[kb + q] - first;
              if (w >= 0 && w < rows) atomicAdd(&R[w * nc + min(C, Q) - 2], 2u);
            }
          }
        }
      }
      __syncthreads();
      for (int64_t p = threadIdx.x; p < n; p += kManyThreads) {
        const uint2 e = g.hadj[hb + p];
        const int64_t b = ent_id(e);
        const int B = ent_size(e);
        const int cl = class2(entry_omega(e.y, A), B, Q);
        if (inside) {
          if (A <= kMaskedMax) {
            for (uint32_t m = e.y; m; m &= m - 1u) {
              const int i = __ffs(m) - 1;
              const int r = i - first;
              if (r >= 0 && r < rows) {
                atomicAdd(&cell[r * ncl + cl], 1u);
                // MT: both orders of each pair of common nodes
                for (uint32_t mj = m & (m - 1u); mj; mj &= mj - 1u) {
                  const int j = __ffs(mj) - 1;
                  const uint32_t* v = mp + (j * (j - 1) / 2 + i) * nc;
                  for (int c = 0; c < nc; ++c)
                    if (v[c]) shared_bin_add(l_out, cl * nc + c, 2ll * v[c]);
                }
              }
            }
          } else {
            const int32_t* bn = g.enode + g.eoff[b];
            for (int r = 0; r < rows; ++r)
              if (in_sorted(bn, B, anodes[first + r])) {
                atomicAdd(&cell[r * ncl + cl], 1u);
                for (int j = first + r + 1; j < A; ++j)
                  if (in_sorted(bn, B, anodes[j])) {
                    const uint32_t* v = mp + (j * (j - 1) / 2 + first + r) * nc;
                    for (int c = 0; c < nc; ++c)
                      if (v[c]) shared_bin_add(l_out, cl * nc + c, 2ll * v[c]);
                  }
              }
          }
        } else {
          const uint16_t* hub = g.ehub + g.eoff[b];
          for (int q = 0; q < B; ++q) {
            const int r = (int)hub[q] - first;
            if (r >= 0 && r < rows) atomicAdd(&cell[r * ncl + cl], 1u);
          }
        }
      }
      __syncthreads();
      if (!inside) {
        // the hubs that a holds were counted as nodes of a
        for (int i = 0; i < A; ++i) {
          const int r = (int)ahub[i] - first;
          if (ahub[i] != 0xffff && r >= 0 && r < rows)
            for (int q = threadIdx.x; q < ncl; q += kManyThreads) cell[r * ncl + q] = 0u;
        }
        __syncthreads();
      }
      // level 1
      if (inside) {
        for (int m = threadIdx.x; m < ncl * Q; m += kManyThreads) {
          const int cl = m / Q, c = m - cl * Q;
          const int x = cl / Q + 2, B = x + cl % Q;
          unsigned long long s = 0ull, o = 0ull, tot = 0ull;
          for (int r = 0; r < rows; ++r) {
            const unsigned long long v = cell[r * ncl + cl];
            if (!v) continue;
            tot += v;
            s += v * g.ncls[(int64_t)anodes[first + r] * Q + c];
            if (c > 0) o += v * (unsigned long long)(long long)coef[(first + r) * nc + c - 1];
          }
          if (c == min(A, Q) - 1) s -= tot;   // a and b hold each node of T themselves
          if (c == min(B, Q) - 1) s -= tot;
          if (s) shared_bin_add(l_in, m, (long long)s);
          if (o) shared_bin_add(l_out, cl * nc + c - 1, (long long)o);
        }
      } else {
        const int parts = max(1, kManyThreads / (ncl * nc));
        for (int w = threadIdx.x; w < ncl * nc * parts; w += kManyThreads) {
          const int part = w / (ncl * nc), m = w - part * (ncl * nc);
          const int cl = m / nc, c = m - cl * nc;
          unsigned long long o = 0ull;
          for (int r = part; r < rows; r += parts)
            o += (unsigned long long)cell[r * ncl + cl] * R[r * nc + c];
          if (o) shared_bin_add(l_out, m, (long long)o);
        }
      }
      // level 2
      int64_t* out = tab + (inside ? g.o_in2 : g.o_out2) + level2_at(A, Q);
      if (n < 32 * ncl && psh) {
        // few partners for the number of classes: warp per node, its non-empty
        // classes pair by pair
        for (int r = warp; r < rows; r += kManyThreads / 32) {
          const uint32_t* nr = cell + r * ncl;
          for (int i0 = 0; i0 < ncl; i0 += 32) {
            const uint32_t ni0 = i0 + lane < ncl ? nr[i0 + lane] : 0u;
            for (unsigned bi = __ballot_sync(0xffffffffu, ni0 != 0u); bi; bi &= bi - 1u) {
              const int i = i0 + __ffs(bi) - 1;
              const uint32_t ni = __shfl_sync(0xffffffffu, ni0, __ffs(bi) - 1);
              for (int j = i + lane; j < ncl; j += 32) {
                const unsigned long long nj = nr[j];
                const unsigned long long v =
                    j == i ? nj * (nj - 1) / 2 : (unsigned long long)ni * nj;
                if (nj && v) shared_bin_add(pacc, j * (j + 1) / 2 + i, (long long)v);
              }
            }
          }
        }
        __syncthreads();
        for (int m = threadIdx.x; m < npairs; m += kManyThreads) {
          const unsigned long long v = pacc[m];
          if (!v) continue;
          int i, j;
          nth_pair(m, i, j);   // j (j - 1) / 2 + i with i < j: shift to i <= j - 1
          gadd(out + i * ncl + j - 1, (int64_t)v);
          pacc[m] = 0ull;
        }
      } else {
        const int parts = max(1, kManyThreads / npairs);
        for (int w = threadIdx.x; w < npairs * parts; w += kManyThreads) {
          const int part = w / npairs, m = w - part * npairs;
          int i, j;
          nth_pair(m, i, j);
          --j;
          unsigned long long s = 0ull, si = 0ull;
          for (int r = part; r < rows; r += parts) {
            const uint32_t ni = cell[r * ncl + i], nj = cell[r * ncl + j];
            s += (unsigned long long)ni * nj;
            si += ni;
          }
          if (i == j) s = (s - si) / 2;
          if (s) gadd(out + i * ncl + j, (int64_t)s);
        }
      }
      __syncthreads();
      h0 = inside ? (h0 + rows < 0 ? h0 + rows : 0) : h0 + rows;
    }
    // level 1 of this row
    for (int m = threadIdx.x; m < ncl * Q; m += kManyThreads) {
      const int cl = m / Q, c = m - cl * Q;
      const int x = cl / Q + 2;
      const int at = level1_at(x, A, x + cl % Q, Q) + c;
      if (l_in[m]) gadd(tab + g.o_in1 + at, (int64_t)l_in[m]);
      if (c > 0 && l_out[cl * nc + c - 1]) gadd(tab + g.o_out1 + at, (int64_t)l_out[cl * nc + c - 1]);
    }
  }
}

// Level 1, light-light part: warp per pair of light nodes (u, w) that some
// hyperedge holds, lanes over the pairs (a, b) of their hyperedges.
__global__ void __launch_bounds__(kRowThreads)
k_lv_light_pairs(LevelArgs g, const int64_t* __restrict__ bscan) {
  extern __shared__ unsigned long long acc[];   // [kL1Rows][Q^3]
  const int lane = threadIdx.x & 31;
  const int Q = g.Q, n_sh = min(kL1Rows, g.S - 1) * Q * Q * Q;
  for (int q = threadIdx.x; q < n_sh; q += blockDim.x) acc[q] = 0ull;
  __syncthreads();
  const int64_t n = (int64_t)g.hmask + 1;
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  const int64_t w0 = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  for (int64_t s0 = w0 * 32; s0 < n; s0 += nw * 32) {
    const uint64_t k0 = s0 + lane < n ? g.hkey[s0 + lane] : 0ull;
    bool light = k0 != 0ull;
    if (light) {
      const int32_t u = (int32_t)(k0 >> 32), w = (int32_t)(k0 & 0xffffffffu);
      light = !is_hub(bscan, u) && !is_hub(bscan, w);
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, light); todo; todo &= todo - 1u) {
      const int src = __ffs(todo) - 1;
      const uint64_t k = __shfl_sync(0xffffffffu, k0, src);
      const int64_t s = s0 + src;
      const int32_t u = (int32_t)(k >> 32), w = (int32_t)(k & 0xffffffffu);
      const int64_t ub = g.voff[u], wb = g.voff[w];
      const int64_t du = g.voff[u + 1] - ub, dw = g.voff[w + 1] - wb;
      const int un_i = unit_of(g.nseg, g.n_units, u);
      const LevelUnit un = g.unit[un_i];
      int64_t* tab = g.tab + un_i * g.tab_stride + g.o_out1;
      for (int64_t i = lane; i < du * dw; i += 32) {
        const int64_t a = g.vedge[ub + i / dw], b = g.vedge[wb + i % dw];
        if (a == b) continue;
        const int x = heavy_omega(g, un, a, g.hoff[a + 1] - g.hoff[a], b, g.hoff[b + 1] - g.hoff[b]);
        if (x < 2) continue;
        const int at = level1_at(x, (int)(g.eoff[a + 1] - g.eoff[a]),
                                 (int)(g.eoff[b + 1] - g.eoff[b]), Q);
        for (int c = 1; c < Q; ++c) {
          const uint32_t m = g.hcnt[(uint64_t)s * g.CP + c - 1];
          if (!m) continue;
          if (g.n_units == 1 && x - 2 < kL1Rows) shared_bin_add(acc, at + c, 2ll * m);
          else gadd(tab + at + c, 2ll * m);
        }
      }
    }
  }
  __syncthreads();
  if (g.n_units == 1)
    for (int q = threadIdx.x; q < n_sh; q += blockDim.x)
      if (acc[q]) gadd(g.tab + g.o_out1 + q, (int64_t)acc[q]);
}

// Level 2, light nodes outside the centre, for the centres of many heavy
// pairs: warp per hyperedge b; the hyperedges k after it (in the order of
// heavy degree) that share a light node with it are listed, and every heavy
// partner a of b without that node is looked up in k's row.
constexpr int kLightList = 64;
constexpr int kLightSlices = 4;

__global__ void __launch_bounds__(kRowThreads) k_lv_light(LevelArgs g) {
  __shared__ int32_t lk[kRowWarps][kLightList];
  __shared__ uint8_t lpos[kRowWarps][kLightList];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  // a warp takes every kLightSlices-th group of 64 heavy partners of b
  for (int64_t w = (int64_t)blockIdx.x * kRowWarps + warp; w < g.n_edges * kLightSlices; w += nw) {
    const int64_t b = w % g.n_edges;
    const int slice = (int)(w / g.n_edges);
    const int64_t h0 = g.hoff[b], hb = g.hoff[b + 1] - h0;
    if (hb <= 64 * slice) continue;
    const int64_t eb = g.eoff[b];
    const int B = (int)(g.eoff[b + 1] - eb);
    const int u = unit_of(g.eseg, g.n_units, b);
    const LevelUnit un = g.unit[u];
    int64_t* tab = g.tab + u * g.tab_stride + g.o_out2;
    int n = 0;
    auto drain = [&]() {
      __syncwarp();
      for (int64_t q = 64 * slice + lane; q < hb; q += (q & 32) ? 64 * kLightSlices - 32 : 32) {
        const uint2 e = g.hadj[h0 + q];
        const int64_t a = ent_id(e);
        const int64_t ha = g.hoff[a + 1] - g.hoff[a];
        if (ha <= kFewHeavy) continue;   // counted pair by pair
        const int A = ent_size(e);
        for (int l = 0; l < n; ++l) {
          const int64_t k = lk[warp][l];
          const int pos = lpos[warp][l];
          if (a == k) continue;
          const bool v_in = B <= kMaskedMax ? ((e.y >> pos) & 1u) != 0u
                                            : in_sorted(g.enode + g.eoff[a], A, g.enode[eb + pos]);
          if (v_in) continue;              // counted as a node of a
          const int z = heavy_omega(g, un, a, ha, k, g.hoff[k + 1] - g.hoff[k]);
          if (z < 2) continue;
          const int C = (int)(g.eoff[k + 1] - g.eoff[k]);
          gadd(tab + level2_at(A, g.Q) + class2(entry_omega(e.y, B), B, g.Q) * ((A - 1) * g.Q) +
                   class2(z, C, g.Q), 1);
        }
      }
      n = 0;
      __syncwarp();
    };
    for (int q = 0; q < B; ++q) {
      if (g.ehub[eb + q] != 0xffff) continue;
      const int32_t v = g.enode[eb + q];
      const int64_t vb = g.voff[v], ve = g.voff[v + 1];
      for (int64_t p0 = vb; p0 < ve; p0 += 32) {
        const int64_t p = p0 + lane;
        const int64_t k = p < ve ? g.vedge[p] : b;
        bool take = false;
        if (k != b) {
          const int64_t hk = g.hoff[k + 1] - g.hoff[k];
          take = after(hk, k, hb, b);
        }
        const unsigned m = __ballot_sync(0xffffffffu, take);
        if (n + __popc(m) > kLightList) drain();
        if (take) {
          lk[warp][n + __popc(m & lt)] = (int32_t)k;
          lpos[warp][n + __popc(m & lt)] = (uint8_t)q;
        }
        n += __popc(m);
      }
    }
    if (n) drain();
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Motif codes and what a counted tuple adds to a histogram (in shared or in
// global memory)
// ---------------------------------------------------------------------------
struct Coder {
  const uint16_t* lut;
  int k, t1, t2;   // states: 0, then 1 + thresholds exceeded
  __device__ __forceinline__ int state(int r) const {
    return r <= 0 ? 0 : 1 + (r > t1 ? 1 : 0) + (r > t2 ? 1 : 0);
  }
  __device__ __forceinline__ int id(int a, int b, int c, int ab, int bc, int ca, int abc) const {
    int code = state(abc);
    code = code * k + state(ca);
    code = code * k + state(bc);
    code = code * k + state(ab);
    code = code * k + state(c);
    code = code * k + state(b);
    return lut[code * k + state(a)];
  }
};

// hist[id] += v: a histogram in shared memory, or one in global memory, which
// other kernels may be adding to, so by one atomic of the bin's whole width
template <bool kShared>
__device__ __forceinline__ void bin_add(unsigned long long* hist, int id, long long v) {
  if (kShared) shared_bin_add(hist, id, v);
  else atomicAdd(&hist[id], (unsigned long long)v);
}

// n closed instances of sizes A, B, C, overlaps x, y, z and t (F)
template <bool kShared>
__device__ __noinline__ void add_closed(unsigned long long* hist, const Coder& cd, int A, int B,
                                        int C, int x, int y, int z, int t, long long n) {
  if (!n) return;
  bin_add<kShared>(hist, cd.id(A - x - z + t, B - x - y + t, C - y - z + t, x - t, y - t, z - t, t),
                   n);
  if (x + z <= A) bin_add<kShared>(hist, cd.id(A - x - z, B - x, C - z, x, 0, z, 0), -n);
  if (x + y <= B) bin_add<kShared>(hist, cd.id(B - x - y, A - x, C - y, x, 0, y, 0), -n);
  if (z + y <= C) bin_add<kShared>(hist, cd.id(C - z - y, A - z, B - y, z, 0, y, 0), -n);
}

// n instances of three heavy pairs, less what the levels 0 to 2 count for them,
// into a histogram in global memory
__device__ void add_triple(unsigned long long* hist, const Coder& cd, int A, int B, int C, int x,
                           int y, int z, int t, long long n) {
  add_closed<false>(hist, cd, A, B, C, x, y, z, t, n);
  long long ft = -((long long)x * y * z - (long long)t * (x + y + z) + 2 * t);
  int a = A, b = B, c = C, xo = x, yo = y, zo = z;
  for (int i = 0; i < 3; ++i) {
    // centre a with pairs (a, b) of overlap xo and (a, c) of zo; opposite yo
    add_closed<false>(hist, cd, a, b, c, xo, 1, zo, 1, -n * t);
    add_closed<false>(hist, cd, a, b, c, xo, 1, zo, 0, -n * (yo - t));
    ft += (long long)t * (xo - 1) * (zo - 1) + (long long)(yo - t) * xo * zo;
    // pair (a, b), third member c
    const long long out = -(long long)(yo - t) * (zo - t) + (long long)(yo - t) * zo +
                          (long long)(zo - t) * yo;
    add_closed<false>(hist, cd, a, b, c, xo, 1, 1, 1, n * t);
    add_closed<false>(hist, cd, a, b, c, xo, 1, 1, 0, n * out);
    ft -= out * xo;
    // rotate: a -> b -> c -> a
    const int ta = a, tx = xo;
    a = b; b = c; c = ta;
    xo = yo; yo = zo; zo = tx;
  }
  add_closed<false>(hist, cd, A, B, C, 1, 1, 1, 1, -n * t);
  add_closed<false>(hist, cd, A, B, C, 1, 1, 1, 0, n * ft);
}

// ---------------------------------------------------------------------------
// Level 3: instances with three heavy pairs.  Each is found once, from its
// first member a in the order of heavy degree: among a's later partners,
// taken in ascending id, every pair b before k is looked up in the matrix.
//
// A warp takes 32 partners k of a row, one a lane, and goes over the partners
// b before them, staged 32 at a time.  The usual tuples are counted in a
// shared table whose index is a sum of bit fields, the matrix word, a
// popcount and one value each for b and k, so a candidate costs about a dozen
// instructions; the table is kept while rows of one size class are counted
// and then emptied into the global table of tuples.  The others (about 3 %)
// are queued per warp and worked out 32 at a time.
// ---------------------------------------------------------------------------
constexpr int kTripThreads = 1024;
constexpr int kTripWarps = kTripThreads / 32;
constexpr int kTripItems = 16;     // items a block, of kTripMin rows or more
constexpr int kTripMin = 8;
constexpr int kTripBlocks = 1;     // blocks per SM
constexpr int kTripRows = 64;      // rows taken at a time by a block
// table: [omega_bk - 1][x - 2 : 1 bit][own nodes of b past x, at most 7 : 3]
// [z - 2 : 2][own nodes of k past z, at most 7 : 3][t : 2]; omega_bk - 1 = 0 (no
// heavy pair) is counted and dropped.  x is at most 3, z at most 5, and
// omega_bk at most 6 - theta, up to which the caps of 7 are exact.
constexpr int kTripSlot = 1 << 11;           // entries per value of omega_bk - 1
constexpr int kTripShift = 13;               // of their byte addresses
constexpr uint32_t kTripFar = 1u << 20;      // marks x or z outside the table
constexpr int kTripQueue = 9 * 32;

// a tuple outside the global table, n times: into the hash of such tuples, or,
// when that is full, straight into the histogram
__device__ __noinline__ void trip_other(const LevelArgs& g, const Coder& cd,
                                        unsigned long long* hist, int unit, int t, int p, int q,
                                        int r, int a1, int b1, int c1, unsigned long long n) {
  // p, q, r and t fit 6 bits, the capped regions 7, the unit the rest
  const unsigned long long key =
      1ull + ((((((((unsigned long long)unit << 6 | t) << 6 | p) << 6 | q) << 6 | r) << 7 | a1) << 7 |
               b1) << 7 | c1);
  uint64_t s = mix64(key) & g.omask;
  for (int probe = 0; probe < 256; ++probe) {
    unsigned long long k = g.okey[s];
    if (k == 0ull) k = atomicCAS(&g.okey[s], 0ull, key);
    if (k == 0ull || k == key) {
      atomicAdd(&g.ocnt[s], n);
      return;
    }
    s = (s + 1) & g.omask;
  }
  const int x = t + p, y = t + q, z = t + r;
  add_triple(hist, cd, a1 + x + r, b1 + x + q, c1 + y + r, x, y, z, t, (long long)n);
}

// n instances of one tuple (own regions a1, b1, c1 not yet capped) into the
// global table
__device__ __forceinline__ void trip_add(const LevelArgs& g, const Coder& cd,
                                         unsigned long long* hist, int unit, int t, int p, int q,
                                         int r, int a1, int b1, int c1, unsigned long long n) {
  const int cap = t + g.theta + 1;
  a1 = min(a1, cap);
  b1 = min(b1, cap);
  c1 = min(c1, cap);
  if (t < kTripleT) {
    const int lo = g.tt.lo[t], m = g.tt.n[t];
    if (max(p, max(q, r)) < lo + m) {
      const int w = cap + 1;
      const int at = ((((((p - lo) * m + (q - lo)) * m + (r - lo)) * w + a1) * w + b1) * w) + c1;
      gadd(g.tab + unit * g.tab_stride + g.o_trip + g.tt.off[t] + at, (int64_t)n);
      return;
    }
  }
  trip_other(g, cd, hist, unit, t, p, q, r, a1, b1, c1, n);
}

// the candidate (b, k) of row a, given by their entries in its row
__device__ __noinline__ void trip_one(const LevelArgs& g, const Coder& cd,
                                      unsigned long long* hist, int unit, int64_t a, uint2 eb,
                                      uint2 ek) {
  const LevelUnit& un = g.unit[unit];
  const int64_t b = ent_id(eb), k = ent_id(ek);
  int y = mat_omega(g, un, b, k);
  if (y == 0) return;
  const int A = g.esize[a], B = ent_size(eb), C = ent_size(ek);
  const int x = entry_omega(eb.y, A), z = entry_omega(ek.y, A);
  const int32_t* bn = g.enode + g.eoff[b];
  const int32_t* kn = g.enode + g.eoff[k];
  if (y == kMatMax) y = sorted_overlap(bn, B, kn, C);
  const int t = A <= kMaskedMax ? __popc(eb.y & ek.y)
                                : sorted_overlap3(g.enode + g.eoff[a], A, bn, B, kn, C);
  trip_add(g, cd, hist, unit, t, x - t, y - t, z - t, A - x - z + t, B - x - y + t, C - y - z + t,
           1ull);
}

// first rows of the classes: exclusive sums of the counts of units x classes
__global__ void __launch_bounds__(1024) k_lv_classes(const uint32_t* __restrict__ count, int n,
                                                     int64_t* __restrict__ first) {
  __shared__ int64_t ws[34];
  int64_t carry = 0;
  for (int base = 0; base < n; base += blockDim.x) {
    const int i = base + threadIdx.x;
    int64_t total;
    const int64_t ex = block_scan_i64(i < n ? count[i] : 0, ws, &total);
    if (i < n) first[i] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) first[n] = carry;
}

__global__ void __launch_bounds__(kTripThreads, kTripBlocks) k_lv_triples(LevelArgs g, Coder cd,
                                                                  unsigned long long* hist_out,
                                                                  int n_bins) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slots = trip_slots(g.theta), ncls = trip_classes(g.theta);
  const int entries = slots * kTripSlot;
  uint4* s_b = (uint4*)smem + warp * 32;    // staged partners b
  uint32_t* s_q = (uint32_t*)(smem + kTripWarps * 512) + warp * kTripQueue;
  uint32_t* table = (uint32_t*)(smem + kTripWarps * (512 + kTripQueue * 4));
  __shared__ int32_t s_row[kTripRows], s_n[kTripRows];
  __shared__ int s_blk[kTripRows + 1];
  __shared__ int64_t s_item, s_seg[3];
  __shared__ int s_take, s_next, s_segi;
  __shared__ unsigned long long s_pairs;
  __shared__ uint32_t s_qn[kTripWarps];
  const uint32_t my_table = (uint32_t)__cvta_generic_to_shared(table);
  const uint32_t far_at = (uint32_t)slots << kTripShift;
  for (int q = threadIdx.x; q < entries; q += kTripThreads) table[q] = 0u;
  if (lane == 0) s_qn[warp] = 0u;
  const int n_seg = g.n_units * ncls;
  const int64_t n_rows = g.tfirst[n_seg];
  // rows per item: kTripItems items a block
  const int per = (int)max((int64_t)kTripMin, min((int64_t)kTripRows, n_rows / ((int64_t)gridDim.x * kTripItems)));
  int cur = -1, unit = 0;         // segment whose counts the table holds
  unsigned long long done = 0;    // pairs counted since it was emptied
  auto flush = [&]() {
    __syncthreads();
    if (cur >= 0) {
      const int A = cur % ncls + 2;   // its size class
      unsigned long long* hist = hist_out + (int64_t)unit * n_bins;
      for (int q = threadIdx.x; q < entries; q += kTripThreads) {
        const uint32_t n = table[q];
        table[q] = 0u;
        const int y = (q >> 11) + 1;
        if (!n || y < 2) continue;
        const int x = (q >> 10 & 1) + 2, d = q >> 7 & 7, z = (q >> 5 & 3) + 2, e = q >> 2 & 7;
        const int t = q & 3, o = y - t;
        trip_add(g, cd, hist, unit, t, x - t, o, z - t, A - x - z + t, d - o, e - o, n);
      }
    }
    done = 0;
    __syncthreads();
  };
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = (int64_t)atomicAdd(g.queue + 1, 1) * per;
    __syncthreads();
    int64_t r0 = s_item;
    const int64_t end = min(r0 + per, n_rows);
    if (r0 >= n_rows) break;
    while (r0 < end) {
      // the segment (unit, class) of row r0, and the rows of this pass: of one
      // segment, and few enough for the table's 32-bit counts
      __syncthreads();
      if (threadIdx.x == 0) {
        s_segi = seg_of(g.tfirst, n_seg, r0);
        s_next = 0;
      }
      __syncthreads();
      const int seg = s_segi, cls = seg % ncls, u = seg / ncls;
      if (seg != cur) {
        flush();
        cur = seg;
        unit = u;
      }
      const int64_t first = g.tfirst[seg];
      const int want = (int)(min(end, g.tfirst[seg + 1]) - r0);
      if (warp == 0) {
        int blk = 0;
        unsigned long long pairs = 0;
        int take = 0;
        for (int q0 = 0; q0 < want; q0 += 32) {
          const int q = q0 + lane;
          int n = 0;
          if (q < want) {
            const int64_t at = (int64_t)cls * g.n_edges + (g.n_units > 1 ? g.eseg[u] : 0) +
                               (r0 - first) + q;
            const int32_t a = g.tlist[at];
            n = g.hplus[a];
            s_row[q] = a;
            s_n[q] = n;
          }
          int b = (n + 31) >> 5;
          unsigned long long p = (unsigned long long)n * (unsigned)n / 2;
          for (int d = 1; d < 32; d <<= 1) {
            const int ob = __shfl_up_sync(0xffffffffu, b, d);
            const unsigned long long op = __shfl_up_sync(0xffffffffu, p, d);
            if (lane >= d) {
              b += ob;
              p += op;
            }
          }
          if (q < want) s_blk[q + 1] = blk + b;
          const bool fits = q < want && (pairs + p < (1ull << 32) || q == 0);
          const int k = __popc(__ballot_sync(0xffffffffu, fits));
          take += k;
          blk += __shfl_sync(0xffffffffu, b, 31);
          if (k > 0) pairs += __shfl_sync(0xffffffffu, p, k - 1);
          if (k < min(32, want - q0)) break;
        }
        if (lane == 0) {
          s_blk[0] = 0;
          s_take = take;
          s_pairs = pairs;
        }
      }
      __syncthreads();
      const int take = s_take;
      if (done + s_pairs >= (1ull << 32)) flush();
      done += s_pairs;
      const LevelUnit& un = g.unit[u];
      const uint32_t* mat = g.mat + un.moff;
      const int64_t dbase = un.dbase;
      const uint32_t row_bytes = (uint32_t)(4 * un.mstride);
      unsigned long long* hist = hist_out + (int64_t)u * n_bins;
      const int n_work = s_blk[take];
      const bool masked = cls < ncls - 1;
      while (true) {
        int w = 0;
        if (lane == 0) w = atomicAdd(&s_next, 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= n_work) break;
        int ri = 0;
        for (int hi = take; hi - ri > 1;) {
          const int m = (ri + hi) >> 1;
          if (s_blk[m] <= w) ri = m; else hi = m;
        }
        const int64_t a = s_row[ri];
        const int n = s_n[ri];
        const uint2* L = g.hadj + g.hoff[a];
        // the row's last blocks first: they are the longest
        const int blk = s_blk[ri + 1] - 1 - w, k0 = blk * 32, kp = k0 + lane;
        const bool has = kp < n;
        const uint2 ek = has ? L[kp] : make_uint2(0u, 0u);
        if (!masked) {
          for (int i = 0; i < min(k0 + 32, n); ++i)
            if (has && i < kp) trip_one(g, cd, hist, unit, a, L[i], ek);
          __syncwarp();
          continue;
        }
        const uint32_t mk = ek.y;
        const int ik = has ? (int)(g.dscan[ent_id(ek)] - dbase) : 0;
        const int z = __popc(mk), e = ent_size(ek) - z;
        const char* col = (const char*)(mat + (ik >> 3));
        // omega_bk - 1 (a nibble) to the bits of its table slots; 0 without k
        const uint32_t rot = (4u * (ik & 7) + 32u - kTripShift) & 31u;
        const uint32_t nib = has ? 15u << kTripShift : 0u;
        const uint32_t kk = !has ? 0u : (z > 5 ? kTripFar : (uint32_t)(z - 2) << 7) +
                                            (uint32_t)(min(e, 7) << 4);
        auto drain = [&](uint32_t from, uint32_t to) {
          // queued candidates, 32 at a time
          for (uint32_t q = from + lane; q < to; q += 32) {
            const uint32_t v = s_q[q];
            trip_one(g, cd, hist, unit, a, L[v >> 16], L[v & 0xffffu]);
          }
          __syncwarp();
        };
        for (int b0 = 0; b0 <= k0; b0 += 32) {
          {
            const int bp = b0 + lane;
            uint4 s = make_uint4(0u, 0u, 0u, 0u);
            if (bp < n) {
              const uint2 eb = L[bp];
              const int x = __popc(eb.y);
              s.x = eb.y;
              s.y = (uint32_t)(g.dscan[ent_id(eb)] - dbase);
              s.z = (x > 3 ? kTripFar : (uint32_t)(x - 2) << 12) +
                    (uint32_t)(min(ent_size(eb) - x, 7) << 9);
            }
            __syncwarp();
            s_b[lane] = s;
            __syncwarp();
          }
          const bool diag = b0 == k0;
          const int nb = min(32, n - b0);
          for (int i0 = 0; i0 < nb; i0 += 8) {
            uint32_t far = 0u;
            uint32_t word[8], at[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              const uint4 s = s_b[i0 + v];
              word[v] = __ldg((const uint32_t*)(col + (uint64_t)s.y * (uint64_t)row_bytes));
              at[v] = s.z + 4u * (uint32_t)__popc(s.x & mk);
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              uint32_t y = __funnelshift_r(word[v], word[v], rot) & nib;
              if (diag && i0 + v >= lane) y = 0u;   // only b before k
              const uint32_t addr = at[v] + kk + y;
              if (addr < far_at) {
                asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(my_table + addr) : "memory");
              } else if (y) {
                far |= 1u << v;
              }
            }
            if (__any_sync(0xffffffffu, far != 0u)) {
              for (; far; far &= far - 1u) {
                const uint32_t q = atomicAdd(&s_qn[warp], 1u);
                s_q[q] = (uint32_t)(b0 + i0 + __ffs(far) - 1) << 16 | (uint32_t)kp;
              }
              __syncwarp();
              const uint32_t qn = s_qn[warp];
              if (qn >= 32u) {
                drain(qn & 31u, qn);
                if (lane == 0) s_qn[warp] = qn & 31u;
                __syncwarp();
              }
            }
          }
        }
        const uint32_t qn = s_qn[warp];
        if (qn) {
          drain(0u, qn);
          if (lane == 0) s_qn[warp] = 0u;
          __syncwarp();
        }
      }
      r0 += take;
    }
  }
  flush();
}

// ---------------------------------------------------------------------------
// Open pairs, from the heavy rows and the nodes' size classes alone: among
// the neighbours of a centre c, those with overlap 1 are, per size class, the
// hyperedges of c's nodes less c itself and omega times each heavy partner.
// ---------------------------------------------------------------------------
constexpr int kOpenSlots = 256;   // classes (omega, own nodes up to theta + 1) of a centre

__global__ void __launch_bounds__(kRowThreads)
k_lv_open(LevelArgs g, Coder cd, unsigned long long* __restrict__ hist_out, int n_bins) {
  extern __shared__ unsigned long long hist[];
  __shared__ int32_t tkey[kRowWarps][kOpenSlots];
  __shared__ int32_t tcnt[kRowWarps][kOpenSlots];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t* key = tkey[warp];
  int32_t* cnt = tcnt[warp];
  const bool lone = g.n_units == 1;
  if (lone)
    for (int q = threadIdx.x; q < n_bins; q += blockDim.x) hist[q] = 0ull;
  __syncthreads();
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t c = (int64_t)blockIdx.x * kRowWarps + warp; c < g.n_edges; c += nw) {
    if (g.noff[c + 1] - g.noff[c] < 2) continue;
    const int64_t eb = g.eoff[c];
    const int A = (int)(g.eoff[c + 1] - eb);
    unsigned long long* out =
        lone ? hist : hist_out + (int64_t)unit_of(g.eseg, g.n_units, c) * n_bins;
    auto put = [&](int id, long long n) {
      if (lone) shared_bin_add(hist, id, n);
      else atomicAdd(&out[id], (unsigned long long)n);
    };
    for (int q = lane; q < kOpenSlots; q += 32) { key[q] = -1; cnt[q] = 0; }
    __syncwarp();
    auto insert = [&](int k, int n) {
      unsigned h = ((unsigned)k * 2654435761u) >> 24;
      for (int probe = 0; probe < kOpenSlots; ++probe) {
        const int old = atomicCAS(&key[h], -1, k);
        if (old == -1 || old == k) { atomicAdd(&cnt[h], n); return true; }
        h = (h + 1) & (kOpenSlots - 1);
      }
      return false;
    };
    // hyperedges of c's nodes by size class (lane q < Q holds class q + 1)
    int mine = 0;
    if (lane < g.Q) {
      for (int q = 0; q < A; ++q) mine += (int)g.ncls[(int64_t)g.enode[eb + q] * g.Q + lane];
      if (lane == min(A, g.Q) - 1) mine -= A;
    }
    bool overflow = false;
    for (int64_t p0 = g.hoff[c]; p0 < g.hoff[c + 1]; p0 += 32) {
      const int64_t p = p0 + lane;
      const bool has = p < g.hoff[c + 1];
      const uint2 e = has ? g.hadj[p] : make_uint2(0u, 0u);
      const int x = has ? entry_omega(e.y, A) : 0, B = has ? ent_size(e) : 0;
      if (has && !insert((x << 8) | min(B - x, g.theta + 1), 1)) overflow = true;
      for (int q = 0; q < g.Q; ++q) {
        const int s = __reduce_add_sync(0xffffffffu, has && min(B, g.Q) - 1 == q ? x : 0);
        if (lane == q) mine -= s;
      }
    }
    // neighbours with overlap 1: the sizes theta + 2 and theta + 3 are one class
    if (lane < g.Q && mine > 0 && !insert((1 << 8) | min(lane, g.theta + 1), mine)) overflow = true;
    overflow = __any_sync(0xffffffffu, overflow);
    __syncwarp();
    if (overflow) {
      // more distinct classes than the table holds: enumerate the pairs
      for (int64_t p = g.noff[c]; p < g.noff[c + 1]; ++p) {
        const uint2 ep = g.nadj[p];
        const int x1 = entry_omega(ep.y, A);
        for (int64_t q = p + 1 + lane; q < g.noff[c + 1]; q += 32) {
          const uint2 eq = g.nadj[q];
          const int x2 = entry_omega(eq.y, A);
          if (x1 + x2 > A) continue;
          put(cd.id(A - x1 - x2, ent_size(ep) - x1, ent_size(eq) - x2, x1, 0, x2, 0), 1);
        }
      }
      __syncwarp();
      continue;
    }
    // the used slots to the front, in place
    constexpr int kPer = kOpenSlots / 32;
    int32_t rk[kPer], rc[kPer];
    int used = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      rk[q] = key[lane * kPer + q];
      rc[q] = cnt[lane * kPer + q];
      used += rk[q] != -1 ? 1 : 0;
    }
    int incl = used;
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    const int P = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    int pos = incl - used;
#pragma unroll
    for (int q = 0; q < kPer; ++q)
      if (rk[q] != -1) { key[pos] = rk[q]; cnt[pos] = rc[q]; ++pos; }
    __syncwarp();
    for (int i = lane; i < P; i += 32) {
      const int x1 = key[i] >> 8, s1 = key[i] & 255;
      const long long n1 = cnt[i];
      for (int j = i; j < P; ++j) {
        const int x2 = key[j] >> 8, s2 = key[j] & 255;
        if (x1 + x2 > A) continue;
        const long long n2 = cnt[j];
        const long long n = i == j ? n1 * (n1 - 1) / 2 : n1 * n2;
        if (n) put(cd.id(A - x1 - x2, s1, s2, x1, 0, x2, 0), n);
      }
    }
    __syncwarp();
  }
  __syncthreads();
  if (lone)
    for (int q = threadIdx.x; q < n_bins; q += blockDim.x)
      if (hist[q]) atomicAdd(&hist_out[q], hist[q]);
}

// ---------------------------------------------------------------------------
// Tables to motif counts
// ---------------------------------------------------------------------------

// An entry costs up to 60 adds to few and popular bins, and most entries are 0.
// So a block first queues the non-zero entries of its chunk, then gives the
// parts of each (one add_closed, at most kParts) to threads of their own, and
// the lanes of a warp add to copies of the histogram.
// Shared atomics on equal bins bound it: 55 -> 43 us at 2,000 hyperedges, 96 ->
// 61 us at 7,001 with theta = 2, a batch of 54 as a whole 6.4 -> 5.8 ms (a
// thread an entry and one histogram a block before; a call of add_closed for
// each part at a place of its own, where the lanes part, took 350 us at 2,000).
constexpr int kFinishThreads = 256;
constexpr int kFinishChunk = 2048;   // entries of a block, at most
constexpr int kFinishCopies = 8;
constexpr int kParts = 16;

// One add_closed.  The parts are selected into it and added at one place, so
// that the lanes of a warp add together.
struct Part {
  int A, B, C, x, y, z, t;
  long long n;
};

// part p of an instance of three heavy pairs: itself (0), what the levels 1
// and 2 count for it from centre (p - 1) / 4, and what level 0 does (13, 14)
__device__ __forceinline__ Part triple_part(int p, int A, int B, int C, int x, int y, int z, int t,
                                            long long n) {
  Part o = {A, B, C, x, y, z, t, p == 0 ? n : 0};
  if (p >= 13) o = {A, B, C, 1, 1, 1, p == 13 ? 1 : 0, p == 13 ? -n * t : 0};
  long long ft = -((long long)x * y * z - (long long)t * (x + y + z) + 2 * t);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    // centre A with pairs (A, B) of overlap x and (A, C) of z; opposite y
    const long long out =
        -(long long)(y - t) * (z - t) + (long long)(y - t) * z + (long long)(z - t) * y;
    const int k = p - 1 - 4 * i;
    if (k >= 0 && k < 4)
      o = {A, B, C, x, 1, k < 2 ? z : 1, k & 1 ? 0 : 1,
           k == 0 ? -n * t : k == 1 ? -n * (y - t) : k == 2 ? n * t : n * out};
    ft += (long long)t * (x - 1) * (z - 1) + (long long)(y - t) * x * z - out * x;
    // rotate: A -> B -> C -> A
    const int ta = A, tx = x;
    A = B; B = C; C = ta;
    x = y; y = z; z = tx;
  }
  if (p == 14) o.n = n * ft;
  return o;
}

__device__ __forceinline__ Part entry_part(const LevelArgs& g, int64_t at, int part, long long n) {
  const int Q = g.Q;
  if (at >= g.o_trip) {
    int e = (int)(at - g.o_trip), t = kTripleT - 1;
    while (e < g.tt.off[t]) --t;
    e -= g.tt.off[t];
    const int m = g.tt.n[t], lo = g.tt.lo[t], c = t + g.theta + 2;
    const int c1 = e % c, b1 = e / c % c, a1 = e / (c * c) % c;
    e /= c * c * c;
    const int r = e % m + lo, q = e / m % m + lo, p = e / (m * m) + lo;
    const int x = t + p, y = t + q, z = t + r;
    return triple_part(part, a1 + x + r, b1 + x + q, c1 + y + r, x, y, z, t, n);
  }
  if (at >= g.o_in2) {
    const bool inside = at < g.o_out2;
    const int64_t e = at - (inside ? g.o_in2 : g.o_out2);
    int A = 2;
    while (A < g.S && e >= level2_at(A + 1, Q)) ++A;
    const int ncl = (A - 1) * Q;
    const int r = (int)(e - level2_at(A, Q));
    const int i = r / ncl, j = r - i * ncl;
    const int x = i / Q + 2, z = j / Q + 2, B = x + i % Q, C = z + j % Q;
    const int t = inside ? 1 : 0;
    if (part == 0) return {A, B, C, x, 1, z, t, n};
    if (part == 1) return {A, B, C, x, 1, 1, t, inside ? -n : -n * z};
    if (part == 2) return {A, C, B, z, 1, 1, t, inside ? -n : -n * x};
    if (part == 3) return {A, B, C, 1, 1, 1, t, inside ? n : n * x * z};
    return {A, B, C, 1, 1, 1, 0, part == 4 && inside ? -n * (x - 1) * (z - 1) : 0};
  }
  if (at >= g.o_in1) {
    const bool inside = at < g.o_out1;
    const int e = (int)(at - (inside ? g.o_in1 : g.o_out1));
    const int C = e % Q + 1, dB = e / Q % Q, dA = e / (Q * Q) % Q, x = e / (Q * Q * Q) + 2;
    const long long half = n / 2;   // each pair was met from both of its rows
    const int t = inside ? 1 : 0;
    if (part == 0) return {x + dA, x + dB, C, x, 1, 1, t, half};
    return {x + dA, x + dB, C, 1, 1, 1, t, part > 1 ? 0 : inside ? -half : -half * x};
  }
  const bool star = at < g.o_tri;
  const int e = (int)(at - (star ? g.o_star : g.o_tri));
  return {e / (Q * Q) + 1, e / Q % Q + 1, e % Q + 1, 1, 1, 1, star ? 1 : 0, part == 0 ? n : 0};
}

// The blocks go over the units (of one histogram each) and, within a unit, over
// the chunks of its tables, all along grid.x: grid.y ends at 65,535, and a batch
// may have more units.  The hash of tuples outside the table is one for all
// units and is gone over once, by all blocks (there are as many as it has groups
// of slots, up to eight an SM, if the tables have fewer chunks): its tuples are added to the block's histogram
// when there is one unit, else to their units' in global memory.
__global__ void __launch_bounds__(kFinishThreads)
k_lv_finish(LevelArgs g, Coder cd, unsigned long long* __restrict__ hist_out, int n_bins,
            int n_chunks, int chunk, int copies) {
  extern __shared__ unsigned long long hists[];   // [copies][n_bins + 1]
  __shared__ int32_t queue[kFinishChunk];
  __shared__ int32_t n_queue;
  const int unit = min((int)blockIdx.x / n_chunks, g.n_units - 1);
  unsigned long long* hist = hists + (threadIdx.x & (copies - 1)) * (n_bins + 1);
  for (int q = threadIdx.x; q < copies * (n_bins + 1); q += kFinishThreads) hists[q] = 0ull;
  if (threadIdx.x == 0) n_queue = 0;
  __syncthreads();
  const int64_t* tab = g.tab + unit * g.tab_stride;
  const int64_t first = (int64_t)((int)blockIdx.x - unit * n_chunks) * chunk;   // past the end: none
  for (int q = threadIdx.x; q < chunk && first + q < g.n_tab; q += kFinishThreads)
    if (tab[first + q]) queue[atomicAdd(&n_queue, 1)] = q;
  __syncthreads();
  for (int w = threadIdx.x; w < n_queue * kParts; w += kFinishThreads) {
    const int64_t at = first + queue[w / kParts];
    const Part o = entry_part(g, at, w % kParts, tab[at]);
    add_closed<true>(hist, cd, o.A, o.B, o.C, o.x, o.y, o.z, o.t, o.n);
  }
  // the tuples outside the table
  for (int64_t s0 = (int64_t)blockIdx.x * kFinishThreads; s0 <= (int64_t)g.omask;
       s0 += (int64_t)gridDim.x * kFinishThreads) {
    __syncthreads();
    if (threadIdx.x == 0) n_queue = 0;
    __syncthreads();
    const unsigned long long k = g.okey[s0 + threadIdx.x];   // slots: a multiple of the threads
    if (k) queue[atomicAdd(&n_queue, 1)] = threadIdx.x;
    __syncthreads();
    for (int w = threadIdx.x; w < n_queue * kParts; w += kFinishThreads) {
      const int64_t s = s0 + queue[w / kParts];
      const unsigned long long e = g.okey[s] - 1;
      const int c1 = (int)(e & 127), b1 = (int)(e >> 7 & 127), a1 = (int)(e >> 14 & 127);
      const int r = (int)(e >> 21 & 63), q = (int)(e >> 27 & 63), p = (int)(e >> 33 & 63),
                t = (int)(e >> 39 & 63);
      const int x = t + p, y = t + q, z = t + r;
      const Part o = triple_part(w % kParts, a1 + x + r, b1 + x + q, c1 + y + r, x, y, z, t,
                                 (long long)g.ocnt[s]);
      if (g.n_units == 1)
        add_closed<true>(hist, cd, o.A, o.B, o.C, o.x, o.y, o.z, o.t, o.n);
      else
        add_closed<false>(hist_out + (int64_t)(e >> 45) * n_bins, cd, o.A, o.B, o.C, o.x, o.y, o.z,
                          o.t, o.n);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < n_bins; q += kFinishThreads) {
    unsigned long long v = 0ull;
    for (int c = 0; c < copies; ++c) v += hists[c * (n_bins + 1) + q];
    if (v) atomicAdd(&hist_out[(int64_t)unit * n_bins + q], v);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

// Largest theta (or kh threshold) counted by levels: the table of level 3
// must fit shared memory.
constexpr int kMaxTheta = 4;
// Nodes in this many hyperedges are hubs, whose node pairs are a matrix; the
// others' are read from their hyperedges (16: 49 ms at 60,000 hyperedges, 64:
// 3.46 ms at 10,000, against 44 and 2.84).
constexpr int kHubDeg = 32;

// table of tuples for a threshold, with the usual ranges of p, q, r
TripleTable triple_table(int theta) {
  static const int want[kTripleT] = {2, 3, 5, 3, 2};
  TripleTable tt;
  tt.total = 0;
  for (int t = 0; t < kTripleT; ++t) {
    const int n = t + theta + 2;
    tt.lo[t] = std::max(0, 2 - t);
    tt.n[t] = want[t];
    tt.off[t] = tt.total;
    tt.total += want[t] * want[t] * want[t] * n * n * n;
  }
  return tt;
}

}  // namespace

struct Levels {
  bool ready = false;
  int theta = 0;
  LevelArgs g;
  std::vector<LevelUnit> units;
  void* block[2] = {nullptr, nullptr};
  size_t bytes[2] = {0, 0};
  const int64_t* bscan = nullptr;
  const int64_t* nscan = nullptr;
  const uint32_t* cursor = nullptr;
  const uint2* adj = nullptr;
  void* zero = nullptr;       // tables cleared before each count
  size_t zero_bytes = 0;
  int64_t heavy_entries = 0;
  int grid_trip = 0, grid_many = 0;
};

void release_levels(mochy_ctx* ctx) {
  Levels* lv = ctx->levels;
  if (!lv) return;
  ctx->levels = nullptr;
  for (auto& s : ctx->side)
    if (s) cudaStreamSynchronize(s);
  cudaStreamSynchronize(ctx->stream);
  for (int i = 0; i < 2; ++i)
    if (lv->block[i]) dev_free(ctx, lv->block[i], lv->bytes[i]);
  delete lv;
}

// complete structures, in no call's use: none allocates between preparing the
// levels and launching their kernels, and release_levels waits for these
bool levels_kept(const mochy_ctx* ctx) { return ctx->levels && ctx->levels->ready; }

bool levels_cover(int theta, int64_t n_edges, int n_units) {
  // a tuple key has 19 bits left for the unit
  return theta >= 1 && theta <= kMaxTheta && n_edges > 0 && n_units < (1 << 18);
}

double levels_unit_us(double entries, double n_edges) {
  return 9.3e-5 * pow(entries * n_edges, 0.65);
}

double split_unit_us(double n_edges, double deg2, double wedges) {
  const double words = wedges * n_edges / 32.0;
  return 0.015 * n_edges + std::min(1.2e-5 * deg2, 0.24 * n_edges + 2.5e-6 * words);
}

int64_t level_entries(int max_size, int theta) {
  const int Q = theta + 3, S = std::max(max_size, 2);
  const int64_t n0 = (int64_t)Q * Q * Q;
  return 2 * n0 + 2 * (S - 1) * n0 + 2 * level2_at(S + 1, Q) + triple_table(theta).total;
}

// What prepare() takes at most for one hypergraph: heavy pairs share two nodes,
// so there are no more entries of them than sum_v C(d_v, 2) (wedges).
double levels_bytes(double n_nodes, double n_edges, double n_inc, int max_size, int theta,
                    double wedges, double node_pairs, double hubs) {
  const int Q = theta + 3, CP = Q - 1 <= 4 ? 4 : 8;
  const double heavy = std::min(wedges, n_edges * n_edges);
  const double scan = 8.0 * (3.0 * n_edges + 2.0 * n_nodes + 4.0);
  hubs = std::min(hubs, (double)kMaxHubs);
  return 2.25 * scan + (4.0 * Q + 44.0) * n_nodes + (12.0 + 4.0 * trip_classes(theta)) * n_edges +
         2.0 * n_inc + 8.0 * heavy + std::min(32.0 * heavy, 16777216.0) + 16.0 * node_pairs + n_edges * (n_edges + 8.0) / 2.0 +
         4.0 * (node_pairs + 16.0) * (8.0 + 4.0 * CP) + 4.0 * CP * hubs * hubs +
         8.0 * (double)level_entries(max_size, theta) + 65536.0;
}

static unsigned row_grid(const mochy_ctx* ctx, int64_t rows, int per_sm) {
  return (unsigned)std::max<int64_t>(
      1, std::min<int64_t>(ceil_div(rows, kRowWarps), (int64_t)ctx->num_sms * per_sm));
}

// Side streams: kernels that do not depend on each other run on them between
// fork and join (small hypergraphs leave most of the device idle in each).
static int make_sides(mochy_ctx* ctx) {
  for (auto& s : ctx->side)
    if (!s) MOCHY_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  for (auto& e : ctx->side_ev)
    if (!e) MOCHY_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  return MOCHY_OK;
}

static int fork_sides(mochy_ctx* ctx, int n) {
  MOCHY_CUDA(cudaEventRecord(ctx->side_ev[kSides], ctx->stream));
  for (int s = 0; s < n; ++s)
    MOCHY_CUDA(cudaStreamWaitEvent(ctx->side[s], ctx->side_ev[kSides], 0));
  return MOCHY_OK;
}

static int join_sides(mochy_ctx* ctx, int n) {
  for (int s = 0; s < n; ++s) {
    MOCHY_CUDA(cudaEventRecord(ctx->side_ev[s], ctx->side[s]));
    MOCHY_CUDA(cudaStreamWaitEvent(ctx->stream, ctx->side_ev[s], 0));
  }
  return MOCHY_OK;
}

static size_t triples_smem(int theta) {
  return (size_t)kTripWarps * (512 + kTripQueue * 4) +
         (size_t)trip_slots(theta) * kTripSlot * 4;
}

// Do the levels take less time than what would count instead, the split kernels
// or (kh-motifs) the scan?  Microseconds of each, from a first look at what
// they go over, fitted on random hypergraphs of 60 to 400,000 hyperedges (a
// first count, with its preparation; in ms, levels against split):
//   * split, sparse rows: a pass over the pairs of each row's neighbours.
//     250,000 hyperedges of 6 in communities of 200: 51 against 14; 400,000: 96
//     against 23.
//   * split, dense rows: a word scan a hyperwedge and 32 dense rows, where the
//     cost model of tune.cu takes them; it is only asked when the sparse pass
//     would win.  100,000 hyperedges in such communities: 13 against 51.
//   * levels, light nodes: a look-up in the overlap matrix a pair of hyperedges
//     at each light node pair, 7 ps, up to 27 where most rows are in a matrix
//     past the caches; and at light nodes around rows of many heavy pairs, 20 and
//     100 ps.  100,000 hyperedges of 10, all nodes of degree 100: 595 against
//     413 where rows share many heavy pairs, 300 against 393 where they do not.
//     This term is the least certain one (it does not know how often a look-up
//     is repeated), so a lone hypergraph keeps the levels up to 1.3 times the
//     other's time: 201,000 hyperedges of 6 in communities of 50, 187 against
//     510, would else be on the wrong side, and the 595 stay there.
//   * levels, matrix: clearing and mapping it, 0.2 us a MB.
//   * levels, tables of classes: they grow with the square of the hyperedge
//     size, and rows fill few of their entries.  1,500 uniform hyperedges of up
//     to 60: 0.91 against 0.42; 300 Zipf ones, theta = 4: 0.68 against 0.58, and
//     below 512 the levels are taken as they are (launches are most of both).
//     In a batch a unit takes 9.3e-5 (entries x hyperedges)^0.65 against 0.015 a
//     hyperedge and 1.2e-5 a squared line degree (from 20,000 a hyperedge on,
//     where dense rows pay, that much and the words of these), us: units of 60
//     hyperedges of up to 25, 6.7 against 4.0 a unit, of 250 uniform ones 20
//     against 14, of 250 Zipf ones 19 against 30, of 2,000 Zipf ones 111 against
//     481, of 2,000 to 20,000 1,800 against 14,800.  The light nodes' share is in
//     it, unless a unit's own matrix is past the caches.
//   * the scan, thresholds to 4 (levels against scan): 250,000 hyperedges in
//     communities of 200 88 against 33, of 50 20 against 12; 6,000 uniform ones
//     of up to 60 4.0 against 1.0; 4,001 Zipf ones 1.3 against 28.
static int levels_pay(mochy_ctx* ctx, int theta, LevelsAgainst against, const Work& w,
                      int64_t entries, size_t mat_bytes, int64_t n_dense, bool* pay) {
  const double E = (double)ctx->n_edges, U = (double)ctx->n_units, deg2 = (double)w.deg2;
  const bool lone = ctx->n_units == 1;
  *pay = true;
  if (lone && ctx->n_edges < 512 && against == LevelsAgainst::kSplit) return MOCHY_OK;
  const double f = (double)n_dense / E;
  const bool far = mat_bytes / (size_t)ctx->n_units >= ((size_t)256 << 20);
  double levels = 150.0 + 0.2e-6 * (double)mat_bytes;
  if (lone || far)   // else in what a unit takes
    levels += 1e-6 * 1024.0 * ((double)w.light_pairs * (7.0 + (far ? 20.0 * f * f : 0.0)) +
                               (double)w.light_rows * (far ? 100.0 : 20.0));
  levels += lone ? 3.7e-4 * (double)entries : U * levels_unit_us((double)entries, E / U);
  if (against == LevelsAgainst::kScan) {
    *pay = levels * (theta + 3) / 4.0 <= 1.25 * (300.0 + 0.03 * E + 1e-5 * deg2);
    return MOCHY_OK;
  }
  *pay = levels <= (lone ? 1.3 * (340.0 + 0.01 * E + 5e-6 * deg2)
                         : 340.0 + U * split_unit_us(E / U, deg2 / U, (double)ctx->n_wedges / U));
  if (*pay || !lone) return MOCHY_OK;
  double sparse = 0.0, words = 0.0;
  const int rc = model_split_work(ctx, &sparse, &words);
  if (rc < 0) {
    *pay = rc == MOCHY_E_UNSUPPORTED;   // the split kernels cannot count it
    return *pay ? MOCHY_OK : rc;
  }
  *pay = levels <= 1.3 * (340.0 + 0.01 * E + 5e-6 * sparse + 2.5e-6 * words);
  return MOCHY_OK;
}

// against: only when the levels take less time than that, else
// MOCHY_E_UNSUPPORTED
static int prepare(mochy_ctx* ctx, Levels* lv, int theta, LevelsAgainst against) {
  cudaStream_t st = ctx->stream;
  const int64_t E = ctx->n_edges, N = ctx->n_nodes, T = ctx->n_inc;
  if (!ctx->heavy_deg) return fail(MOCHY_E_NOMEM, "its memory holds the row order");
  MOCHY_TRY(make_sides(ctx));
  const int U = ctx->n_units, Q = theta + 3, S = std::max(ctx->max_size, 2);
  LevelArgs& g = lv->g;
  memset(&g, 0, sizeof(g));
  lv->theta = theta;
  g.n_edges = E;
  g.n_nodes = N;
  g.eoff = ctx->eoff;
  g.enode = ctx->enode;
  g.esize = ctx->esize;
  g.voff = ctx->voff;
  g.vedge = ctx->vedge;
  g.noff = ctx->noff;
  g.nadj = ctx->nadj;
  g.theta = theta;
  g.Q = Q;
  g.S = S;
  g.n_units = U;
  g.nseg = ctx->d_nseg;
  g.eseg = ctx->d_nseg ? ctx->d_nseg + U + 1 : nullptr;
  g.CP = Q - 1 <= 4 ? 4 : 8;
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  // 1. sizes: heavy degrees, dense rows, node pairs, hubs and node-graph
  // bounds, one scan over all five
  const int64_t o_d = E, o_p = 2 * E, o_b = 3 * E, o_n = 3 * E + N, n_seg = 3 * E + 2 * N;
  const size_t b_scan = al((size_t)(n_seg + 1) * 8), b_ncls = al((size_t)N * Q * 4),
               b_hplus = al((size_t)E * 4), b_ehub = al((size_t)T * 2),
               b_unit = al((size_t)U * sizeof(LevelUnit)),
               b_tot = al((size_t)(3 + 2 * (U + 1) + 4) * 8);
  lv->bytes[0] = b_scan + b_ncls + 2 * b_hplus + b_ehub + b_unit + b_tot;
  if (!room_for(ctx, lv->bytes[0] + scratch_growth(ctx, 0, (size_t)(n_seg + 1) * 8 + sizeof(Work))))
    return fail(MOCHY_E_NOMEM, "level structures past the reserved memory");
  MOCHY_TRY(dev_alloc(ctx, &lv->block[0], lv->bytes[0]));
  char* c = (char*)lv->block[0];
  auto carve = [&](size_t b) { char* r = c; c += b; return r; };
  int64_t* scan = (int64_t*)carve(b_scan);
  uint32_t* ncls = (uint32_t*)carve(b_ncls);
  int32_t* hplus = (int32_t*)carve(b_hplus);
  uint16_t* ehub = (uint16_t*)carve(b_ehub);
  LevelUnit* d_unit = (LevelUnit*)carve(b_unit);
  int64_t* d_tot = (int64_t*)carve(b_tot);
  int32_t* many = (int32_t*)carve(b_hplus);
  void* t;
  MOCHY_TRY(scratch(ctx, 0, (size_t)(n_seg + 1) * 8 + sizeof(Work), &t));
  int64_t* seg = (int64_t*)t;
  Work* d_work = (Work*)(seg + n_seg + 1);
  MOCHY_CUDA(cudaMemsetAsync(seg + n_seg, 0, 8 + sizeof(Work), st));
  k_lv_rows<<<ceil_div(E, kRowThreads), kRowThreads, 0, st>>>(
      E, ctx->noff, ctx->heavy_deg, ctx->esize, seg, seg + o_d, seg + o_p, d_work);
  MOCHY_LAUNCHED();
  k_lv_nodes<<<row_grid(ctx, N, 8), kRowThreads, 0, st>>>(g, kHubDeg, ctx->heavy_deg, ncls, seg + o_b,
                                                         seg + o_n, d_work);
  MOCHY_LAUNCHED();
  std::vector<int64_t> tot((size_t)3 + 2 * (U + 1) + 4);
  const int64_t* hub_tot = tot.data() + 3 + U + 1;   // first hub of each unit
  for (bool ranked = false;; ranked = true) {
    MOCHY_TRY(scan_exclusive_i64(ctx, seg, scan, n_seg + 1));
    if (ranked) {
      MOCHY_CUDA(cudaMemsetAsync(&d_work->light_pairs, 0, 16, st));
      k_lv_light_work<<<ceil_div(E, kRowThreads), kRowThreads, 0, st>>>(g, ctx->heavy_deg, scan + o_b,
                                                                       d_work);
      MOCHY_LAUNCHED();
    }
    k_lv_totals<<<ceil_div(U + 1, 128), 128, 0, st>>>(g, scan, o_d, o_p, o_b, o_n, n_seg, d_work, d_tot);
    MOCHY_LAUNCHED();
    MOCHY_CUDA(cudaMemcpyAsync(tot.data(), d_tot, tot.size() * 8, cudaMemcpyDeviceToHost, st));
    MOCHY_CUDA(cudaStreamSynchronize(st));
    bool crowded = false;
    for (int u = 0; u < U; ++u) crowded = crowded || hub_tot[u + 1] - hub_tot[u] > kMaxHubs;
    if (!crowded || ranked) break;
    MOCHY_TRY(scratch(ctx, 2, (size_t)N * 8, &t));
    uint32_t* key = (uint32_t*)t;
    uint32_t* val = key + N;
    k_lv_degree_keys<<<ceil_div(N, 256), 256, 0, st>>>(g, key, val);
    MOCHY_LAUNCHED();
    MOCHY_TRY(radix_sort_pairs_u32(ctx, key, val, N, 32));
    if (U > 1) {
      k_lv_unit_keys<<<ceil_div(N, 256), 256, 0, st>>>(g, val, key);
      MOCHY_LAUNCHED();
      MOCHY_TRY(radix_sort_pairs_u32(ctx, key, val, N, bits_for(U)));
    }
    k_lv_pick_hubs<<<ceil_div(N, 256), 256, 0, st>>>(g, val, kHubDeg, seg + o_b);
    MOCHY_LAUNCHED();
  }
  const int64_t H = tot[0], P = tot[1], NB = tot[2];
  // a row has at most sqrt(H) later partners (each has as many itself), whose
  // pairs then fit 32 bits
  if (H >= (int64_t)1 << 32) return fail(MOCHY_E_UNSUPPORTED, "too many heavy pairs");
  lv->heavy_entries = H;
  const int64_t d0 = H;   // the scan's second segment (dense indices) starts here
  lv->units.resize(U);
  int64_t mwords = 0, hub_pairs = 0;
  for (int u = 0; u < U; ++u) {
    LevelUnit& un = lv->units[u];
    const int64_t nd = tot[3 + u + 1] - tot[3 + u];
    un.dbase = d0 + tot[3 + u];
    un.n_dense = nd;
    un.mstride = (nd + 7) / 8;
    un.moff = mwords;
    mwords += nd * un.mstride;
    un.hbase = hub_tot[u];
    un.n_hubs = hub_tot[u + 1] - un.hbase;
    un.hmoff = hub_pairs;
    hub_pairs += un.n_hubs * un.n_hubs;
  }
  // 2. heavy rows, matrix, node pairs, tables
  g.tt = triple_table(theta);
  const int classes = trip_classes(theta);
  const int64_t n0 = (int64_t)Q * Q * Q, n1 = (S - 1) * n0, n2 = level2_at(S + 1, Q);
  g.o_star = 0;
  g.o_tri = n0;
  g.o_in1 = 2 * n0;
  g.o_out1 = g.o_in1 + n1;
  g.o_in2 = g.o_out1 + n1;
  g.o_out2 = g.o_in2 + n2;
  g.o_trip = g.o_out2 + n2;
  g.n_tab = g.o_trip + g.tt.total;
  g.tab_stride = (g.n_tab + 31) & ~(int64_t)31;
  const int64_t* tw = tot.data() + 3 + 2 * (U + 1);
  const Work w{(unsigned long long)tw[0], (unsigned long long)tw[1], (unsigned long long)tw[2],
               (unsigned long long)tw[3]};
  if (against != LevelsAgainst::kNothing) {
    bool pay;
    MOCHY_TRY(levels_pay(ctx, theta, against, w, g.n_tab, (size_t)mwords * 4, tot[3 + U], &pay));
    if (!pay) {
      ctx->levels_declined[(int)against] = theta;
      return fail(MOCHY_E_UNSUPPORTED, "the levels take more time");
    }
  }
  MOCHY_CUDA(cudaMemcpyAsync(d_unit, lv->units.data(), (size_t)U * sizeof(LevelUnit),
                             cudaMemcpyHostToDevice, st));
  uint64_t slots = 64;
  while (slots < (uint64_t)(2 * P)) slots <<= 1;
  // The hash of tuples outside the table.  A tuple that finds no slot costs 256
  // probes and some 60 global atomics, so it is sized for the distinct ones: up
  // to 0.07 a heavy entry where overlaps are 1.2 on average, 0.37 and 0.71 where
  // they are 1.4 and 3.5 (700 hyperedges of 6 to 16 of 70 nodes, theta = 4: 87 ms
  // with a quarter of a slot an entry, 7.3 with one).
  const bool wide = (double)w.overlaps > 1.3 * (double)ctx->n_wedges;
  const int64_t want = wide ? H : H / 4;
  uint64_t oslots = 1 << 12;
  while (oslots < (wide ? 1u << 20 : 1u << 18) && (int64_t)oslots < want) oslots <<= 1;
  const size_t b_hadj = al((size_t)std::max<int64_t>(H, 1) * 8),
               b_adj = al((size_t)std::max<int64_t>(NB, 1) * 8),
               b_mat = al((size_t)std::max<int64_t>(mwords, 1) * 4), b_key = al(slots * 8),
               b_cnt = al(slots * g.CP * 4), b_cur = al((size_t)(N + 1 + U * classes) * 4),
               b_list = al((size_t)E * classes * 4), b_first = al((size_t)(U * classes + 1) * 8),
               b_hubm = al((size_t)std::max<int64_t>(hub_pairs, 1) * g.CP * 4),
               b_tab = al((size_t)U * g.tab_stride * 8), b_other = al(oslots * 16);
  lv->bytes[1] = b_hadj + b_adj + b_list + b_first + b_mat + b_key + b_cnt + b_cur + b_hubm + b_tab + b_other + 256;
  if (!room_for(ctx, lv->bytes[1]))
    return fail(MOCHY_E_NOMEM, "level structures past the reserved memory");
  MOCHY_TRY(dev_alloc(ctx, &lv->block[1], lv->bytes[1]));
  c = (char*)lv->block[1];
  uint2* hadj = (uint2*)carve(b_hadj);
  uint2* adj = (uint2*)carve(b_adj);
  int32_t* tlist = (int32_t*)carve(b_list);
  int64_t* tfirst = (int64_t*)carve(b_first);
  char* z0 = c;
  g.mat = (uint32_t*)carve(b_mat);
  uint64_t* hkey = (uint64_t*)carve(b_key);
  uint32_t* hcnt = (uint32_t*)carve(b_cnt);
  uint32_t* cursor = (uint32_t*)carve(b_cur);
  uint32_t* tcount = cursor + N + 1;
  uint32_t* hubm = (uint32_t*)carve(b_hubm);
  MOCHY_CUDA(cudaMemsetAsync(z0, 0, (size_t)(c - z0), st));
  lv->zero = c;
  g.tab = (int64_t*)carve(b_tab);
  g.okey = (unsigned long long*)carve(b_other);
  g.ocnt = g.okey + oslots;
  g.omask = oslots - 1;
  g.queue = (int32_t*)carve(256);
  lv->zero_bytes = (size_t)(c - (char*)lv->zero);
  g.unit = d_unit;
  g.hoff = scan;
  g.hplus = hplus;
  g.hadj = hadj;
  g.dscan = scan + o_d;
  g.many = many;
  g.n_many = (int32_t*)cursor + N;
  g.tlist = tlist;
  g.tfirst = tfirst;
  g.ncls = ncls;
  g.ehub = ehub;
  g.hkey = hkey;
  g.hcnt = hcnt;
  g.hmask = slots - 1;
  g.hubm = hubm;
  MOCHY_TRY(fork_sides(ctx, 1));
  k_lv_fill<<<row_grid(ctx, E, 8), kRowThreads, 0, st>>>(g, hadj, hplus, many, (int32_t*)cursor + N,
                                                        tlist, tcount);
  MOCHY_LAUNCHED();
  k_lv_classes<<<1, 1024, 0, st>>>(tcount, U * classes, tfirst);
  MOCHY_LAUNCHED();
  k_lv_matrix<<<row_grid(ctx, E, 8), kRowThreads, 0, st>>>(g);
  MOCHY_LAUNCHED();
  cudaStream_t s0 = ctx->side[0];
  k_lv_pairs<<<row_grid(ctx, E, 8), kRowThreads, 0, s0>>>(g, scan + o_b, hkey, hcnt, ehub);
  MOCHY_LAUNCHED();
  const unsigned slot_grid =
      (unsigned)std::min<uint64_t>(slots / 256 + 1, (uint64_t)ctx->num_sms * 8);
  k_lv_orient<<<slot_grid, 256, 0, s0>>>(g, scan + o_n, cursor, adj);
  MOCHY_LAUNCHED();
  k_lv_hub_matrix<<<slot_grid, 256, 0, s0>>>(g, scan + o_b, hubm);
  MOCHY_LAUNCHED();
  MOCHY_TRY(join_sides(ctx, 1));
  lv->bscan = scan + o_b;
  lv->nscan = scan + o_n;
  lv->cursor = cursor;
  lv->adj = adj;
  // launch shapes
  const size_t smem = triples_smem(theta);
  if (smem + 2048 > ctx->smem_optin)
    return fail(MOCHY_E_UNSUPPORTED, "level table too large for shared memory");
  MOCHY_TRY(ensure_dynamic_smem((const void*)k_lv_triples, smem));
  MOCHY_TRY(ensure_dynamic_smem((const void*)k_lv_many, kManyBytes));
  lv->grid_trip = (int)std::max<int64_t>(1, std::min<int64_t>(kTripBlocks * ctx->num_sms, E / 16));
  lv->grid_many = 2 * ctx->num_sms;
  lv->ready = true;
  return MOCHY_OK;
}

int prepare_levels(mochy_ctx* ctx, int theta, LevelsAgainst against) {
  if (ctx->levels && ctx->levels->ready && ctx->levels->theta == theta) return MOCHY_OK;
  if (against != LevelsAgainst::kNothing &&
      ctx->levels_declined[(int)against] == theta)   // of this line graph
    return fail(MOCHY_E_UNSUPPORTED, "the levels take more time");
  release_levels(ctx);
  ctx->levels = new (std::nothrow) Levels();
  if (!ctx->levels) return fail(MOCHY_E_NOMEM, "host allocation failed");
  const int rc = prepare(ctx, ctx->levels, theta, against);
  if (rc < 0) release_levels(ctx);
  // a budget counts what is held: the preparation's scratch is not kept there
  if (ctx->budget > 0) release_scratch(ctx);
  return rc;
}

// The counting kernels (stream operations only): the motif histograms of all
// units (n_bins bins each, cleared by the caller) from the prepared levels.
int launch_levels(mochy_ctx* ctx, unsigned long long* d_hist, int n_bins, const uint16_t* lut, int k,
                  int t1, int t2, PhaseTimer* timer) {
  const Levels* lv = ctx->levels;
  const LevelArgs& g = lv->g;
  cudaStream_t st = ctx->stream;
  const int64_t E = g.n_edges, N = g.n_nodes;
  const int Q = g.Q;
  const Coder cd{lut, k, t1, t2};
  MOCHY_CUDA(cudaMemsetAsync(lv->zero, 0, lv->zero_bytes, st));
  const size_t s3 = (size_t)Q * Q * Q * 8, s1 = (size_t)std::min(kL1Rows, g.S - 1) * s3;
  auto few = Q == 4 ? k_lv_few<4> : Q == 5 ? k_lv_few<5> : Q == 6 ? k_lv_few<6> : k_lv_few<7>;
  MOCHY_TRY(ensure_dynamic_smem((const void*)few, 2 * s1));
  MOCHY_TRY(fork_sides(ctx, kSides));
  k_lv_triples<<<lv->grid_trip, kTripThreads, triples_smem(lv->theta), st>>>(g, cd, d_hist, n_bins);
  MOCHY_LAUNCHED();
  k_lv_many<<<lv->grid_many, kManyThreads, kManyBytes, ctx->side[0]>>>(g);
  MOCHY_LAUNCHED();
  few<<<row_grid(ctx, E, 8), kRowThreads, 2 * s1, ctx->side[1]>>>(g);
  MOCHY_LAUNCHED();
  k_lv_tri<<<row_grid(ctx, std::max(E, N), 8), kRowThreads, s3, ctx->side[1]>>>(g, lv->nscan,
                                                                               lv->cursor, lv->adj);
  MOCHY_LAUNCHED();
  k_lv_light<<<row_grid(ctx, E * kLightSlices, 8), kRowThreads, 0, ctx->side[2]>>>(g);
  MOCHY_LAUNCHED();
  k_lv_light_pairs<<<row_grid(ctx, (int64_t)g.hmask / 32 + 1, 8), kRowThreads, s1, ctx->side[2]>>>(
      g, lv->bscan);
  MOCHY_LAUNCHED();
  k_lv_open<<<row_grid(ctx, E, 4), kRowThreads, (size_t)n_bins * 8, ctx->side[2]>>>(g, cd, d_hist,
                                                                                   n_bins);
  MOCHY_LAUNCHED();
  k_lv_star<<<(unsigned)std::min<int64_t>(ceil_div(N, kRowThreads), (int64_t)ctx->num_sms * 4),
              kRowThreads, s3, ctx->side[2]>>>(g);
  MOCHY_LAUNCHED();
  MOCHY_TRY(join_sides(ctx, kSides));
  if (timer) timer->mark("level 3");
  // chunks of one entry a thread while all blocks fit four waves
  int chunk = kFinishThreads, copies = kFinishCopies;
  while (chunk < kFinishChunk &&
         ceil_div(g.n_tab, chunk) * (int64_t)g.n_units > (int64_t)ctx->num_sms * 32)
    chunk *= 2;
  while (copies > 1 && (size_t)copies * (n_bins + 1) * 8 > 32 * 1024) copies /= 2;
  const int n_chunks = ceil_div(g.n_tab, chunk);
  const unsigned n_blocks =
      std::max((unsigned)n_chunks * (unsigned)g.n_units,
               (unsigned)std::min<uint64_t>((g.omask + 1) / kFinishThreads, (uint64_t)ctx->num_sms * 8));
  k_lv_finish<<<n_blocks, kFinishThreads,
                (size_t)copies * (n_bins + 1) * 8, st>>>(g, cd, d_hist, n_bins, n_chunks, chunk,
                                                         copies);
  MOCHY_LAUNCHED();
  if (timer) timer->mark("finish");
  return MOCHY_OK;
}

}  // namespace mochy

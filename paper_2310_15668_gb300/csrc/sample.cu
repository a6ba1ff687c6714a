// Sampled counting: MoCHy-A (Algorithm "sampling_ver1", hyperedge sampling)
// and MoCHy-A+ (Algorithm "sampling_ver2", hyperwedge sampling), Section 3.3.
//
// Both reduce to hyperwedge work items (e_i, e_j): A+ draws one hyperwedge
// per sample; A draws a hyperedge e_i and takes every hyperwedge (e_i, e_j)
// of it.  For a work item every e_k in N_i u N_j \ {e_i, e_j} is classified:
//   A+ : every such e_k;
//   A  : e_k outside N_i, or e_k in N_i with j < k (the rule of
//        Algorithm sampling_ver1).
// Two kernels do this.  k_sample_merge: a warp merges the sorted rows of e_i
// and e_j tile by tile (short rows, or more hyperedges than shared memory has
// codes for).  k_sample_pairs (A+) and k_sample_rows (A): a block keeps the
// overlaps of one row as 4-bit codes in shared memory and only streams the
// other; what the first is the centre of comes from a histogram of its row.
// Random draws: Philox4x32-10 (Salmon et al., SC'11) on counter
// (n_lo, n_hi, stream, 0) with key (seed_lo, seed_hi); the 64-bit output u
// selects floor(u * range / 2^64).
#include <mutex>

#include "classify.cuh"
#include "philox.cuh"

namespace mochy {

// index in [0, n) of lower_bound-style search: largest r with pre[r] <= x
__device__ __forceinline__ int64_t upper_index(const int64_t* __restrict__ pre, int64_t n,
                                               int64_t x) {
  int64_t lo = 0, hi = n;  // pre[0] <= x < pre[n]
  while (hi - lo > 1) {
    const int64_t m = (lo + hi) >> 1;
    if (pre[m] <= x) lo = m; else hi = m;
  }
  return lo;
}

namespace {

constexpr int kSampThreads = 256;
constexpr int kSampWarps = kSampThreads / 32;

struct SampleArgs {
  int64_t n_edges;
  int64_t n_wedges;
  const int64_t* eoff;
  const int32_t* enode;
  const int64_t* noff;
  const uint2* nadj;
  const int64_t* ustart;
  const int64_t* uprefix;
  const uint16_t* lut3;
  unsigned long long* hist;
  int theta;
  int method;
  uint64_t seed;
  int64_t samples;
  const int64_t* item_prefix;  // A: prefix of |N_i| over samples [samples + 1]
  const int64_t* sample_row;   // A: sampled row per sample
};

// rows drawn by MoCHy-A and their degrees
__global__ void k_draw_rows(SampleArgs g, int64_t* __restrict__ row, int64_t* __restrict__ deg) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= g.samples) return;
  const uint64_t u = philox_u64(g.seed, (uint64_t)n, 1u, 0u);
  const int64_t i = (int64_t)__umul64hi(u, (uint64_t)g.n_edges);
  row[n] = i;
  deg[n] = g.noff[i + 1] - g.noff[i];
}

// classify one candidate e_k of work item (i, j)
__device__ __forceinline__ int cand_code(int A, int B, int C, int x, int y, int z, uint32_t mij,
                                         uint32_t mik, bool closed, int64_t i, int64_t j,
                                         int64_t k, const SampleArgs& g,
                                         const int32_t* __restrict__ enode,
                                         const int64_t* __restrict__ eoff) {
  int t = 0;
  if (closed) {
    if (A <= kMaskedMax) {
      t = __popc(mij & mik);
    } else {
      t = sorted_overlap3(enode + eoff[i], A, enode + eoff[j], B, enode + eoff[k], C);
    }
  }
  return ternary_code(A, B, C, x, y, z, t, g.theta);
}

__global__ void __launch_bounds__(kSampThreads)
k_sample_merge(SampleArgs g, int64_t n_items) {
  __shared__ unsigned long long hist[432];
  __shared__ uint16_t lut[2187];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = threadIdx.x; q < 432; q += kSampThreads) hist[q] = 0ull;
  for (int q = threadIdx.x; q < 2187; q += kSampThreads) lut[q] = g.lut3[q];
  __syncthreads();
  RunCache rc;
  const int64_t nwarps = (int64_t)gridDim.x * kSampWarps;
  for (int64_t it = (int64_t)blockIdx.x * kSampWarps + warp; it < n_items; it += nwarps) {
    int64_t i, pj;
    if (g.method == MOCHY_A_PLUS) {
      const uint64_t u = philox_u64(g.seed, (uint64_t)it, 2u, 0u);
      const int64_t w = (int64_t)__umul64hi(u, (uint64_t)g.n_wedges);
      i = upper_index(g.uprefix, g.n_edges, w);
      pj = g.ustart[i] + (w - g.uprefix[i]);
    } else {
      const int64_t n = upper_index(g.item_prefix, g.samples, it);
      i = g.sample_row[n];
      pj = g.noff[i] + (it - g.item_prefix[n]);
    }
    const uint2 eij = g.nadj[pj];
    const int64_t j = ent_id(eij);
    const int A = (int)(g.eoff[i + 1] - g.eoff[i]);
    const int B = ent_size(eij);
    const int x = entry_omega(eij.y, A);
    const uint32_t mij = eij.y;
    int64_t p1 = g.noff[i], e1 = g.noff[i + 1];
    int64_t p2 = g.noff[j], e2 = g.noff[j + 1];
    const uint32_t INF = 0xffffffffu;
    while (p1 < e1 || p2 < e2) {
      const uint2 t1 = p1 + lane < e1 ? g.nadj[p1 + lane] : make_uint2(INF, 0u);
      const uint2 t2 = p2 + lane < e2 ? g.nadj[p2 + lane] : make_uint2(INF, 0u);
      const uint32_t k1 = t1.x == INF ? INF : ent_id(t1);
      const uint32_t k2 = t2.x == INF ? INF : ent_id(t2);
      const uint32_t m1 = __shfl_sync(0xffffffffu, k1, 31);
      const uint32_t m2 = __shfl_sync(0xffffffffu, k2, 31);
      const uint32_t bound = min(m1, m2);
      // search own key in the other tile (keys ascending, INF padded)
      int lo = 0;
#pragma unroll
      for (int s = 16; s; s >>= 1) {
        const uint32_t probe = __shfl_sync(0xffffffffu, k2, lo + s - 1);
        if (probe < k1) lo += s;
      }
      const uint32_t at2 = __shfl_sync(0xffffffffu, k2, lo & 31);
      const uint32_t w2 = __shfl_sync(0xffffffffu, t2.y, lo & 31);
      const bool in2 = lo < 32 && at2 == k1 && k1 != INF;
      int lo2 = 0;
#pragma unroll
      for (int s = 16; s; s >>= 1) {
        const uint32_t probe = __shfl_sync(0xffffffffu, k1, lo2 + s - 1);
        if (probe < k2) lo2 += s;
      }
      const uint32_t at1 = __shfl_sync(0xffffffffu, k1, lo2 & 31);
      const bool in1 = lo2 < 32 && at1 == k2 && k2 != INF;
      // tile 1 elements (k in N_i): closed when also in N_j, else open centre i
      if (k1 <= bound && k1 != INF && (int64_t)k1 != j) {
        const int64_t k = k1;
        const bool keep = g.method == MOCHY_A_PLUS || k > j;
        if (keep) {
          const int C = ent_size(t1);
          const int z = entry_omega(t1.y, A);
          const int y = in2 ? entry_omega(w2, B) : 0;
          rc.add(lut[cand_code(A, B, C, x, y, z, mij, t1.y, in2, i, j, k, g, g.enode, g.eoff)],
                 hist);
        }
      }
      // tile 2 elements only in N_j: open centre j
      if (k2 <= bound && k2 != INF && (int64_t)k2 != i && !in1) {
        const int C = ent_size(t2);
        const int y = entry_omega(t2.y, B);
        rc.add(lut[ternary_code(A, B, C, x, y, 0, 0, g.theta)], hist);
      }
      p1 += __popc(__ballot_sync(0xffffffffu, k1 <= bound && k1 != INF));
      p2 += __popc(__ballot_sync(0xffffffffu, k2 <= bound && k2 != INF));
    }
  }
  rc.flush(hist);
  __syncthreads();
  for (int q = threadIdx.x; q < 432; q += kSampThreads)
    if (hist[q]) atomicAdd(&g.hist[q], hist[q]);
}

// ---------------------------------------------------------------------------
// Work items of long rows.  For a hyperwedge of a staged row e_i and a streamed
// row e_j, with the staged row as codes min(omega, 14) and as a histogram of
// classes (omega_ik, min(|e_k| - omega_ik, theta + 1)),
//   * e_k in N_j \ N_i (open, centre e_j) and e_k in N_i & N_j (closed) are
//     found by streaming row e_j alone;
//   * the open instances with centre e_i are the pairs (e_j, e_k) of the
//     histogram, less one "as if open" term for every closed instance.
// A+ stages the longer of its two rows and groups the draws by it.  A, which
// takes closed instances with j < k only, streams just those entries: the
// pairs of every centre e_j come from class
// histograms of all rows, made by one pass over the line graph (k_row_classes),
// and a closed instance takes off a term for each of its three centres.
// Bound by instructions, 50 to 80 per 32 entries (100,000 Zipf hyperedges,
// 200,000 draws of A+: 13.4 ms against 59.4 for the merge, whose searches by
// shuffles go over both rows; 30,011 hyperedges, 500 samples of A: 24.3 against
// 140.7).
// ---------------------------------------------------------------------------
constexpr int kRowsThreads = 256;
constexpr int kRowsWarps = kRowsThreads / 32;
// table of candidates of one hyperwedge: omega_ik 1..3, omega_jk 1..3, t 0..3,
// min(|e_k|, 15)
constexpr int kKeys = 3 * 4 * 4 * 16;
constexpr int kRowsItems = 256;         // work items of a row taken together
constexpr int kRowsSegment = 4096;      // entries of row e_j that a warp takes at a time
constexpr int kClassKeys = 64 * 8;      // (omega_ik, s) of row e_i
constexpr int kRowsMaxTheta = 4;        // sizes of 15 and more have the same states

struct RowsArgs {
  SampleArgs g;
  int64_t n_items, chunk;
  const uint32_t* row;        // A+: staged row of the draws, grouped
  const uint32_t* draw;       //     and which draw it is (null: the draw of that place)
  const uint2* other;         //     streamed row of each draw: id and size, omega
  const uint32_t* classes;    // A: class histograms of all rows
  int n_classes;              //    [largest size][theta + 2] each
  unsigned long long* queue;
};

// A+: the rows of every draw, the longer one staged
__global__ void k_draw_wedges(SampleArgs g, const uint8_t* __restrict__ esize,
                              uint32_t* __restrict__ row, uint32_t* __restrict__ draw,
                              uint2* __restrict__ other) {
  const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= g.samples) return;
  const uint64_t u = philox_u64(g.seed, (uint64_t)n, 2u, 0u);
  const int64_t w = (int64_t)__umul64hi(u, (uint64_t)g.n_wedges);
  const int64_t i = upper_index(g.uprefix, g.n_edges, w);
  const uint2 e = g.nadj[g.ustart[i] + (w - g.uprefix[i])];
  const int64_t j = ent_id(e);
  const int A = esize[i];
  const bool swap = g.noff[j + 1] - g.noff[j] > g.noff[i + 1] - g.noff[i];
  row[n] = (uint32_t)(swap ? j : i);
  if (draw) draw[n] = (uint32_t)n;
  other[n] = make_uint2(swap ? (uint32_t)i | (uint32_t)A << kIdBits : e.x,
                        (uint32_t)entry_omega(e.y, A));
}

// Warp per row: neighbours by (omega, min(own nodes, theta + 1)).
__global__ void __launch_bounds__(kRowsThreads)
k_row_classes(SampleArgs g, int n_classes, uint32_t* __restrict__ out) {
  extern __shared__ uint32_t sh[];
  const int lane = threadIdx.x & 31;
  uint32_t* h = sh + (threadIdx.x >> 5) * n_classes;
  const int ns = g.theta + 2;
  for (int q = lane; q < n_classes; q += 32) h[q] = 0u;
  __syncwarp();
  const int64_t nw = (int64_t)gridDim.x * kRowsWarps;
  for (int64_t i = (int64_t)blockIdx.x * kRowsWarps + (threadIdx.x >> 5); i < g.n_edges; i += nw) {
    const int A = (int)(g.eoff[i + 1] - g.eoff[i]);
    const int64_t pe = g.noff[i + 1];
    uint32_t ones[4] = {0u, 0u, 0u, 0u};   // omega 1, s = 0..3
    for (int64_t p0 = g.noff[i]; p0 < pe; p0 += 128) {
      uint2 e[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int64_t p = p0 + 32 * v + lane;
        e[v] = p < pe ? g.nadj[p] : make_uint2(0u, 0u);
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int z = entry_omega(e[v].y, A), s = min(ent_size(e[v]) - z, g.theta + 1);
        if (z == 0) continue;
        if (z == 1 && s < 4) {
#pragma unroll
          for (int q = 0; q < 4; ++q) ones[q] += s == q ? 1u : 0u;
        } else {
          atomicAdd(&h[(z - 1) * ns + s], 1u);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t n = __reduce_add_sync(0xffffffffu, ones[q]);
      if (lane == 0 && q < ns) h[q] += n;
    }
    __syncwarp();
    for (int q = lane; q < n_classes; q += 32) {
      out[i * n_classes + q] = h[q];
      h[q] = 0u;
    }
    __syncwarp();
  }
}

// a candidate outside the table, z = min(omega_ik, 3): classified at once
__device__ __noinline__ void rows_other(const SampleArgs& g, unsigned long long* hist,
                                        const uint16_t* lut, const int32_t* inodes, int A,
                                        const int32_t* jnodes, int B, int x, uint32_t mji, uint2 e,
                                        int z, bool half) {
  const int C = ent_size(e), y = entry_omega(e.y, B);
  if (z == 0) {
    shared_bin_add(hist, lut[ternary_code(B, A, C, x, 0, y, 0, g.theta)], 1);
    return;
  }
  const int32_t* kn = g.enode + g.eoff[ent_id(e)];
  const int t = B <= kMaskedMax ? __popc(mji & e.y) : sorted_overlap3(inodes, A, jnodes, B, kn, C);
  if (z == 3) z = sorted_overlap(inodes, A, kn, C);
  shared_bin_add(hist, lut[ternary_code(A, B, C, x, y, z, t, g.theta)], 1);
  if (x + z <= A) shared_bin_add(hist, lut[ternary_code(A, B, C, x, 0, z, 0, g.theta)], -1);
  if (half && x + y <= B) shared_bin_add(hist, lut[ternary_code(B, A, C, x, 0, y, 0, g.theta)], -1);
  if (half && z + y <= C) shared_bin_add(hist, lut[ternary_code(C, A, B, z, 0, y, 0, g.theta)], -1);
}

// MoCHy-A: a round takes up to kRowsItems hyperwedges of the staged row, ordered
// by (omega_ij, |e_j|); a warp streams one segment of one of them at a time,
// into a table of its own that it settles when that pair changes (settling
// after every hyperwedge took twice the time of the stream).
__global__ void __launch_bounds__(kRowsThreads, 4) k_sample_rows(RowsArgs r) {
  extern __shared__ uint32_t codes[];   // four bits per hyperedge, as in k_sample_pairs
  __shared__ unsigned long long hist[432];
  __shared__ uint16_t lut[2192];
  __shared__ uint32_t tables[kRowsWarps][kKeys];
  __shared__ uint2 waits[kRowsWarps][64];
  __shared__ int32_t cls[kClassKeys];
  __shared__ uint16_t used[kClassKeys];                       // classes that occur
  __shared__ int32_t inodes[64], jnodes_all[kRowsWarps][64];
  __shared__ uint2 s_eij[kRowsItems];                             // the round's items: e_j, omega
  __shared__ int s_first[kRowsItems + 1];                         // first segment of each
  __shared__ int64_t s_chunk, s_sample;
  __shared__ int s_next, s_used;
  constexpr int kGroups = 15 * 16;
  static_assert(kGroups <= kRowsThreads, "one group a thread");
  __shared__ int s_group[kGroups];
  __shared__ int64_t ws[34];
  const SampleArgs& g = r.g;
  uint2* wait = waits[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int theta = g.theta, smax = theta + 1;
  for (int64_t q = threadIdx.x; q < (g.n_edges + 7) / 8; q += kRowsThreads) codes[q] = 0u;
  for (int q = threadIdx.x; q < 432; q += kRowsThreads) hist[q] = 0ull;
  for (int q = threadIdx.x; q < 2187; q += kRowsThreads) lut[q] = g.lut3[q];
  for (int q = lane; q < kKeys; q += 32) tables[warp][q] = 0u;
  for (int q = threadIdx.x; q < kClassKeys; q += kRowsThreads) cls[q] = 0;
  int64_t cur = -1;      // staged row
  int A = 0;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) s_chunk = (int64_t)atomicAdd(r.queue, 1ull) * r.chunk;
    __syncthreads();
    int64_t it = s_chunk;
    const int64_t end = min(it + r.chunk, r.n_items);
    if (it >= r.n_items) break;
    if (warp == 0) {
      // the sample of the chunk's first item, 32 probes a round
      int64_t lo = 0, hi = g.samples;   // item_prefix[lo] <= it < item_prefix[hi]
      while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) / 32, q = lo + (lane + 1) * step;
        const int c = __popc(__ballot_sync(0xffffffffu, q < hi && g.item_prefix[q] <= it));
        hi = min(hi, lo + (c + 1) * step);
        lo = lo + c * step;
      }
      if (lane == 0) s_sample = lo;
    }
    while (it < end) {
      // a round: consecutive items of one row
      __syncthreads();
      int64_t sample = s_sample;
      while (g.item_prefix[sample + 1] <= it) ++sample;   // samples of empty rows
      const int64_t i = g.sample_row[sample];
      if (threadIdx.x == 0) {
        s_next = 0;
        s_used = 0;
      }
      if (i != cur) {
        if (cur >= 0) {
          for (int64_t p = g.noff[cur] + threadIdx.x; p < g.noff[cur + 1]; p += kRowsThreads)
            codes[ent_id(g.nadj[p]) >> 3] = 0u;
          if (threadIdx.x == 0) codes[cur >> 3] = 0u;
          for (int q = threadIdx.x; q < kClassKeys; q += kRowsThreads) cls[q] = 0;
        }
        cur = i;
        A = (int)(g.eoff[i + 1] - g.eoff[i]);
        __syncthreads();
        if (threadIdx.x < A) inodes[threadIdx.x] = g.enode[g.eoff[i] + threadIdx.x];
        if (threadIdx.x == 0) atomicOr(&codes[i >> 3], 15u << (4 * (i & 7)));
        uint32_t ones[4] = {0u, 0u, 0u, 0u};   // omega 1, s = 0..3
        for (int64_t p = g.noff[i] + threadIdx.x; p < g.noff[i + 1]; p += kRowsThreads) {
          const uint2 e = g.nadj[p];
          const uint32_t k = ent_id(e);
          const int z = entry_omega(e.y, A), s = min(ent_size(e) - z, smax);
          atomicOr(&codes[k >> 3], (uint32_t)min(z, 14) << (4 * (k & 7)));
          if (z == 1 && s < 4) {
#pragma unroll
            for (int v = 0; v < 4; ++v) ones[v] += s == v ? 1u : 0u;
          } else {
            atomicAdd(&cls[z * 8 + s], 1);
          }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const uint32_t n = __reduce_add_sync(0xffffffffu, ones[v]);
          if (lane == 0 && n) atomicAdd(&cls[8 + v], (int)n);
        }
      }
      for (int q = threadIdx.x; q < kGroups; q += kRowsThreads) s_group[q] = 0;
      __syncthreads();
      // the items of this row, by group, and their segments
      const int take = (int)(min(min(end, it + kRowsItems), g.item_prefix[sample + 1]) - it);
      const uint2* items = g.nadj + g.noff[i] + (it - g.item_prefix[sample]);
      auto group_of = [&](int x, int B) { return (min(x, 15) - 1) * 16 + min(B - x, theta + 4); };
      for (int q = threadIdx.x; q < take; q += kRowsThreads) {
        const uint2 e = items[q];
        atomicAdd(&s_group[group_of(entry_omega(e.y, A), ent_size(e))], 1);
      }
      __syncthreads();
      {
        int64_t total;
        const int64_t ex = block_scan_i64(threadIdx.x < kGroups ? s_group[threadIdx.x] : 0, ws, &total);
        if (threadIdx.x < kGroups) s_group[threadIdx.x] = (int)ex;
      }
      __syncthreads();
      for (int q = threadIdx.x; q < take; q += kRowsThreads) {
        uint2 e = items[q];
        e.y = (uint32_t)entry_omega(e.y, A);
        s_eij[atomicAdd(&s_group[group_of((int)e.y, ent_size(e))], 1)] = e;
      }
      __syncthreads();
      {
        constexpr int kPer = kRowsItems / kRowsThreads;   // consecutive items a thread
        int seg[kPer], sum = 0;
#pragma unroll
        for (int v = 0; v < kPer; ++v) {
          const int q = threadIdx.x * kPer + v;
          seg[v] = 0;
          if (q < take) {
            const int64_t j = ent_id(s_eij[q]);
            seg[v] = (int)((g.noff[j + 1] - g.ustart[j] + kRowsSegment - 1) / kRowsSegment);
          }
          sum += seg[v];
        }
        int64_t total;
        int at = (int)block_scan_i64(sum, ws, &total);
#pragma unroll
        for (int v = 0; v < kPer; ++v) {
          const int q = threadIdx.x * kPer + v;
          if (q < take) s_first[q] = at;
          at += seg[v];
        }
        if (threadIdx.x == 0) s_first[take] = (int)total;
      }
      __syncthreads();
      for (int q = threadIdx.x; q < kClassKeys; q += kRowsThreads)
        if (cls[q]) used[atomicAdd(&s_used, 1)] = (uint16_t)q;
      const int n_seg = s_first[take];
      uint2 mine_eij = make_uint2(0u, 0u);   // group of what the warp's table holds
      // nodes of e_j, and which of them lie in e_i (rows of e_j carry masks up to
      // 32 nodes), into slot w
      auto nodes_of = [&](int64_t j, int B, int w) {
        for (int q = lane; q < B; q += 32) jnodes_all[w][q] = g.enode[g.eoff[j] + q];
        __syncwarp();
        bool in = false;
        if (lane < B) {
          const int32_t v = jnodes_all[w][lane];
          int lo = 0, hi = A;
          while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if (inodes[m] < v) lo = m + 1; else hi = m;
          }
          in = lo < A && inodes[lo] == v;
        }
        return __ballot_sync(0xffffffffu, in);
      };
      // what a table of item eij stands for
      auto settle = [&](uint32_t* table, uint2 eij) {
        const int B = ent_size(eij), x = (int)eij.y;
        for (int q = lane; q < kKeys; q += 32) {
          const uint32_t n = table[q];
          if (!n) continue;
          table[q] = 0u;
          const int C = q & 15, t = q >> 4 & 3, y = q >> 6 & 3, z = (q >> 8) + 1;
          shared_bin_add(hist, lut[ternary_code(A, B, C, x, y, z, t, theta)], n);
          if (x + z <= A)
            shared_bin_add(hist, lut[ternary_code(A, B, C, x, 0, z, 0, theta)], -(long long)n);
          if (x + y <= B)
            shared_bin_add(hist, lut[ternary_code(B, A, C, x, 0, y, 0, theta)], -(long long)n);
          if (z + y <= C)
            shared_bin_add(hist, lut[ternary_code(C, A, B, z, 0, y, 0, theta)], -(long long)n);
        }
      };
      while (true) {
        int w = 0;
        if (lane == 0) w = atomicAdd(&s_next, 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= n_seg) break;
        int item = 0;
        for (int hi = take; hi - item > 1;) {
          const int m = (item + hi) >> 1;
          if (s_first[m] <= w) item = m; else hi = m;
        }
        const uint2 eij = s_eij[item];
        const int64_t j = ent_id(eij);
        // sizes past x + theta + 4 leave every region of e_j at its cap
        if (mine_eij.y != eij.y || min(ent_size(mine_eij), (int)eij.y + theta + 4) !=
                                       min(ent_size(eij), (int)eij.y + theta + 4)) {
          if (mine_eij.y) settle(tables[warp], mine_eij);
          __syncwarp();
          mine_eij = eij;
        }
        const int B = ent_size(eij), x = (int)eij.y;
        const bool masked = B <= kMaskedMax;
        uint32_t* table = tables[warp];
        int32_t* jnodes = jnodes_all[warp];
        const uint32_t mji = nodes_of(j, B, warp);
        const int64_t ps = g.ustart[j] +
                           (int64_t)(w - s_first[item]) * kRowsSegment;
        const int64_t pe = min(g.noff[j + 1], ps + kRowsSegment);
        // only closed candidates k > j are in this part of the row
        uint32_t hot = 0u;   // of the warp: key (1, 1, 1, 2)
        int waiting = 0;
        auto other = [&](uint2 e) {
          const uint32_t k = ent_id(e), z = codes[k >> 3] >> (4 * (k & 7)) & 15u;
          rows_other(g, hist, lut, inodes, A, jnodes, B, x, mji, e, (int)min(z, 3u), true);
        };
        for (int64_t p0 = ps; p0 < pe; p0 += 128) {
          uint2 e[4];   // four loads in flight a lane
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int64_t p = p0 + 32 * v + lane;
            e[v] = p < pe ? g.nadj[p] : make_uint2((uint32_t)i, 0u);   // e_i: code 15
          }
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const uint32_t k = ent_id(e[v]);
            const uint32_t z = codes[k >> 3] >> (4 * (k & 7)) & 15u;
            const uint32_t y = __popc(e[v].y), t = __popc(mji & e[v].y);
            const uint32_t key = z * 256u + y * 64u + t * 16u + (uint32_t)min(ent_size(e[v]), 15);
            const bool is_hot = key == 256u + 64u + 16u + 2u && masked;
            hot += __popc(__ballot_sync(0xffffffffu, is_hot));
            const bool closed = z != 0u && z != 15u, in_table = z < 4u && y < 4u && masked;
            if (closed && in_table && !is_hot) atomicAdd(&table[key - 256u], 1u);
            // the others (about 1 %) wait until there are 32 of them
            const unsigned m = __ballot_sync(0xffffffffu, closed && !in_table);
            if (m) {
              if (closed && !in_table) wait[waiting + __popc(m & ((1u << lane) - 1u))] = e[v];
              waiting += __popc(m);
              __syncwarp();
              if (waiting >= 32) {
                waiting -= 32;
                other(wait[waiting + lane]);
                __syncwarp();
              }
            }
          }
        }
        if (lane < waiting) other(wait[lane]);
        __syncwarp();
        if (lane == 0) table[64 + 16 + 2] += hot;
        __syncwarp();
      }
      if (mine_eij.y) settle(tables[warp], mine_eij);
      __syncthreads();
      const int n_used = s_used;
      {
        // pairs of e_i with the other neighbours of e_j, as if open
        for (int w = warp; w < take; w += kRowsWarps) {
          const uint2 eij = s_eij[w];
          const int B = ent_size(eij), x = (int)eij.y;
          const uint32_t* hj = r.classes + (int64_t)ent_id(eij) * r.n_classes;
          const int mine = (x - 1) * (theta + 2) + min(A - x, smax);
          for (int q = lane; q < r.n_classes; q += 32) {
            const int n = (int)hj[q] - (q == mine ? 1 : 0);
            const int y = q / (theta + 2) + 1;
            if (n > 0 && x + y <= B)
              shared_bin_add(hist, lut[ternary_code(B, A, y + q % (theta + 2), x, 0, y, 0, theta)],
                             n);
          }
        }
      }
      if (it == g.item_prefix[sample]) {
        // all pairs of neighbours of e_i, once per sample
        for (int w = threadIdx.x; w < n_used * n_used; w += kRowsThreads) {
          const int a = w / n_used, b = w % n_used;
          if (b < a) continue;
          const long long n1 = cls[used[a]], n2 = cls[used[b]];
          const int z1 = used[a] >> 3, s1 = used[a] & 7, z2 = used[b] >> 3, s2 = used[b] & 7;
          const long long n = a == b ? n1 * (n1 - 1) / 2 : n1 * n2;
          if (n && z1 + z2 <= A)
            shared_bin_add(hist, lut[ternary_code(A, z1 + s1, z2 + s2, z1, 0, z2, 0, theta)], n);
        }
      }
      it += take;
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 432; q += kRowsThreads)
    if (hist[q]) atomicAdd(&g.hist[q], hist[q]);
}

// MoCHy-A+: the block streams one draw's row at a time, into one table.
//   codes: min(omega, 14) of the staged row, four bits a hyperedge; 15 marks e_i
//   table key: omega_ik (0: open, 1..7), omega_jk 1..3, t 0..3, min(|e_k|, 15)
// Every field is used as it is (the caps on regions come when the table is
// settled), so an entry costs about 40 instructions; the one key that most
// lanes share, closed with both overlaps 1, t = 1 and |e_k| = 2, is counted by
// ballots.  1 in 1,000 candidates lies outside the key.
constexpr int kPlusThreads = 512;
constexpr int kPlusKeys = 8 * 4 * 4 * 16;

__global__ void __launch_bounds__(kPlusThreads, 2) k_sample_pairs(RowsArgs r) {
  extern __shared__ uint32_t codes[];   // four bits per hyperedge, all zero between rows
  __shared__ unsigned long long hist[432];
  __shared__ uint16_t lut[2192];
  __shared__ uint32_t table[kPlusKeys];
  __shared__ int32_t cls[kClassKeys];
  __shared__ uint16_t used[kClassKeys];
  __shared__ int32_t inodes[64], jnodes[64];
  __shared__ int64_t s_chunk;
  __shared__ int s_used;
  const SampleArgs& g = r.g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int theta = g.theta, smax = theta + 1;
  for (int64_t q = threadIdx.x; q < (g.n_edges + 7) / 8; q += kPlusThreads) codes[q] = 0u;
  for (int q = threadIdx.x; q < 432; q += kPlusThreads) hist[q] = 0ull;
  for (int q = threadIdx.x; q < 2187; q += kPlusThreads) lut[q] = g.lut3[q];
  for (int q = threadIdx.x; q < kPlusKeys; q += kPlusThreads) table[q] = 0u;
  for (int q = threadIdx.x; q < kClassKeys; q += kPlusThreads) cls[q] = 0;
  int64_t cur = -1;      // staged row
  int A = 0;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) s_chunk = (int64_t)atomicAdd(r.queue, 1ull) * r.chunk;
    __syncthreads();
    const int64_t first = s_chunk, end = min(first + r.chunk, r.n_items);
    if (first >= r.n_items) break;
    for (int64_t it = first; it < end; ++it) {
      const int64_t i = r.row[it];
      const uint2 eij = r.other[r.draw ? r.draw[it] : it];
      const int64_t j = ent_id(eij);
      const int B = ent_size(eij), x = (int)eij.y;
      const int64_t pb = g.noff[j], pe = g.noff[j + 1];
      if (i != cur) {
        if (cur >= 0) {
          for (int64_t p = g.noff[cur] + threadIdx.x; p < g.noff[cur + 1]; p += kPlusThreads)
            codes[ent_id(g.nadj[p]) >> 3] = 0u;
          if (threadIdx.x == 0) codes[cur >> 3] = 0u;
          for (int q = threadIdx.x; q < kClassKeys; q += kPlusThreads) cls[q] = 0;
        }
        cur = i;
        A = (int)(g.eoff[i + 1] - g.eoff[i]);
        if (threadIdx.x == 0) s_used = 0;
        __syncthreads();
        if (threadIdx.x < A) inodes[threadIdx.x] = g.enode[g.eoff[i] + threadIdx.x];
        if (threadIdx.x == 0) atomicOr(&codes[i >> 3], 15u << (4 * (i & 7)));
        uint32_t ones[4] = {0u, 0u, 0u, 0u};   // omega 1, s = 0..3
        for (int64_t p0 = g.noff[i] + warp * 128; p0 < g.noff[i + 1]; p0 += 4 * kPlusThreads) {
          uint2 e[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int64_t p = p0 + 32 * v + lane;
            e[v] = p < g.noff[i + 1] ? g.nadj[p] : make_uint2(0u, 0u);
          }
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const uint32_t k = ent_id(e[v]);
            const int z = entry_omega(e[v].y, A), s = min(ent_size(e[v]) - z, smax);
            if (z == 0) continue;
            atomicOr(&codes[k >> 3], (uint32_t)min(z, 14) << (4 * (k & 7)));
            if (z == 1 && s < 4) {
#pragma unroll
              for (int q = 0; q < 4; ++q) ones[q] += s == q ? 1u : 0u;
            } else {
              atomicAdd(&cls[z * 8 + s], 1);
            }
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t n = __reduce_add_sync(0xffffffffu, ones[q]);
          if (lane == 0 && n) atomicAdd(&cls[8 + q], (int)n);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < kClassKeys; q += kPlusThreads)
          if (cls[q]) used[atomicAdd(&s_used, 1)] = (uint16_t)q;
      }
      // nodes of e_j that lie in e_i (rows of e_j carry masks up to 32 nodes)
      const bool masked = B <= kMaskedMax;
      uint32_t mji = 0u;
      {
        bool in = false;
        if (lane < B) {
          const int32_t v = g.enode[g.eoff[j] + lane];
          if (warp == 0) jnodes[lane] = v;
          int lo = 0, hi = A;
          while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if (inodes[m] < v) lo = m + 1; else hi = m;
          }
          in = lo < A && inodes[lo] == v;
        }
        mji = __ballot_sync(0xffffffffu, in);
        if (warp == 0 && lane + 32 < B) jnodes[lane + 32] = g.enode[g.eoff[j] + lane + 32];
      }
      if (!masked) __syncthreads();   // rows_other reads jnodes
      uint32_t hot = 0u;   // of the warp: key (1, 1, 1, 2)
      auto entry = [&](uint2 e, bool has) {
        const uint32_t k = ent_id(e);
        const uint32_t z = codes[k >> 3] >> (4 * (k & 7)) & 15u;
        const uint32_t y = __popc(e.y), t = __popc(mji & e.y);
        const uint32_t key = z * 256u + y * 64u + t * 16u + (uint32_t)min(ent_size(e), 15);
        const bool is_hot = has && key == 256u + 64u + 16u + 2u && masked;
        hot += __popc(__ballot_sync(0xffffffffu, is_hot));
        if (has && !is_hot) {
          if (z < 8u && y < 4u && masked) {
            atomicAdd(&table[key], 1u);
          } else if (z != 15u) {
            rows_other(g, hist, lut, inodes, A, jnodes, B, x, mji, e, z < 3u ? (int)z : 3, false);
          }
        }
      };
      // 128 consecutive entries a warp, four loads in flight a lane
      for (int64_t p0 = pb + warp * 128; p0 < pe; p0 += 4 * kPlusThreads) {
        uint2 e[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int64_t p = p0 + 32 * v + lane;
          e[v] = p < pe ? g.nadj[p] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) entry(e[v], p0 + 32 * v + lane < pe);
      }
      if (lane == 0 && hot) atomicAdd(&table[256 + 64 + 16 + 2], hot);
      __syncthreads();
      // what the table of this draw stands for, and the pairs of e_j with the
      // other neighbours of e_i, as if open
      for (int q = threadIdx.x; q < kPlusKeys; q += kPlusThreads) {
        const uint32_t n = table[q];
        if (!n) continue;
        table[q] = 0u;
        const int C = q & 15, t = q >> 4 & 3, y = q >> 6 & 3, z = q >> 8;
        shared_bin_add(hist, lut[z ? ternary_code(A, B, C, x, y, z, t, theta)
                                   : ternary_code(B, A, C, x, 0, y, 0, theta)], n);
        if (z && x + z <= A)
          shared_bin_add(hist, lut[ternary_code(A, B, C, x, 0, z, 0, theta)], -(long long)n);
      }
      for (int w = threadIdx.x; w < s_used; w += kPlusThreads) {
        const int q = used[w], z = q >> 3;
        const int n = cls[q] - (q == x * 8 + min(B - x, smax) ? 1 : 0);
        if (n > 0 && x + z <= A)
          shared_bin_add(hist, lut[ternary_code(A, B, z + (q & 7), x, 0, z, 0, theta)], n);
      }
      __syncthreads();
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 432; q += kPlusThreads)
    if (hist[q]) atomicAdd(&g.hist[q], hist[q]);
}

size_t rows_smem_bytes(int64_t n_edges) { return (size_t)((n_edges + 7) / 8) * 4; }

// Average degrees from which rows are streamed: the block's barriers per work
// item cost about as much as merging rows of a few hundred entries by a warp.
// Streamed / merged at average degree 124, 174, 246, 369, 2,507: A+ (20,000
// draws; 4,000 at the last) 0.34 / 0.14, 0.32 / 0.18, 0.32 / 0.24, 0.33 / 0.35,
// 0.24 / 0.48 ms; A (300 draws; 80) 0.24 / 0.19, 0.29 / 0.31, 0.32 / 0.53,
// 0.47 / 1.23, 2.1 / 10.4 ms.
constexpr int64_t kPlusMinDegree = 256, kRowsMinDegree = 160;

// Draws from which they are sorted by row: the small launches take about 30 us
// (1,000 and 4,000 draws: 0.165 and 0.273 ms sorted, 0.132 and 0.241 not;
// 16,000: 0.58 and 0.70).
constexpr int64_t kGroupDraws = 4096;

// work items per hyperedge from which MoCHy-A makes the class histograms
constexpr int64_t kClassesFrom = 1;

bool use_rows(const mochy_ctx* ctx, int method) {
  const int64_t degree = method == MOCHY_A_PLUS ? kPlusMinDegree : kRowsMinDegree;
  return ctx->theta <= kRowsMaxTheta && ctx->n_wedges * 2 >= degree * ctx->n_edges &&
         rows_smem_bytes(ctx->n_edges) + 50 * 1024 <= ctx->smem_optin;
}

int launch_rows(mochy_ctx* ctx, RowsArgs r, unsigned long long* queue) {
  cudaStream_t st = ctx->stream;
  r.queue = queue;
  MOCHY_CUDA(cudaMemsetAsync(queue, 0, 8, st));
  const bool plus = r.g.method == MOCHY_A_PLUS;
  const size_t smem = rows_smem_bytes(ctx->n_edges);
  auto kern = plus ? k_sample_pairs : k_sample_rows;
  const int threads = plus ? kPlusThreads : kRowsThreads;
  MOCHY_TRY(ensure_dynamic_smem((const void*)kern, smem));
  int per_sm = 0;
  MOCHY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
  const int64_t blocks = (int64_t)ctx->num_sms * std::max(per_sm, 1);
  // chunks of up to kRowsItems hyperwedges of a row (A) or a few draws (A+)
  r.chunk = std::max<int64_t>(1, std::min<int64_t>(plus ? 16 : kRowsItems,
                                                   r.n_items / (blocks * 8)));
  const int64_t chunks = (r.n_items + r.chunk - 1) / r.chunk;
  kern<<<(unsigned)std::min(blocks, chunks), threads, smem, st>>>(r);
  MOCHY_LAUNCHED();
  return MOCHY_OK;
}

}  // namespace

int count_sampled(mochy_ctx* ctx, int method, int64_t samples, uint64_t seed,
                  unsigned long long* d_hist) {
  if (!ctx->projected) return fail(MOCHY_E_NOT_PROJECTED, "call mochy_project first");
  if (method != MOCHY_A && method != MOCHY_A_PLUS) return fail(MOCHY_E_INVALID, "bad method");
  if (samples <= 0) return fail(MOCHY_E_INVALID, "samples must be positive");
  cudaStream_t st = ctx->stream;
  MOCHY_CUDA(cudaMemsetAsync(d_hist, 0, 432 * 8, st));
  SampleArgs g;
  g.n_edges = ctx->n_edges;
  g.n_wedges = ctx->n_wedges;
  g.eoff = ctx->eoff;
  g.enode = ctx->enode;
  g.noff = ctx->noff;
  g.nadj = ctx->nadj;
  g.ustart = ctx->ustart;
  g.uprefix = ctx->uprefix;
  g.lut3 = ctx->tables.lut3;
  g.hist = d_hist;
  g.theta = ctx->theta;
  g.method = method;
  g.seed = seed;
  g.samples = samples;
  g.item_prefix = nullptr;
  g.sample_row = nullptr;
  int64_t n_items = samples;
  if (method == MOCHY_A_PLUS) {
    if (ctx->n_wedges == 0) return fail(MOCHY_E_INVALID, "the hypergraph has no hyperwedge");
  } else {
    if (ctx->n_edges == 0) return fail(MOCHY_E_INVALID, "the hypergraph has no hyperedge");
    void* t;
    MOCHY_TRY(scratch(ctx, 0, (size_t)(samples + 1) * 8 * 3, &t));
    int64_t* row = (int64_t*)t;
    int64_t* deg = row + (samples + 1);
    int64_t* pre = deg + (samples + 1);
    MOCHY_CUDA(cudaMemsetAsync(deg, 0, (size_t)(samples + 1) * 8, st));
    k_draw_rows<<<ceil_div(samples, 256), 256, 0, st>>>(g, row, deg);
    MOCHY_LAUNCHED();
    MOCHY_TRY(scan_exclusive_i64(ctx, deg, pre, samples + 1));
    MOCHY_CUDA(cudaMemcpyAsync(&n_items, pre + samples, 8, cudaMemcpyDeviceToHost, st));
    MOCHY_CUDA(cudaStreamSynchronize(st));
    g.item_prefix = pre;
    g.sample_row = row;
  }
  if (n_items == 0) return MOCHY_OK;
  if (use_rows(ctx, method) && samples <= 0xffffffffll &&
      (method == MOCHY_A_PLUS || n_items >= kClassesFrom * ctx->n_edges)) {
    RowsArgs r{};
    r.g = g;
    r.n_items = n_items;
    void* t;
    int rc;
    if (method == MOCHY_A_PLUS) {
      // the draws, grouped by row when there are enough for rows to repeat
      const bool group = samples >= kGroupDraws;
      // (with the sort's scratch, 24 bytes a draw and a few KB)
      rc = room_for(ctx, scratch_growth(ctx, 0, (size_t)samples * 16 + 16) +
                             (group ? scratch_growth(ctx, 1, (size_t)samples * 24 + (1 << 16)) : 0))
               ? scratch(ctx, 0, (size_t)samples * 16 + 16, &t) : MOCHY_E_NOMEM;
      if (rc == MOCHY_OK) {
        uint2* other = (uint2*)t;
        uint32_t* row = (uint32_t*)(other + samples);
        uint32_t* draw = group ? row + samples : nullptr;
        k_draw_wedges<<<ceil_div(samples, 256), 256, 0, st>>>(g, ctx->esize, row, draw, other);
        MOCHY_LAUNCHED();
        if (group) rc = radix_sort_pairs_u32(ctx, row, draw, samples, bits_for(ctx->n_edges));
        r.row = row;
        r.draw = draw;
        r.other = other;
      }
    } else {
      r.n_classes = std::max(ctx->max_size, 1) * (ctx->theta + 2);
      rc = room_for(ctx, scratch_growth(ctx, 2, (size_t)r.n_classes * ctx->n_edges * 4))
               ? scratch(ctx, 2, (size_t)r.n_classes * ctx->n_edges * 4, &t) : MOCHY_E_NOMEM;
      if (rc == MOCHY_OK) {
        k_row_classes<<<(unsigned)std::min<int64_t>(ceil_div(ctx->n_edges, kRowsWarps),
                                                    (int64_t)ctx->num_sms * 8),
                        kRowsThreads, (size_t)r.n_classes * 4 * kRowsWarps, st>>>(
            g, r.n_classes, (uint32_t*)t);
        MOCHY_LAUNCHED();
        r.classes = (const uint32_t*)t;
      }
    }
    if (rc == MOCHY_OK) return launch_rows(ctx, r, (unsigned long long*)(ctx->counters + 4));
    if (rc != MOCHY_E_NOMEM) return rc;   // no room for these: merge
  }
  const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(n_items, kSampWarps),
                                                    (int64_t)ctx->num_sms * 8);
  k_sample_merge<<<grid, kSampThreads, 0, st>>>(g, n_items);
  MOCHY_LAUNCHED();
  return MOCHY_OK;
}

// ---------------------------------------------------------------------------
// Sampled counting without any device allocation.
//
// For callers that cannot allocate device memory while they run: a process
// whose memory is handed out by another runtime or pool, a serving loop with
// a fixed memory reservation, code that must not grow the context's footprint
// between calls.  The working memory of this path (the motif histogram, the
// drawn rows of MoCHy-A and their prefix sums) lives in one file-scope
// __device__ array of kNoAllocBytes bytes, which every GPU that loads the
// library holds until the process exits.  The first call on a device looks
// up the array's device address (cudaGetSymbolAddress, with that device
// current); that call should come before any stream capture.  All calls
// share the array: each call clears what must start at zero, and calls whose
// work overlaps on the GPU race on it.
// ---------------------------------------------------------------------------
namespace {

constexpr int64_t kNoAllocMaxSamplesA = 65536;   // MoCHy-A draws per call
constexpr size_t kNoAllocHist = 432 * 8;
constexpr size_t kNoAllocBytes = kNoAllocHist + 256 + 3 * (kNoAllocMaxSamplesA + 1) * 8;

__global__ void __launch_bounds__(1024) k_noalloc_scan(const int64_t* __restrict__ in,
                                                       int64_t* __restrict__ out, int64_t n) {
  // exclusive scan of n values by one block, tile by tile
  __shared__ int64_t ws[34];
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < n; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const int64_t v = i < n ? in[i] : 0;
    int64_t total;
    const int64_t ex = block_scan_i64(v, ws, &total);
    const int64_t c = carry;
    if (i < n) out[i] = c + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry = c + total;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(512) k_noalloc_finish(
    const unsigned long long* __restrict__ hist, const uint8_t* __restrict__ t2h,
    const uint8_t* __restrict__ hopen, int method, double numer, double samples,
    int64_t* __restrict__ raw_h, int64_t* __restrict__ raw_3h, double* __restrict__ est_h,
    double* __restrict__ est_3h) {
  __shared__ unsigned long long h[27];
  if (threadIdx.x < 27) h[threadIdx.x] = 0ull;
  __syncthreads();
  for (int t = threadIdx.x + 1; t <= MOCHY_N_3H; t += blockDim.x) {
    raw_3h[t - 1] = (int64_t)hist[t];
    const double w = method == MOCHY_A ? 3.0 : (hopen[t2h[t]] ? 2.0 : 3.0);
    est_3h[t - 1] = __ddiv_rn(__dmul_rn((double)hist[t], numer), __dmul_rn(w, samples));
    atomicAdd(&h[t2h[t]], hist[t]);
  }
  __syncthreads();
  if (threadIdx.x < MOCHY_N_H) {
    const int id = threadIdx.x + 1;
    raw_h[threadIdx.x] = (int64_t)h[id];
    const double w = method == MOCHY_A ? 3.0 : (hopen[id] ? 2.0 : 3.0);
    est_h[threadIdx.x] = __ddiv_rn(__dmul_rn((double)h[id], numer), __dmul_rn(w, samples));
  }
}

}  // namespace

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Device address of g_noalloc_scratch on the current device, looked up once
// per device and kept for the life of the process.  A device reset
// (cudaDeviceReset) or a new primary context invalidates the kept address;
// callers that reset a device must not use this entry point afterwards.
static int noalloc_scratch(int device, unsigned char** out) {
  static std::mutex mu;
  static unsigned char* addr[256] = {nullptr};
  if (device < 0 || device >= 256) return fail(MOCHY_E_INVALID, "bad device ordinal");
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[device]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress", __FILE__, __LINE__);
    addr[device] = (unsigned char*)p;
  }
  *out = addr[device];
  return MOCHY_OK;
}

}  // namespace mochy

extern "C" int mochy_count_sampled_noalloc(mochy_ctx* ctx, int method, int64_t samples,
                                           uint64_t seed, int64_t* d_raw_h, int64_t* d_raw_3h,
                                           double* d_est_h, double* d_est_3h) {
  using namespace mochy;
  if (!ctx) return fail(MOCHY_E_INVALID, "null context");
  if (!d_raw_h || !d_raw_3h || !d_est_h || !d_est_3h) return fail(MOCHY_E_INVALID, "null output");
  if (!ctx->projected) return fail(MOCHY_E_NOT_PROJECTED, "call mochy_project first");
  if (method != MOCHY_A && method != MOCHY_A_PLUS) return fail(MOCHY_E_INVALID, "bad method");
  if (samples <= 0) return fail(MOCHY_E_INVALID, "samples must be positive");
  if (method == MOCHY_A && samples > kNoAllocMaxSamplesA)
    return fail(MOCHY_E_UNSUPPORTED, "the allocation-free MoCHy-A takes at most 65536 samples "
                                     "per call (its fixed working memory)");
  if (method == MOCHY_A_PLUS && ctx->n_wedges == 0)
    return fail(MOCHY_E_INVALID, "the hypergraph has no hyperwedge");
  if (method == MOCHY_A && ctx->n_edges == 0)
    return fail(MOCHY_E_INVALID, "the hypergraph has no hyperedge");
  MOCHY_CUDA(cudaSetDevice(ctx->device));
  unsigned char* base = nullptr;
  MOCHY_TRY(noalloc_scratch(ctx->device, &base));
  cudaStream_t st = ctx->stream;
  unsigned long long* hist = (unsigned long long*)base;
  int64_t* row = (int64_t*)(base + kNoAllocHist + 256);
  int64_t* deg = row + (kNoAllocMaxSamplesA + 1);
  int64_t* pre = deg + (kNoAllocMaxSamplesA + 1);
  MOCHY_CUDA(cudaMemsetAsync(hist, 0, kNoAllocHist, st));
  SampleArgs g;
  g.n_edges = ctx->n_edges;
  g.n_wedges = ctx->n_wedges;
  g.eoff = ctx->eoff;
  g.enode = ctx->enode;
  g.noff = ctx->noff;
  g.nadj = ctx->nadj;
  g.ustart = ctx->ustart;
  g.uprefix = ctx->uprefix;
  g.lut3 = ctx->tables.lut3;
  g.hist = hist;
  g.theta = ctx->theta;
  g.method = method;
  g.seed = seed;
  g.samples = samples;
  g.item_prefix = nullptr;
  g.sample_row = nullptr;
  int64_t n_items = samples;
  if (method == MOCHY_A) {
    MOCHY_CUDA(cudaMemsetAsync(deg, 0, (size_t)(samples + 1) * 8, st));
    k_draw_rows<<<ceil_div(samples, 256), 256, 0, st>>>(g, row, deg);
    MOCHY_LAUNCHED();
    k_noalloc_scan<<<1, 1024, 0, st>>>(deg, pre, samples + 1);
    MOCHY_LAUNCHED();
    MOCHY_CUDA(cudaMemcpyAsync(&n_items, pre + samples, 8, cudaMemcpyDeviceToHost, st));
    MOCHY_CUDA(cudaStreamSynchronize(st));
    g.item_prefix = pre;
    g.sample_row = row;
  }
  if (n_items > 0) {
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(n_items, kSampWarps),
                                                      (int64_t)ctx->num_sms * 8);
    k_sample_merge<<<grid, kSampThreads, 0, st>>>(g, n_items);
    MOCHY_LAUNCHED();
  }
  const double numer = method == MOCHY_A ? (double)ctx->n_edges : (double)ctx->n_wedges;
  k_noalloc_finish<<<1, 512, 0, st>>>(hist, ctx->tables.t2h, ctx->tables.hopen, method, numer,
                                      (double)samples, d_raw_h, d_raw_3h, d_est_h, d_est_3h);
  MOCHY_LAUNCHED();
  return MOCHY_OK;
}

// MoCHy-A+ without the line graph (Section 3.4 "Motif Counting without Line
// Graphs"; Appendix "Details of On-the-Fly MoCHy", Algorithms "alg_memdeg"
// and "alg_memdeg_adv").
//
// The paper memoizes whole neighbourhoods N_e in a hash map within a budget.
// Here no neighbourhood is ever materialized: a neighbourhood is the union
// of the incidence lists E_v of a hyperedge's nodes, and the hyperedge-id
// space is scanned 32 words per warp step (32 x 32 ids), with
//   * a membership bitmap over hyperedge ids for each popular node (the
//     memoized part: built once, as many as the budget allows, most popular
//     first), and
//   * the sorted incidence lists E_v of the other nodes, merged into the
//     scan chunk by chunk.
// Three uses of the scan:
//   1. the number of neighbours after each hyperedge i (the ascending (i, j)
//      order of hyperwedges that MoCHy-A+ draws from);
//   2. the draw: hyperwedge n is index floor(u |wedges| / 2^64) of that
//      order, as for the projected MoCHy-A+, so e_j is the o-th neighbour of
//      e_i after i, found by popcounts along the scan;
//   3. classification: for every e_k in N_i u N_j \ {e_i, e_j}, the counts
//      xa = |e_k & (e_i \ e_j)|, xb = |e_k & (e_j \ e_i)|, xt = |e_k & e_i &
//      e_j| are bit-sliced (3 bits and an overflow flag) from the bitmaps and
//      lists of the nodes of each part; omega_ik = xa + xt, omega_jk = xb +
//      xt and the triple intersection xt give the seven regions (Lemma
//      "motif:time").  For theta = 1 the four commonest (xa, xb, xt) are
//      popcounted per size class; other candidates are grouped per warp by
//      (xa, xb, xt, effective size) in a shared table and classified once
//      per group at the end of the hyperwedge, counts of 4 to 7 are
//      classified at once, and only counts of 8 or more (the slices'
//      overflow) from node lists.
// Every classified instance equals the projected MoCHy-A+'s for the same
// draws, so raw counts and estimates are the same bit for bit.
#include "classify.cuh"
#include "philox.cuh"

namespace mochy {
namespace {

constexpr int kOtfThreads = 256;
constexpr int kOtfWarps = kOtfThreads / 32;
constexpr int kOtfNodes = 128;     // nodes of e_i u e_j
constexpr int kOtfCeff = 16;
constexpr int kOtfKeys = 64 * kOtfCeff;

struct OtfArgs {
  int64_t n_edges, W;             // hyperedges; 32-bit words over hyperedge ids
  const int64_t* eoff;
  const int32_t* enode;
  const uint8_t* esize;
  const int64_t* voff;
  const int32_t* vedge;
  const int32_t* hidx;            // [N] bitmap index of a node, or -1
  const uint32_t* hbits;          // [n_bitmaps][W]
  const uint32_t* sbits;          // per word 4 words: bits 0..3 of min(|e_k|, 15)
  const int64_t* uprefix;         // [E+1] exclusive prefix of the neighbours after i
  int64_t n_wedges;
  const uint16_t* lut3;
  unsigned long long* hist;
  int theta;
  uint64_t seed;
  int64_t samples;
  int32_t* queue;
  int64_t* up;                    // degree pass: the neighbours after i
  unsigned long long* stats;      // [4] candidates, words scanned, list entries, exact
  // the draws and the bitmaps in order of size (k_otf_draw, k_otf_classify)
  int64_t first, n_draws, n_seg;  // this launch's draws, parts of a draw's scan
  int2* draws;                    // e_i, e_j of each (e_j < 0: none)
  int64_t Wp;                     // words of a bitmap in order of size
  const uint32_t* pbits;          // [n_bitmaps][Wp]
  const int32_t* cls;             // [kOtfSizes + 1] first word of each size
  const int32_t* id_of;           // [32 Wp] hyperedge at a position
};

__device__ __forceinline__ void slice_add(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& ovf,
                                          uint32_t m) {
  const uint32_t k0 = c0 & m;
  c0 ^= m;
  const uint32_t k1 = c1 & k0;
  c1 ^= k0;
  ovf |= c2 & k1;
  c2 ^= k1;
}

__device__ __forceinline__ int sval(uint32_t c0, uint32_t c1, uint32_t c2, int bit) {
  return (int)((c0 >> bit) & 1u) + 2 * (int)((c1 >> bit) & 1u) + 4 * (int)((c2 >> bit) & 1u);
}

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t* __restrict__ a, int64_t lo,
                                                   int64_t hi, int64_t x) {
  while (lo < hi) {
    const int64_t m = (lo + hi) >> 1;
    if ((int64_t)a[m] < x) lo = m + 1; else hi = m;
  }
  return lo;
}

// Per-warp state: the nodes of e_i u e_j split by part (0: e_i only, 1: e_j
// only, 2: both) into bitmap nodes and list nodes, the list cursors, and
// the table of grouped candidates.
struct OtfWarp {
  int32_t anodes[64], bnodes[64];
  int32_t hb[kOtfNodes];          // bitmap index
  int32_t hpart[kOtfNodes];
  int32_t ln[kOtfNodes];          // list node
  int32_t lpart[kOtfNodes];
  int64_t lpos[kOtfNodes], lend[kOtfNodes];
  int64_t lnext[kOtfNodes];       // id of the list's next entry (INT64_MAX when done)
  uint32_t lw[32];                // one list's entries of a chunk, as word masks
  int64_t lmin;                   // smallest next entry over the lists
  int32_t nh, nl;
  uint32_t table[kOtfKeys];
  uint32_t dirty[kOtfKeys / 32];
};

// smallest next entry over the warp's lists, into me.lmin (warp-wide)
__device__ __forceinline__ void update_lmin(OtfWarp& me) {
  const int lane = threadIdx.x & 31;
  int64_t best = INT64_MAX;
  for (int q = lane; q < me.nl; q += 32) best = min(best, me.lnext[q]);
  for (int d = 16; d; d >>= 1) best = min(best, (int64_t)__shfl_xor_sync(0xffffffffu, best, d));
  __syncwarp();
  if (lane == 0) me.lmin = best;
  __syncwarp();
}

// Sort the nodes of e (a = 0) or of e_i and e_j (a = 2) into bitmap and list
// nodes with their parts; list cursors start at the first entry >= from.
__device__ void split_nodes(const OtfArgs& g, OtfWarp& me, int A, int B, bool pair, int64_t from) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) me.nh = me.nl = 0;
  __syncwarp();
  for (int side = 0; side < (pair ? 2 : 1); ++side) {
    const int n = side == 0 ? A : B;
    const int32_t* mine = side == 0 ? me.anodes : me.bnodes;
    const int32_t* other = side == 0 ? me.bnodes : me.anodes;
    const int no = pair ? (side == 0 ? B : A) : 0;
    for (int base = 0; base < n; base += 32) {
      const int l = base + lane;
      const int32_t v = l < n ? mine[l] : -1;
      bool in_other = false;
      if (l < n) {
        int lo = 0, hi = no;
        while (lo < hi) {
          const int m = (lo + hi) >> 1;
          if (other[m] < v) lo = m + 1; else hi = m;
        }
        in_other = lo < no && other[lo] == v;
      }
      // e_j's nodes that e_i also has were taken with e_i (part 2)
      const bool take = l < n && !(side == 1 && in_other);
      const int part = side == 0 ? (in_other ? 2 : 0) : 1;
      const int h = take ? g.hidx[v] : -1;
      const bool isb = take && h >= 0, isl = take && h < 0;
      const unsigned bb = __ballot_sync(0xffffffffu, isb), bl = __ballot_sync(0xffffffffu, isl);
      const int nh0 = me.nh, nl0 = me.nl;
      __syncwarp();
      if (isb) {
        const int q = nh0 + __popc(bb & ((1u << lane) - 1u));
        me.hb[q] = h;
        me.hpart[q] = part;
      }
      if (isl) {
        const int q = nl0 + __popc(bl & ((1u << lane) - 1u));
        me.ln[q] = v;
        me.lpart[q] = part;
        const int64_t vb = g.voff[v], ve = g.voff[v + 1];
        const int64_t ps = lower_bound_i32(g.vedge, vb, ve, from);
        me.lpos[q] = ps;
        me.lend[q] = ve;
        me.lnext[q] = ps < ve ? (int64_t)g.vedge[ps] : INT64_MAX;
      }
      __syncwarp();
      if (lane == 0) {
        me.nh = nh0 + __popc(bb);
        me.nl = nl0 + __popc(bl);
      }
      __syncwarp();
    }
  }
  update_lmin(me);
}

// The bit-sliced counters of the 32 words [w0, w0 + 32) of the three parts
// (this lane's word w0 + lane): bitmap nodes OR-ed in word by word, list
// entries below hi (ids) added one by one by the lane that owns their word.
struct Slices {
  uint32_t c[3][4];   // part -> (bit 0, bit 1, bit 2, overflow)
};

__device__ __forceinline__ void gather_chunk(const OtfArgs& g, OtfWarp& me, int64_t w0,
                                             Slices& s, unsigned long long& n_entries) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int p = 0; p < 3; ++p) s.c[p][0] = s.c[p][1] = s.c[p][2] = s.c[p][3] = 0u;
  const int64_t w = w0 + lane;
  const bool inr = w < g.W;
  const int nh = me.nh, nl = me.nl;
  // bitmap nodes, eight loads in flight before their words are added
  for (int q0 = 0; q0 < nh; q0 += 8) {
    uint32_t wd[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      wd[u] = (inr && q0 + u < nh) ? __ldg(&g.hbits[(int64_t)me.hb[q0 + u] * g.W + w]) : 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int p = q0 + u < nh ? me.hpart[q0 + u] : 3;   // 3: no node (word 0)
      if (p == 0) slice_add(s.c[0][0], s.c[0][1], s.c[0][2], s.c[0][3], wd[u]);
      else if (p == 1) slice_add(s.c[1][0], s.c[1][1], s.c[1][2], s.c[1][3], wd[u]);
      else if (p == 2) slice_add(s.c[2][0], s.c[2][1], s.c[2][2], s.c[2][3], wd[u]);
    }
  }
  // list nodes: a list's entries are distinct hyperedges, so its entries in
  // this chunk are one mask per word (shared-memory OR), added once per list
  const int64_t hi = (w0 + 32) * 32;
  if (me.lmin >= hi) return;           // uniform: no list has an entry here
  for (int q = 0; q < nl; ++q) {
    if (me.lnext[q] >= hi) continue;   // uniform: nothing of this list here
    const int p = me.lpart[q];
    while (true) {
      const int64_t pos = me.lpos[q], end = me.lend[q];
      const int64_t e = pos + lane < end ? (int64_t)g.vedge[pos + lane] : INT64_MAX;
      const bool in = e < hi;
      const int nin = __popc(__ballot_sync(0xffffffffu, in));
      if (in) atomicOr(&me.lw[(e >> 5) - w0], 1u << (e & 31));
      n_entries += (unsigned long long)nin;
      const int64_t nx = __shfl_sync(0xffffffffu, e, nin & 31);
      __syncwarp();
      if (lane == 0) {
        me.lpos[q] = pos + nin;
        me.lnext[q] = nin < 32 ? nx : INT64_MAX;
      }
      __syncwarp();
      if (nin < 32) break;
      if (me.lpos[q] >= end) {
        if (lane == 0) me.lnext[q] = INT64_MAX;
        __syncwarp();
        break;
      }
    }
    const uint32_t m = me.lw[lane];
    me.lw[lane] = 0u;
    __syncwarp();
    if (p == 0) slice_add(s.c[0][0], s.c[0][1], s.c[0][2], s.c[0][3], m);
    else if (p == 1) slice_add(s.c[1][0], s.c[1][1], s.c[1][2], s.c[1][3], m);
    else slice_add(s.c[2][0], s.c[2][1], s.c[2][2], s.c[2][3], m);
  }
  update_lmin(me);
}

// first word, at or after w0, that holds an entry of a list node (for
// scans without bitmap nodes); W when none is left
__device__ __forceinline__ int64_t next_list_word(const OtfArgs& g, const OtfWarp& me) {
  return me.lmin == INT64_MAX ? g.W : min(g.W, me.lmin >> 5);
}

__device__ __forceinline__ uint32_t any_of(const Slices& s, int p) {
  return s.c[p][0] | s.c[p][1] | s.c[p][2] | s.c[p][3];
}

// Neighbours after each hyperedge: one warp per e_i; they are the hyperedges
// marked after i in the union over its nodes.
__global__ void __launch_bounds__(kOtfThreads) k_otf_degrees(OtfArgs g) {
  extern __shared__ __align__(16) unsigned char smem[];
  OtfWarp& me = ((OtfWarp*)smem)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * kOtfWarps;
  me.lw[lane] = 0u;
  __syncwarp();
  for (int64_t i = (int64_t)blockIdx.x * kOtfWarps + (threadIdx.x >> 5); i < g.n_edges;
       i += nwarps) {
    const int A = (int)(g.eoff[i + 1] - g.eoff[i]);
    if (lane < A) me.anodes[lane] = g.enode[g.eoff[i] + lane];
    if (lane + 32 < A) me.anodes[lane + 32] = g.enode[g.eoff[i] + lane + 32];
    __syncwarp();
    split_nodes(g, me, A, 0, false, 0);
    unsigned long long u = 0, ent = 0;
    const bool scan_all = me.nh > 0;
    int64_t w0 = scan_all ? 0 : next_list_word(g, me);
    while (w0 < g.W) {
      Slices s;
      gather_chunk(g, me, w0, s, ent);
      const int64_t w = w0 + lane;
      const uint32_t m = w < g.W ? any_of(s, 0) : 0u;
      if (w > (i >> 5)) u += __popc(m);
      else if (w == (i >> 5) && (i & 31) != 31) u += __popc(m & (0xffffffffu << ((i & 31) + 1)));
      w0 = scan_all ? w0 + 32 : max(w0 + 32, next_list_word(g, me));
    }
    for (int dd = 16; dd; dd >>= 1) u += __shfl_xor_sync(0xffffffffu, u, dd);
    if (lane == 0) g.up[i] = (int64_t)u;
    __syncwarp();
  }
}

// The neighbours after each hyperedge, when every node of degree `long_list`
// or more has a bitmap: one warp per hyperedge e_i.
//   * No bitmap node: nothing.  One: the entries of its list after i.  More:
//     the union of their bitmaps from i on, four words a lane at a time.
//   * The other nodes' lists from i on, an entry a lane: e_k counts at the
//     first node of e_i that it holds, in the order bitmap nodes, then list
//     nodes.
// Only words after i are read, and a list entry costs a few loads instead of
// a step of the merge in k_otf_degrees (500,000 Zipf(1.1) hyperedges: 96.2 ms
// there, 3.6 ms here).
constexpr int kAfterThreads = 256;

__global__ void __launch_bounds__(kAfterThreads) k_otf_after(OtfArgs g) {
  __shared__ int32_t s_hub[kAfterThreads / 32][64], s_list[kAfterThreads / 32][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t* hub = s_hub[warp];
  int32_t* list = s_list[warp];
  const int64_t nwarps = (int64_t)gridDim.x * (kAfterThreads / 32);
  for (int64_t i = (int64_t)blockIdx.x * (kAfterThreads / 32) + warp; i < g.n_edges; i += nwarps) {
    const int64_t eb = g.eoff[i];
    const int A = (int)(g.eoff[i + 1] - eb);
    int nh = 0, nl = 0;
    int32_t one = -1;   // the first bitmap node
    for (int q0 = 0; q0 < A; q0 += 32) {
      const int q = q0 + lane;
      const int32_t v = q < A ? g.enode[eb + q] : -1;
      const int h = q < A ? g.hidx[v] : -1;
      const unsigned bh = __ballot_sync(0xffffffffu, q < A && h >= 0);
      const unsigned bl = __ballot_sync(0xffffffffu, q < A && h < 0);
      const unsigned lt = (1u << lane) - 1u;
      if (q < A && h >= 0) hub[nh + __popc(bh & lt)] = h;
      if (q < A && h < 0) list[nl + __popc(bl & lt)] = v;
      if (one < 0 && bh) one = __shfl_sync(0xffffffffu, v, __ffs(bh) - 1);
      nh += __popc(bh);
      nl += __popc(bl);
    }
    __syncwarp();
    int64_t n = 0;   // of this lane
    if (nh == 1) {
      if (lane == 0) {
        const int64_t b = g.voff[one], e = g.voff[one + 1];
        n = e - lower_bound_i32(g.vedge, b, e, i + 1);
      }
    } else if (nh > 1) {
      const int64_t from = (i + 1) >> 5;
      int c = 0;
      for (int64_t w = (from & ~(int64_t)3) + 4 * lane; w < g.W; w += 128) {
        uint4 u = make_uint4(0u, 0u, 0u, 0u);
        for (int h = 0; h < nh; ++h) {
          const uint4 v = __ldg((const uint4*)(g.hbits + (int64_t)hub[h] * g.W + w));
          u.x |= v.x;
          u.y |= v.y;
          u.z |= v.z;
          u.w |= v.w;
        }
        if (w <= from) {   // the words before i + 1, and its bits in its own word
          const uint32_t part = 0xffffffffu << ((i + 1) & 31);
          u.x &= w < from ? 0u : part;
          u.y &= w + 1 < from ? 0u : w + 1 == from ? part : 0xffffffffu;
          u.z &= w + 2 < from ? 0u : w + 2 == from ? part : 0xffffffffu;
          u.w &= w + 3 < from ? 0u : w + 3 == from ? part : 0xffffffffu;
        }
        c += __popc(u.x) + __popc(u.y) + __popc(u.z) + __popc(u.w);
      }
      n = c;
    }
    for (int q = 0; q < nl; ++q) {
      const int32_t v = list[q];
      const int64_t e = g.voff[v + 1];
      for (int64_t p = lower_bound_i32(g.vedge, g.voff[v], e, i + 1) + lane; p < e; p += 32) {
        const int32_t k = g.vedge[p];
        bool first = true;
        for (int h = 0; h < nh && first; ++h)
          first = !(__ldg(&g.hbits[(int64_t)hub[h] * g.W + (k >> 5)]) >> (k & 31) & 1u);
        if (first && q > 0) {
          const int64_t ke = g.eoff[k + 1];
          for (int64_t s = g.eoff[k]; s < ke && first; ++s) {
            const int32_t u = g.enode[s];
            for (int r = 0; r < q; ++r)
              if (list[r] == u) first = false;
          }
        }
        n += first ? 1 : 0;
      }
    }
    for (int d = 16; d; d >>= 1) n += __shfl_xor_sync(0xffffffffu, n, d);
    if (lane == 0) g.up[i] = n;
    __syncwarp();
  }
}

__device__ __forceinline__ int64_t upper_row(const int64_t* __restrict__ pre, int64_t n,
                                             int64_t x) {
  int64_t lo = 0, hi = n;   // pre[0] <= x < pre[n]
  while (hi - lo > 1) {
    const int64_t m = (lo + hi) >> 1;
    if (pre[m] <= x) lo = m; else hi = m;
  }
  return lo;
}

// exact overlaps of e_k with e_i (z), e_j (y) and both (t)
__device__ __forceinline__ void exact_overlaps(const int32_t* a, int A, const int32_t* b, int B,
                                               const int32_t* k, int C, int& z, int& y, int& t) {
  z = y = t = 0;
  for (int q = 0; q < C; ++q) {
    const int32_t u = k[q];
    int lo = 0, hi = A;
    while (lo < hi) { const int m = (lo + hi) >> 1; if (a[m] < u) lo = m + 1; else hi = m; }
    const bool ia = lo < A && a[lo] == u;
    lo = 0; hi = B;
    while (lo < hi) { const int m = (lo + hi) >> 1; if (b[m] < u) lo = m + 1; else hi = m; }
    const bool ib = lo < B && b[lo] == u;
    z += ia; y += ib; t += ia && ib;
  }
}

// Popcounted bins for theta = 1: (xa, xb, xt, effective size).  The motif
// depends on |e_k| only through min(|e_k|, xa + xb + 2 xt + 2), so the last
// size class of each combination stands for every larger size.
__constant__ int kPopBin[13][4] = {
    {0, 0, 1, 1}, {0, 0, 1, 2}, {0, 0, 1, 3}, {0, 0, 1, 4},   // closed through e_i & e_j only
    {1, 0, 0, 1}, {1, 0, 0, 2}, {1, 0, 0, 3},                 // open, centre e_i
    {0, 1, 0, 1}, {0, 1, 0, 2}, {0, 1, 0, 3},                 // open, centre e_j
    {1, 1, 0, 2}, {1, 1, 0, 3}, {1, 1, 0, 4}};                // closed, empty triple region

// One warp per drawn hyperwedge (work queue over the samples).
// Shared: hist[432] | lut[2192] | OtfWarp[kOtfWarps]
__global__ void __launch_bounds__(kOtfThreads) k_otf_sample(OtfArgs g) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long* hist = (unsigned long long*)smem;
  uint16_t* lut = (uint16_t*)(hist + 432);
  OtfWarp& me = ((OtfWarp*)(lut + 2192))[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  for (int q = threadIdx.x; q < 432; q += kOtfThreads) hist[q] = 0ull;
  for (int q = threadIdx.x; q < 2187; q += kOtfThreads) lut[q] = g.lut3[q];
  for (int q = lane; q < kOtfKeys; q += 32) me.table[q] = 0u;
  me.dirty[lane] = 0u;
  me.lw[lane] = 0u;
  __syncthreads();
  const int theta = g.theta;
  unsigned long long st_cand = 0, st_words = 0, st_ent = 0, st_exact = 0;
  while (true) {
    int64_t n = 0;
    if (lane == 0) n = atomicAdd((unsigned long long*)g.queue, 1ull);
    n = __shfl_sync(0xffffffffu, n, 0);
    if (n >= g.samples) break;
    // the draw: hyperwedge index w of the ascending (i, j) order
    const uint64_t uu = philox_u64(g.seed, (uint64_t)n, 2u, 0u);
    const int64_t wi = (int64_t)__umul64hi(uu, (uint64_t)g.n_wedges);
    const int64_t i = upper_row(g.uprefix, g.n_edges, wi);
    int64_t o = wi - g.uprefix[i];
    const int A = (int)(g.eoff[i + 1] - g.eoff[i]);
    if (lane < A) me.anodes[lane] = g.enode[g.eoff[i] + lane];
    if (lane + 32 < A) me.anodes[lane + 32] = g.enode[g.eoff[i] + lane + 32];
    __syncwarp();
    // e_j: the o-th neighbour of e_i after i
    split_nodes(g, me, A, 0, false, i + 1);
    int64_t j = -1;
    {
      const bool scan_all = me.nh > 0;
      int64_t w0 = scan_all ? ((i + 1) >> 5) : next_list_word(g, me);
      while (w0 < g.W && j < 0) {
        Slices s;
        gather_chunk(g, me, w0, s, st_ent);
        const int64_t w = w0 + lane;
        uint32_t m = w < g.W ? any_of(s, 0) : 0u;
        if (w < ((i + 1) >> 5)) m = 0u;
        if (w == ((i + 1) >> 5)) m &= 0xffffffffu << ((i + 1) & 31);
        const int c = __popc(m);
        int incl = c;
        for (int d = 1; d < 32; d <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += t;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        if (o < tot) {
          const unsigned at = __ballot_sync(0xffffffffu, incl > o);
          const int src = __ffs(at) - 1;
          const int before = __shfl_sync(0xffffffffu, incl - c, src);
          const uint32_t ms = __shfl_sync(0xffffffffu, m, src);
          const int64_t ws = __shfl_sync(0xffffffffu, w, src);
          j = ws * 32 + (int64_t)__fns(ms, 0, (int)(o - before) + 1);
        } else {
          o -= tot;
        }
        w0 = scan_all ? w0 + 32 : max(w0 + 32, next_list_word(g, me));
      }
    }
    if (j < 0) {
      // cannot happen when the degrees are consistent: counted as an
      // instance of no motif, which the host reports as an internal error
      if (lane == 0) atomicAdd(&hist[0], 1ull);
      continue;
    }
    const int B = (int)(g.eoff[j + 1] - g.eoff[j]);
    if (lane < B) me.bnodes[lane] = g.enode[g.eoff[j] + lane];
    if (lane + 32 < B) me.bnodes[lane + 32] = g.enode[g.eoff[j] + lane + 32];
    __syncwarp();
    split_nodes(g, me, A, B, true, 0);
    // x = |e_i & e_j|
    int x = 0;
    for (int q = lane; q < A; q += 32) {
      const int32_t v = me.anodes[q];
      int lo = 0, hi = B;
      while (lo < hi) { const int m = (lo + hi) >> 1; if (me.bnodes[m] < v) lo = m + 1; else hi = m; }
      x += lo < B && me.bnodes[lo] == v;
    }
    for (int d = 16; d; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    // classification of N_i u N_j \ {i, j}
    const bool scan_all = me.nh > 0;
    // theta = 1: per-lane counts of the four commonest (xa, xb, xt) by
    // size class (see kPopBin below); the others go through the table
    uint32_t bins[13];
#pragma unroll
    for (int b = 0; b < 13; ++b) bins[b] = 0u;
    int64_t w0 = scan_all ? 0 : next_list_word(g, me);
    while (w0 < g.W) {
      Slices s;
      gather_chunk(g, me, w0, s, st_ent);
      const int64_t w = w0 + lane;
      const bool inr = w < g.W;
      uint32_t m = inr ? (any_of(s, 0) | any_of(s, 1) | any_of(s, 2)) : 0u;
      if (w == (i >> 5)) m &= ~(1u << (i & 31));
      if (w == (j >> 5)) m &= ~(1u << (j & 31));
      st_words += inr ? 1 : 0;
      st_cand += __popc(m);
      const uint4 ps = inr ? __ldg(&((const uint4*)g.sbits)[w]) : make_uint4(0u, 0u, 0u, 0u);
      const uint32_t p0 = ps.x, p1 = ps.y, p2 = ps.z, p3 = ps.w;
      const uint32_t ovf = s.c[0][3] | s.c[1][3] | s.c[2][3];
      if (theta == 1) {
        const uint32_t az = ~(s.c[0][0] | s.c[0][1] | s.c[0][2] | s.c[0][3]);
        const uint32_t a1 = s.c[0][0] & ~(s.c[0][1] | s.c[0][2] | s.c[0][3]);
        const uint32_t bz = ~(s.c[1][0] | s.c[1][1] | s.c[1][2] | s.c[1][3]);
        const uint32_t b1 = s.c[1][0] & ~(s.c[1][1] | s.c[1][2] | s.c[1][3]);
        const uint32_t tz = ~(s.c[2][0] | s.c[2][1] | s.c[2][2] | s.c[2][3]);
        const uint32_t t1 = s.c[2][0] & ~(s.c[2][1] | s.c[2][2] | s.c[2][3]);
        const uint32_t c001 = m & az & bz & t1, c100 = m & a1 & bz & tz;
        const uint32_t c010 = m & az & b1 & tz, c110 = m & a1 & b1 & tz;
        const uint32_t hi4 = p2 | p3;
        const uint32_t e1 = ~hi4 & ~p1 & p0, e2 = ~hi4 & p1 & ~p0, e3 = ~hi4 & p1 & p0;
        const uint32_t ge3 = e3 | hi4;
        bins[0] += __popc(c001 & e1);
        bins[1] += __popc(c001 & e2);
        bins[2] += __popc(c001 & e3);
        bins[3] += __popc(c001 & hi4);
        bins[4] += __popc(c100 & e1);
        bins[5] += __popc(c100 & e2);
        bins[6] += __popc(c100 & ge3);
        bins[7] += __popc(c010 & e1);
        bins[8] += __popc(c010 & e2);
        bins[9] += __popc(c010 & ge3);
        bins[10] += __popc(c110 & e2);
        bins[11] += __popc(c110 & e3);
        bins[12] += __popc(c110 & hi4);
        m &= ~(c001 | c100 | c010 | c110);
      }
      // remaining candidates, 32 at a time over the whole warp: lane l takes
      // the l-th remaining candidate of this chunk
      const int rc = __popc(m);
      int incl = rc;
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      for (int base = 0; base < total; base += 32) {
        const int item = base + lane;
        int src = 0;
#pragma unroll
        for (int stp = 16; stp; stp >>= 1) {
          const int probe = __shfl_sync(0xffffffffu, incl, src + stp - 1);
          if (probe <= item) src += stp;
        }
        src &= 31;
        const int ex = __shfl_sync(0xffffffffu, incl - rc, src);
        const uint32_t ms = __shfl_sync(0xffffffffu, m, src);
        uint32_t sc[3][4];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
          for (int b = 0; b < 4; ++b) sc[p][b] = __shfl_sync(0xffffffffu, s.c[p][b], src);
        const uint32_t so = __shfl_sync(0xffffffffu, ovf, src);
        const uint32_t q0 = __shfl_sync(0xffffffffu, p0, src), q1 = __shfl_sync(0xffffffffu, p1, src);
        const uint32_t q2 = __shfl_sync(0xffffffffu, p2, src), q3 = __shfl_sync(0xffffffffu, p3, src);
        const int64_t sw = __shfl_sync(0xffffffffu, w, src);
        const bool act = item < total;
        int key = -1;
        if (act) {
          const int bit = __fns(ms, 0, item - ex + 1);
          const int64_t k = sw * 32 + bit;
          int C = (int)((q0 >> bit) & 1u) | ((int)((q1 >> bit) & 1u) << 1) |
                  ((int)((q2 >> bit) & 1u) << 2) | ((int)((q3 >> bit) & 1u) << 3);
          if (C >= 15) C = g.esize[k];
          const int xa = sval(sc[0][0], sc[0][1], sc[0][2], bit);
          const int xb = sval(sc[1][0], sc[1][1], sc[1][2], bit);
          const int xt = sval(sc[2][0], sc[2][1], sc[2][2], bit);
          const int ce = min(C, xa + xb + 2 * xt + theta + 1);
          const bool over = (so >> bit) & 1u;   // some count is 8 or more
          if (!over && xa < 4 && xb < 4 && xt < 4 && ce <= kOtfCeff) {
            key = ((xa * 4 + xb) * 4 + xt) * kOtfCeff + ce - 1;
          } else if (!over) {
            // counts below 8 are exact: classified at once
            atomicAdd(&hist[lut[ternary_code(A, B, C, x, xb + xt, xa + xt, xt, theta)]], 1ull);
          } else {
            int z, y, t;
            exact_overlaps(me.anodes, A, me.bnodes, B, g.enode + g.eoff[k], C, z, y, t);
            atomicAdd(&hist[lut[ternary_code(A, B, C, x, y, z, t, theta)]], 1ull);
            ++st_exact;
          }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        if (key >= 0 && (peers & ((1u << lane) - 1u)) == 0) {
          atomicAdd(&me.table[key], (uint32_t)__popc(peers));
          atomicOr(&me.dirty[key >> 5], 1u << (key & 31));
        }
      }
      w0 = scan_all ? w0 + 32 : max(w0 + 32, next_list_word(g, me));
    }
    // the popcounted bins: (xa, xb, xt) and the size they stand for
    if (theta == 1) {
      uint32_t mine = 0u;
#pragma unroll
      for (int b = 0; b < 13; ++b) {
        const uint32_t v = __reduce_add_sync(0xffffffffu, bins[b]);
        if (lane == b) mine = v;
      }
      if (lane < 13 && mine) {
        const int xa = kPopBin[lane][0], xb = kPopBin[lane][1], xt = kPopBin[lane][2];
        const int ce = kPopBin[lane][3];
        atomicAdd(&hist[lut[ternary_code(A, B, ce, x, xb + xt, xa + xt, xt, 1)]],
                  (unsigned long long)mine);
      }
    }
    // the groups of this hyperwedge, classified once each
    __syncwarp();
    uint32_t dw = me.dirty[lane];
    me.dirty[lane] = 0u;
    while (dw) {
      const int q = lane * 32 + __ffs(dw) - 1;
      dw &= dw - 1;
      const uint32_t cnt = me.table[q];
      me.table[q] = 0u;
      if (!cnt) continue;
      const int ce = q % kOtfCeff + 1, combo = q / kOtfCeff;
      const int xt = combo & 3, xb = (combo >> 2) & 3, xa = combo >> 4;
      atomicAdd(&hist[lut[ternary_code(A, B, ce, x, xb + xt, xa + xt, xt, theta)]],
                (unsigned long long)cnt);
    }
    __syncwarp();
  }
  if (g.stats) {
    for (int d = 16; d; d >>= 1) {
      st_cand += __shfl_xor_sync(0xffffffffu, st_cand, d);
      st_words += __shfl_xor_sync(0xffffffffu, st_words, d);
      st_ent += __shfl_xor_sync(0xffffffffu, st_ent, d);
      st_exact += __shfl_xor_sync(0xffffffffu, st_exact, d);
    }
    if (lane == 0) {
      atomicAdd(&g.stats[0], st_cand);
      atomicAdd(&g.stats[1], st_words);
      atomicAdd(&g.stats[2], st_ent);
      atomicAdd(&g.stats[3], st_exact);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 432; q += kOtfThreads)
    if (hist[q]) atomicAdd(&g.hist[q], hist[q]);
}

// --- MoCHy-A+ when every popular node has both of its bitmaps -------------
//
// The bitmaps exist twice: over hyperedge ids (the draw's order) and over the
// hyperedges in order of size (each size from a multiple of 128 positions), so
// that a scan for the classification has one |e_k| at a time and needs no size
// planes.  k_otf_draw finds e_j; k_otf_classify scans the bitmaps of e_i u e_j
// as if the other nodes (the list nodes, a few hundred entries altogether) did
// not exist, and then, for each e_k in their lists, takes that instance back
// and adds the one with every node.  Logic and popcounts bound it (9 bitmaps
// of 62 KB a draw, all in L2).  500,000 Zipf(1.1) hyperedges, 20,000 draws:
// 32.8 ms in k_otf_sample, which groups a sixth of the candidates one by one,
// reads four size planes and merges the lists into the scan; 0.7 + 7.1 ms
// here (3.4 of it the scan's popcounts, 2 the list entries, 1 the
// combinations without a popcount).  k_otf_sample and k_otf_degrees remain
// for budgets that do not hold both bitmaps of every popular node, where a
// list may be as long as the hypergraph and an entry at a time would be the
// slow way.

constexpr int kOtfSizes = 65;      // |e_k| is 0 to 64
constexpr int kOtfPop = 19;        // combinations counted by popcounts
constexpr int kOtfDrawWords = 128; // words of a warp step: four a lane
constexpr int kOtfScanThreads = 256;
constexpr size_t kOtfDrawBytes = (size_t)256 << 10;   // at least 32,768 draws a launch
// A launch of few draws cuts each scan, so that 8 come to a resident warp (2:
// the same within 1 % at 20,000 draws).
constexpr int64_t kOtfItems = 8;
constexpr int64_t kOtfMinSteps = 4;   // steps of a part of a scan

// The draws: one warp each (grid-stride), four words a lane per step.  The
// list nodes' entries are ORed into the step's words in shared memory.
struct OtfDrawWarp {
  int32_t hub[64];
  int32_t node[64];
  int64_t pos[64], end[64], next[64];
  uint32_t lw[kOtfDrawWords];
};

__global__ void __launch_bounds__(kOtfScanThreads) k_otf_draw(OtfArgs g) {
  __shared__ __align__(16) OtfDrawWarp s_warp[kOtfScanThreads / 32];
  const int lane = threadIdx.x & 31;
  OtfDrawWarp& me = s_warp[threadIdx.x >> 5];
  const unsigned lt = (1u << lane) - 1u;
  for (int q = lane; q < kOtfDrawWords; q += 32) me.lw[q] = 0u;
  __syncwarp();
  for (int64_t n = (int64_t)blockIdx.x * (kOtfScanThreads / 32) + (threadIdx.x >> 5);
       n < g.n_draws; n += (int64_t)gridDim.x * (kOtfScanThreads / 32)) {
    const uint64_t uu = philox_u64(g.seed, (uint64_t)(g.first + n), 2u, 0u);
    const int64_t wi = (int64_t)__umul64hi(uu, (uint64_t)g.n_wedges);
    const int64_t i = upper_row(g.uprefix, g.n_edges, wi);
    int64_t o = wi - g.uprefix[i];
    const int64_t from = i + 1;
    const int A = (int)(g.eoff[i + 1] - g.eoff[i]);
    int nh = 0, nl = 0;
    for (int q0 = 0; q0 < A; q0 += 32) {
      const int q = q0 + lane;
      const int32_t v = q < A ? g.enode[g.eoff[i] + q] : -1;
      const int h = q < A ? g.hidx[v] : -1;
      const unsigned bh = __ballot_sync(0xffffffffu, q < A && h >= 0);
      const unsigned bl = __ballot_sync(0xffffffffu, q < A && h < 0);
      if (q < A && h >= 0) me.hub[nh + __popc(bh & lt)] = h;
      if (q < A && h < 0) {
        const int r = nl + __popc(bl & lt);
        const int64_t ve = g.voff[v + 1];
        const int64_t ps = lower_bound_i32(g.vedge, g.voff[v], ve, from);
        me.node[r] = v;
        me.pos[r] = ps;
        me.end[r] = ve;
        me.next[r] = ps < ve ? (int64_t)g.vedge[ps] : INT64_MAX;
      }
      nh += __popc(bh);
      nl += __popc(bl);
    }
    __syncwarp();
    auto first_entry = [&]() {
      int64_t best = INT64_MAX;
      for (int q = lane; q < nl; q += 32) best = min(best, me.next[q]);
      for (int d = 16; d; d >>= 1) best = min(best, (int64_t)__shfl_xor_sync(0xffffffffu, best, d));
      return best;
    };
    int64_t lmin = first_entry();
    int64_t j = -1;
    int64_t w0 = nh > 0 ? (from >> 5) & ~(int64_t)3 : lmin == INT64_MAX ? g.W : (lmin >> 5) & ~(int64_t)3;
    while (w0 < g.W && j < 0) {
      const int64_t w = w0 + 4 * lane;
      uint32_t u[4] = {0u, 0u, 0u, 0u};
      if (w < g.W)
        for (int h = 0; h < nh; ++h) {
          const uint4 v = __ldg((const uint4*)(g.hbits + (int64_t)me.hub[h] * g.W + w));
          u[0] |= v.x;
          u[1] |= v.y;
          u[2] |= v.z;
          u[3] |= v.w;
        }
      const int64_t hi = (w0 + kOtfDrawWords) * 32;
      if (lmin < hi) {   // uniform
        for (int q = 0; q < nl; ++q) {
          if (me.next[q] >= hi) continue;   // uniform
          int64_t p = me.pos[q];
          const int64_t end = me.end[q];
          int64_t nx;
          while (true) {
            const int64_t e = p + lane < end ? (int64_t)g.vedge[p + lane] : INT64_MAX;
            const int nin = __popc(__ballot_sync(0xffffffffu, e < hi));
            if (e < hi) atomicOr(&me.lw[(e >> 5) - w0], 1u << (e & 31));
            p += nin;
            nx = __shfl_sync(0xffffffffu, e, nin & 31);
            if (nin < 32) break;
          }
          __syncwarp();
          if (lane == 0) {
            me.pos[q] = p;
            me.next[q] = nx;
          }
        }
        __syncwarp();
        const uint4 v = *(const uint4*)&me.lw[4 * lane];
        *(uint4*)&me.lw[4 * lane] = make_uint4(0u, 0u, 0u, 0u);
        u[0] |= v.x;
        u[1] |= v.y;
        u[2] |= v.z;
        u[3] |= v.w;
        __syncwarp();
        lmin = first_entry();
      }
      int c = 0;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int64_t at = w + r;   // ids before i + 1 are not after i
        if (at < (from >> 5)) u[r] = 0u;
        if (at == (from >> 5)) u[r] &= 0xffffffffu << (from & 31);
        c += __popc(u[r]);
      }
      const int tot = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
      if (o < tot) {
        int incl = c;
        for (int d = 1; d < 32; d <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += t;
        }
        const int src = __ffs(__ballot_sync(0xffffffffu, incl > o)) - 1;
        int left = (int)o - (incl - c);   // of lane src
        int64_t found = -1;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int here = __popc(u[r]);
          if (lane == src && found < 0) {
            if (left < here) found = (w + r) * 32 + (int64_t)__fns(u[r], 0, left + 1);
            else left -= here;
          }
        }
        j = __shfl_sync(0xffffffffu, found, src);
      } else {
        o -= tot;
      }
      w0 += kOtfDrawWords;
      if (nh == 0) w0 = max(w0, lmin == INT64_MAX ? g.W : (lmin >> 5) & ~(int64_t)3);
    }
    if (lane == 0) g.draws[n] = make_int2((int)i, (int)j);
    __syncwarp();
  }
}

// Four words added to the sliced counters (c0, c1, c2, overflow): carry-save,
// 9 three-input operations instead of 24 one word after another.
__device__ __forceinline__ void slice_add4(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& ov,
                                           uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  const uint32_t s = x ^ y ^ z, k0 = (x & y) | (z & (x | y));
  const uint32_t k1 = (c0 & s) | (w & (c0 | s));
  c0 ^= s ^ w;
  const uint32_t k2 = (c1 & k0) | (k1 & (c1 | k0));
  c1 ^= k0 ^ k1;
  ov |= c2 & k2;
  c2 ^= k2;
}

// Popcounted combinations: all (xa, xb, xt) of sum 1 to 3 (97 % of the
// candidates of 500,000 Zipf(1.1) hyperedges), as indices xa + 8 xb + 64 xt.
__constant__ int kOtfPopKey[kOtfPop] = {1,  2,  3,  8,  9,   10,  16,  17,  24, 64,
                                        65, 66, 72, 73, 80, 128, 129, 136, 192};
constexpr int kOtfTab = 512;

struct OtfScanWarp {
  int32_t a[64], b[64];           // the nodes of e_i and e_j, ascending
  int8_t fa[64], fb[64];          // -1: a bitmap node, else its index among the list nodes
  int32_t hub[3][64];             // bitmaps of each part (0: e_i only, 1: e_j only, 2: both)
  int32_t list[kOtfNodes];
  __align__(16) uint32_t tab[kOtfTab];   // candidates of one size by (xa, xb, xt)
};

__device__ __forceinline__ int find_node(const int32_t* a, int n, int32_t v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (a[m] < v) lo = m + 1; else hi = m;
  }
  return lo < n && a[lo] == v ? lo : -1;
}

// One warp per draw and part of its scan (work queue).
__global__ void __launch_bounds__(kOtfScanThreads, 2) k_otf_classify(OtfArgs g) {
  __shared__ unsigned long long hist[432];
  __shared__ uint16_t lut[2192];
  __shared__ int32_t s_word[kOtfSizes + 1], s_step[kOtfSizes + 1];
  __shared__ OtfScanWarp s_warp[kOtfScanThreads / 32];
  const int lane = threadIdx.x & 31;
  OtfScanWarp& me = s_warp[threadIdx.x >> 5];
  const unsigned lt = (1u << lane) - 1u;
  const int theta = g.theta;
  // sizes of 29 + theta and more are one: with counts below 8 the motif
  // depends on |e_k| through min(|e_k|, xa + xb + 2 xt + theta + 1) only
  const int last = min(kOtfSizes - 1, 29 + theta);
  for (int q = threadIdx.x; q < 432; q += kOtfScanThreads) hist[q] = 0ull;
  for (int q = threadIdx.x; q < 2187; q += kOtfScanThreads) lut[q] = g.lut3[q];
  for (int q = lane; q < kOtfTab; q += 32) me.tab[q] = 0u;
  if (threadIdx.x == 0) {
    int steps = 0;
    for (int c = 0; c <= last; ++c) {
      s_word[c] = g.cls[c];
      s_step[c] = steps;
      const int words = g.cls[c == last ? kOtfSizes : c + 1] - g.cls[c];
      steps += (words + kOtfDrawWords - 1) / kOtfDrawWords;
    }
    s_word[last + 1] = g.cls[kOtfSizes];
    s_step[last + 1] = steps;
  }
  __syncthreads();
  const int n_steps = s_step[last + 1];
  unsigned long long st_cand = 0, st_words = 0, st_ent = 0, st_exact = 0;
  while (true) {
    int64_t item = 0;
    if (lane == 0) item = atomicAdd((unsigned long long*)g.queue, 1ull);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= g.n_draws * g.n_seg) break;
    const int64_t n = item / g.n_seg;
    const int seg = (int)(item - n * g.n_seg);
    const int2 ij = g.draws[n];
    const int64_t i = ij.x, j = ij.y;
    if (j < 0) {
      // cannot happen when the degrees are consistent: counted as an
      // instance of no motif, which the host reports as an internal error
      if (lane == 0 && seg == 0) atomicAdd(&hist[0], 1ull);
      continue;
    }
    const int64_t ib = g.eoff[i], jb = g.eoff[j];
    const int A = (int)(g.eoff[i + 1] - ib), B = (int)(g.eoff[j + 1] - jb);
    for (int q = lane; q < A; q += 32) me.a[q] = g.enode[ib + q];
    for (int q = lane; q < B; q += 32) me.b[q] = g.enode[jb + q];
    __syncwarp();
    int na = 0, nb = 0, nt = 0, nl = 0, x = 0;
    for (int q0 = 0; q0 < A; q0 += 32) {
      const int q = q0 + lane;
      const bool in = q < A;
      const int32_t v = in ? me.a[q] : -1;
      const int h = in ? g.hidx[v] : -1;
      const bool both = in && find_node(me.b, B, v) >= 0;
      const unsigned b_t = __ballot_sync(0xffffffffu, in && both && h >= 0);
      const unsigned b_a = __ballot_sync(0xffffffffu, in && !both && h >= 0);
      const unsigned b_l = __ballot_sync(0xffffffffu, in && h < 0);
      x += __popc(__ballot_sync(0xffffffffu, both));
      if (in && h >= 0) {
        if (both) me.hub[2][nt + __popc(b_t & lt)] = h;
        else me.hub[0][na + __popc(b_a & lt)] = h;
        me.fa[q] = -1;
      } else if (in) {
        const int r = nl + __popc(b_l & lt);
        me.list[r] = v;
        me.fa[q] = (int8_t)r;
      }
      nt += __popc(b_t);
      na += __popc(b_a);
      nl += __popc(b_l);
    }
    for (int q0 = 0; q0 < B; q0 += 32) {
      const int q = q0 + lane;
      const bool in = q < B;
      const int32_t v = in ? me.b[q] : -1;
      const bool own = in && find_node(me.a, A, v) < 0;   // the others came with e_i
      const int h = own ? g.hidx[v] : -1;
      const unsigned b_b = __ballot_sync(0xffffffffu, own && h >= 0);
      const unsigned b_l = __ballot_sync(0xffffffffu, own && h < 0);
      if (own && h >= 0) {
        me.hub[1][nb + __popc(b_b & lt)] = h;
        me.fb[q] = -1;
      } else if (own) {
        const int r = nl + __popc(b_l & lt);
        me.list[r] = v;
        me.fb[q] = (int8_t)r;
      }
      nb += __popc(b_b);
      nl += __popc(b_l);
    }
    __syncwarp();
    auto code = [&](int C, int y, int z, int t) {
      return (int)lut[ternary_code(A, B, C, x, y, z, t, theta)];
    };
    // the scan: steps [from, to) of all sizes
    const int from = (int)((int64_t)n_steps * seg / g.n_seg);
    const int to = na + nb + nt > 0 ? (int)((int64_t)n_steps * (seg + 1) / g.n_seg) : from;
    int c = 0;
    uint32_t bins[kOtfPop];
#pragma unroll
    for (int q = 0; q < kOtfPop; ++q) bins[q] = 0u;
    for (int step = from; step < to; ++step) {
      while (step >= s_step[c + 1]) ++c;
      const int w = s_word[c] + (step - s_step[c]) * kOtfDrawWords + 4 * lane;
      const bool in = w < s_word[c + 1];
      uint32_t cnt[3][4][4];   // part, word, slice
#pragma unroll
      for (int p = 0; p < 3; ++p) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) cnt[p][r][q] = 0u;
        const int nh = p == 0 ? na : p == 1 ? nb : nt;
        for (int h0 = 0; h0 < nh; h0 += 4) {
          uint4 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            v[q] = in && h0 + q < nh
                       ? __ldg((const uint4*)(g.pbits + (int64_t)me.hub[p][h0 + q] * g.Wp + w))
                       : make_uint4(0u, 0u, 0u, 0u);
          slice_add4(cnt[p][0][0], cnt[p][0][1], cnt[p][0][2], cnt[p][0][3], v[0].x, v[1].x,
                     v[2].x, v[3].x);
          slice_add4(cnt[p][1][0], cnt[p][1][1], cnt[p][1][2], cnt[p][1][3], v[0].y, v[1].y,
                     v[2].y, v[3].y);
          slice_add4(cnt[p][2][0], cnt[p][2][1], cnt[p][2][2], cnt[p][2][3], v[0].z, v[1].z,
                     v[2].z, v[3].z);
          slice_add4(cnt[p][3][0], cnt[p][3][1], cnt[p][3][2], cnt[p][3][3], v[0].w, v[1].w,
                     v[2].w, v[3].w);
        }
      }
      st_words += in ? 4 : 0;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        uint32_t m[3][4];   // part -> ids with 0, 1, 2, 3 of its bitmap nodes
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          const uint32_t c0 = cnt[p][r][0], c1 = cnt[p][r][1];
          const uint32_t ge4 = cnt[p][r][2] | cnt[p][r][3];
          m[p][0] = ~(c0 | c1 | ge4);
          m[p][1] = c0 & ~(c1 | ge4);
          m[p][2] = c1 & ~(c0 | ge4);
          m[p][3] = c0 & c1 & ~ge4;
        }
        uint32_t rest = m[0][0] & m[1][0] & m[2][0];
        int b = 0;
#pragma unroll
        for (int xt = 0; xt < 4; ++xt)
#pragma unroll
          for (int xb = 0; xb < 4 - xt; ++xb)
#pragma unroll
            for (int xa = 0; xa < 4 - xt - xb; ++xa) {
              if (xa + xb + xt == 0) continue;
              const uint32_t k = m[0][xa] & m[1][xb] & m[2][xt];
              bins[b++] += __popc(k);
              rest |= k;
            }
        // the others, a candidate a lane at a time (the loop is the warp's, or
        // its lanes would part for good)
        const uint32_t ov = cnt[0][r][3] | cnt[1][r][3] | cnt[2][r][3];
        rest = ~(rest | ov);
        while (__any_sync(0xffffffffu, rest != 0u)) {
          const int bit = __ffs(rest) - 1;
          if (rest) {
            const int xa = sval(cnt[0][r][0], cnt[0][r][1], cnt[0][r][2], bit);
            const int xb = sval(cnt[1][r][0], cnt[1][r][1], cnt[1][r][2], bit);
            const int xt = sval(cnt[2][r][0], cnt[2][r][1], cnt[2][r][2], bit);
            atomicAdd(&me.tab[xa + 8 * xb + 64 * xt], 1u);
          }
          rest &= rest - 1;
        }
        // a count of 8 or more: with every node at once
        if (__any_sync(0xffffffffu, ov != 0u)) {
          for (uint32_t todo = ov; todo; todo &= todo - 1) {
            const int64_t k = g.id_of[(int64_t)(w + r) * 32 + __ffs(todo) - 1];
            if (k == i || k == j) continue;
            int z, y, t;
            const int C = g.esize[k];
            exact_overlaps(me.a, A, me.b, B, g.enode + g.eoff[k], C, z, y, t);
            shared_bin_add(hist, code(C, y, z, t), 1);
            ++st_cand;
            ++st_exact;
          }
          __syncwarp();
        }
      }
      if (step + 1 == to || step + 1 == s_step[c + 1]) {   // the end of this size
        uint32_t v = 0u;
#pragma unroll
        for (int q = 0; q < kOtfPop; ++q) {
          const uint32_t sum = __reduce_add_sync(0xffffffffu, bins[q]);
          if (lane == q) v = sum;
          bins[q] = 0u;
        }
        __syncwarp();
        if (lane < kOtfPop) me.tab[kOtfPopKey[lane]] += v;
        __syncwarp();
        for (int q0 = 4 * lane; q0 < kOtfTab; q0 += 128) {
          const uint4 v4 = *(const uint4*)&me.tab[q0];
          if (!(v4.x | v4.y | v4.z | v4.w)) continue;
          *(uint4*)&me.tab[q0] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t num = u == 0 ? v4.x : u == 1 ? v4.y : u == 2 ? v4.z : v4.w;
            if (!num) continue;
            const int q = q0 + u, xa = q & 7, xb = (q >> 3) & 7, xt = q >> 6;
            shared_bin_add(hist, code(c, xb + xt, xa + xt, xt), num);
            st_cand += num;
          }
        }
        __syncwarp();
      }
    }
    // e_i and e_j were candidates of the scan
    if (seg == 0 && lane < 2) {
      const int xa = lane == 0 ? na : 0, xb = lane == 0 ? 0 : nb;
      if (xa + xb + nt > 0 && xa < 8 && xb < 8 && nt < 8) {
        shared_bin_add(hist, code(lane == 0 ? A : B, xb + nt, xa + nt, nt), -1);
        --st_cand;
      }
    }
    // list entries: each e_k at the first list node that it holds
    for (int q = 0; q < nl; ++q) {
      const int32_t v = me.list[q];
      const int64_t end = g.voff[v + 1];
      for (int64_t p = g.voff[v] + seg * 32 + lane; p < end; p += 32 * g.n_seg) {
        const int64_t k = g.vedge[p];
        ++st_ent;
        if (k == i || k == j) continue;
        const int64_t kb = g.eoff[k];
        const int C = (int)(g.eoff[k + 1] - kb);
        int y = 0, z = 0, t = 0, xa = 0, xb = 0, xt = 0, owner = kOtfNodes;
        for (int s = 0; s < C; ++s) {
          const int32_t u = g.enode[kb + s];
          const int pa = find_node(me.a, A, u), pb = find_node(me.b, B, u);
          if (pa < 0 && pb < 0) continue;
          const int f = pa >= 0 ? me.fa[pa] : me.fb[pb];
          z += pa >= 0;
          y += pb >= 0;
          t += pa >= 0 && pb >= 0;
          if (f >= 0) {
            owner = min(owner, f);
          } else if (pa >= 0 && pb >= 0) {
            ++xt;
          } else if (pa >= 0) {
            ++xa;
          } else {
            ++xb;
          }
        }
        if (owner != q || xa >= 8 || xb >= 8 || xt >= 8) continue;
        const int with = code(C, y, z, t);
        if (xa + xb + xt == 0) {
          shared_bin_add(hist, with, 1);
          ++st_cand;
        } else {
          const int without = code(C, xb + xt, xa + xt, xt);
          if (with != without) {
            shared_bin_add(hist, without, -1);
            shared_bin_add(hist, with, 1);
          }
        }
      }
    }
    __syncwarp();
  }
  if (g.stats) {
    for (int d = 16; d; d >>= 1) {
      st_cand += __shfl_xor_sync(0xffffffffu, st_cand, d);
      st_words += __shfl_xor_sync(0xffffffffu, st_words, d);
      st_ent += __shfl_xor_sync(0xffffffffu, st_ent, d);
      st_exact += __shfl_xor_sync(0xffffffffu, st_exact, d);
    }
    if (lane == 0) {
      atomicAdd(&g.stats[0], st_cand);
      atomicAdd(&g.stats[1], st_words);
      atomicAdd(&g.stats[2], st_ent);
      atomicAdd(&g.stats[3], st_exact);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 432; q += kOtfScanThreads)
    if (hist[q]) atomicAdd(&g.hist[q], hist[q]);
}

// Hyperedges of each size (the counts are cleared before): 5, 11 and 30 us for
// the three kernels that order 500,000 hyperedges by size.
__global__ void k_otf_sizes(int64_t E, const uint8_t* __restrict__ esize, int32_t* counts) {
  __shared__ int32_t s[kOtfSizes];
  if (threadIdx.x < kOtfSizes) s[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < E;
       k += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&s[esize[k]], 1);
  __syncthreads();
  if (threadIdx.x < kOtfSizes && s[threadIdx.x]) atomicAdd(&counts[threadIdx.x], s[threadIdx.x]);
}

// first word of each size, a multiple of four; counts -> next free position
__global__ void k_otf_starts(int32_t* counts, int32_t* cls) {
  if (threadIdx.x) return;
  int32_t w = 0;
  for (int c = 0; c < kOtfSizes; ++c) {
    const int32_t n = counts[c];
    cls[c] = w;
    counts[c] = w * 32;
    w += (n + 127) / 128 * 4;
  }
  cls[kOtfSizes] = w;
}

// position of each hyperedge in order of size (any order within a size)
__global__ void k_otf_positions(int64_t E, const uint8_t* __restrict__ esize, int32_t* next,
                                int32_t* __restrict__ pos_of, int32_t* __restrict__ id_of) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int c = k < E ? esize[k] : -1;
  const unsigned peers = __match_any_sync(0xffffffffu, c);
  if (c < 0) return;
  const int lead = __ffs(peers) - 1;
  int32_t at = 0;
  if (lane == lead) at = atomicAdd(&next[c], __popc(peers));
  at = __shfl_sync(peers, at, lead) + __popc(peers & ((1u << lane) - 1u));
  pos_of[k] = at;
  id_of[at] = (int32_t)k;
}

// membership bitmap of each bitmap node (its incidence list as bits); pbits
// (may be null): the same in order of size
__global__ void k_otf_bits(int64_t n_bitmaps, int64_t W, const int32_t* __restrict__ nodes_of,
                           const int64_t* __restrict__ voff, const int32_t* __restrict__ vedge,
                           uint32_t* __restrict__ bits, int64_t Wp,
                           const int32_t* __restrict__ pos_of, uint32_t* __restrict__ pbits) {
  for (int64_t h = blockIdx.x; h < n_bitmaps; h += gridDim.x) {
    const int32_t v = nodes_of[h];
    uint32_t* b = bits + h * W;
    for (int64_t q = voff[v] + threadIdx.x; q < voff[v + 1]; q += blockDim.x) {
      const int32_t e = vedge[q];
      atomicOr(&b[e >> 5], 1u << (e & 31));
      if (pbits) {
        const int32_t at = pos_of[e];
        atomicOr(&pbits[h * Wp + (at >> 5)], 1u << (at & 31));
      }
    }
  }
}

__global__ void k_otf_size_bits(int64_t E, int64_t W, const uint8_t* __restrict__ esize,
                                uint32_t* __restrict__ sbits) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= E) return;
  const int c = min((int)esize[k], 15);
  for (int b = 0; b < 4; ++b)
    if (c & (1 << b)) atomicOr(&sbits[4 * (k >> 5) + b], 1u << (k & 31));
}

}  // namespace

size_t otf_smem_bytes() { return 432 * 8 + 2192 * 2 + sizeof(OtfWarp) * kOtfWarps; }

void release_onthefly(mochy_ctx* ctx) {
  if (ctx->otf_block) {
    cudaStreamSynchronize(ctx->stream);
    dev_free(ctx, ctx->otf_block, ctx->otf_bytes);
  }
  ctx->otf_block = nullptr;
  ctx->otf_bytes = 0;
  ctx->otf_ready = false;
  ctx->otf_hidx = nullptr;
  ctx->otf_hbits = nullptr;
  ctx->otf_sbits = nullptr;
  ctx->otf_uprefix = nullptr;
  ctx->otf_by_size = false;
  ctx->otf_pbits = nullptr;
  ctx->otf_id_of = ctx->otf_cls = nullptr;
  ctx->otf_draws = nullptr;
  ctx->otf_pwords = ctx->otf_max_draws = 0;
  ctx->otf_wedges = ctx->otf_bitmaps = ctx->otf_words = 0;
}

// Bitmaps, size planes, degrees and the prefix of the neighbours after each
// hyperedge.  budget: bytes for bitmaps (<= 0: the library's choice).
int prepare_onthefly(mochy_ctx* ctx, int64_t budget) {
  if (ctx->otf_ready) return MOCHY_OK;
  cudaStream_t st = ctx->stream;
  const int64_t E = ctx->n_edges, N = ctx->n_nodes;
  // words of a bitmap, a multiple of four: its rows start on 16 bytes
  const int64_t W = (std::max<int64_t>((E + 31) / 32, 1) + 3) & ~(int64_t)3;
  // bitmap nodes: degree >= W / 32 (a bitmap costs about what a list of
  // that length costs to merge), most popular first, within the budget
  std::vector<int64_t> voff((size_t)N + 1);
  MOCHY_CUDA(cudaMemcpyAsync(voff.data(), ctx->voff, voff.size() * 8, cudaMemcpyDeviceToHost, st));
  MOCHY_CUDA(cudaStreamSynchronize(st));
  const int64_t thr = std::max<int64_t>(W / 32, 16);
  std::vector<std::pair<int64_t, int32_t>> pop;
  for (int64_t v = 0; v < N; ++v)
    if (voff[v + 1] - voff[v] >= thr) pop.push_back({-(voff[v + 1] - voff[v]), (int32_t)v});
  std::sort(pop.begin(), pop.end());
  const int64_t cap_bytes =
      budget > 0 ? budget : (ctx->budget > 0 ? ctx->budget / 4 : ((int64_t)4 << 30));
  int64_t max_bitmaps = std::min<int64_t>((int64_t)pop.size(), cap_bytes / (W * 4));
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  // bitmaps in order of size as well when all of both fit the budget; each of
  // the 64 sizes begins on four words
  const int64_t Wp = W + 4 * kOtfSizes;
  bool by_size = max_bitmaps == (int64_t)pop.size() &&
                 (int64_t)pop.size() * (W + Wp) * 4 <= cap_bytes;
  const size_t b_hidx = al((size_t)std::max<int64_t>(N, 1) * 4);
  const size_t b_sbits = al((size_t)4 * W * 4);
  const size_t b_pre = al((size_t)(E + 1) * 8);
  const size_t b_pos = al((size_t)std::max<int64_t>(E, 1) * 4), b_id = al((size_t)Wp * 32 * 4);
  size_t b_nodes, b_one, b_bits, b_order, b_up, bytes;
  void* p = nullptr;
  // What makes the call faster takes only the memory that there is: without
  // room for both sets of bitmaps one is left out, then the least popular
  // nodes' bitmaps.
  while (true) {
    b_nodes = al((size_t)std::max<int64_t>(max_bitmaps, 1) * 4);
    b_one = al((size_t)std::max<int64_t>(max_bitmaps, 1) * W * 4);
    b_bits = by_size ? b_one + al((size_t)std::max<int64_t>(max_bitmaps, 1) * Wp * 4) : b_one;
    // by size: the positions (both ways) and the sizes' first words; the draws
    // of a launch take the place of the neighbours after each hyperedge once
    // these are summed (E + 1 entries: the scan reads them all)
    b_order = by_size ? b_pos + b_id + al((2 * kOtfSizes + 1) * 4) : 0;
    b_up = al((size_t)(E + 1) * 8);
    if (by_size) b_up = std::max(b_up, kOtfDrawBytes);
    bytes = b_hidx + b_nodes + b_bits + b_sbits + b_pre + b_order + b_up;
    const int rc = dev_alloc(ctx, &p, bytes);
    if (rc == MOCHY_OK) break;
    if (rc != MOCHY_E_NOMEM || (!by_size && max_bitmaps == 0)) return rc;
    if (by_size) by_size = false;
    else max_bitmaps = max_bitmaps * 3 / 4;
  }
  std::vector<int32_t> hidx((size_t)N, -1), nodes_of((size_t)std::max<int64_t>(max_bitmaps, 1), 0);
  for (int64_t h = 0; h < max_bitmaps; ++h) {
    hidx[(size_t)pop[h].second] = (int32_t)h;
    nodes_of[(size_t)h] = pop[h].second;
  }
  char* c = (char*)p;
  ctx->otf_block = p;
  ctx->otf_bytes = bytes;
  ctx->otf_hidx = (int32_t*)c;
  int32_t* d_nodes_of = (int32_t*)(c + b_hidx);
  ctx->otf_hbits = (uint32_t*)(c + b_hidx + b_nodes);
  ctx->otf_sbits = (uint32_t*)(c + b_hidx + b_nodes + b_bits);
  ctx->otf_uprefix = (int64_t*)(c + b_hidx + b_nodes + b_bits + b_sbits);
  int32_t* pos_of = (int32_t*)(c + b_hidx + b_nodes + b_bits + b_sbits + b_pre);
  int64_t* up = (int64_t*)((char*)pos_of + b_order);
  auto bail = [&](int rc) { release_onthefly(ctx); return rc; };
  if (cudaMemcpyAsync(ctx->otf_hidx, hidx.data(), (size_t)N * 4, cudaMemcpyHostToDevice, st) !=
          cudaSuccess ||
      cudaMemcpyAsync(d_nodes_of, nodes_of.data(), nodes_of.size() * 4, cudaMemcpyHostToDevice,
                      st) != cudaSuccess ||
      cudaMemsetAsync(ctx->otf_hbits, 0, b_bits + b_sbits, st) != cudaSuccess)
    return bail(fail(MOCHY_E_CUDA, "on-the-fly set-up copy failed"));
  ctx->otf_by_size = by_size;
  if (by_size) {
    ctx->otf_pwords = Wp;
    ctx->otf_pbits = (uint32_t*)((char*)ctx->otf_hbits + b_one);
    ctx->otf_id_of = (int32_t*)((char*)pos_of + b_pos);
    ctx->otf_cls = (int32_t*)((char*)pos_of + b_pos + b_id);
    ctx->otf_draws = up;
    ctx->otf_max_draws = (int64_t)(b_up / 8);
    int32_t* counts = ctx->otf_cls + kOtfSizes + 1;
    if (cudaMemsetAsync(counts, 0, kOtfSizes * 4, st) != cudaSuccess)
      return bail(fail(MOCHY_E_CUDA, "on-the-fly set-up copy failed"));
    if (E > 0) {
      k_otf_sizes<<<(unsigned)std::min<int64_t>(ceil_div(E, 256), (int64_t)ctx->num_sms * 4), 256, 0,
                    st>>>(E, ctx->esize, counts);
      k_otf_starts<<<1, 32, 0, st>>>(counts, ctx->otf_cls);
      k_otf_positions<<<(unsigned)ceil_div(E, 256), 256, 0, st>>>(E, ctx->esize, counts,
                                                                 pos_of, ctx->otf_id_of);
      note_launch();
      note_launch();
      note_launch();
    }
  }
  if (max_bitmaps > 0) {
    k_otf_bits<<<(unsigned)std::min<int64_t>(max_bitmaps, 4096), 256, 0, st>>>(
        max_bitmaps, W, d_nodes_of, ctx->voff, ctx->vedge, ctx->otf_hbits, Wp, pos_of,
        by_size ? ctx->otf_pbits : nullptr);
    note_launch();
  }
  if (E > 0 && !by_size) {
    k_otf_size_bits<<<ceil_div(E, 256), 256, 0, st>>>(E, W, ctx->esize, ctx->otf_sbits);
    note_launch();
  }
  OtfArgs g{};
  g.n_edges = E;
  g.W = W;
  g.eoff = ctx->eoff;
  g.enode = ctx->enode;
  g.esize = ctx->esize;
  g.voff = ctx->voff;
  g.vedge = ctx->vedge;
  g.hidx = ctx->otf_hidx;
  g.hbits = ctx->otf_hbits;
  g.sbits = ctx->otf_sbits;
  g.up = up;
  if (E > 0 && max_bitmaps == (int64_t)pop.size()) {
    k_otf_after<<<(unsigned)std::min<int64_t>(ceil_div(E, kAfterThreads / 32),
                                              (int64_t)ctx->num_sms * 16),
                  kAfterThreads, 0, st>>>(g);
    note_launch();
  } else if (E > 0) {
    // nodes of high degree without a bitmap (a small budget): merge the lists
    const size_t smem = sizeof(OtfWarp) * kOtfWarps;
    const int rc = ensure_dynamic_smem((const void*)k_otf_degrees, smem);
    if (rc < 0) return bail(rc);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_otf_degrees, kOtfThreads, smem);
    const int64_t grid = std::min<int64_t>((int64_t)ctx->num_sms * std::max(per_sm, 1),
                                           (E + kOtfWarps - 1) / kOtfWarps);
    k_otf_degrees<<<(unsigned)grid, kOtfThreads, smem, st>>>(g);
    note_launch();
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return bail(cuda_fail(e, "on-the-fly degrees", __FILE__, __LINE__));
  {
    const int rc = scan_exclusive_i64(ctx, up, ctx->otf_uprefix, E + 1);
    if (rc < 0) return bail(rc);
  }
  int64_t total = 0;
  if (cudaMemcpyAsync(&total, ctx->otf_uprefix + E, 8, cudaMemcpyDeviceToHost, st) !=
          cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return bail(fail(MOCHY_E_CUDA, "on-the-fly prefix copy failed"));
  ctx->otf_wedges = total;
  ctx->otf_bitmaps = max_bitmaps;
  ctx->otf_words = W;
  ctx->otf_ready = true;
  return MOCHY_OK;
}

// MoCHy-A+ of `samples` draws without the line graph into d_hist (432,
// cleared here).  stats (may be null): [4] candidates, words, list
// entries, exact classifications.
int count_sampled_onthefly(mochy_ctx* ctx, int64_t samples, uint64_t seed, int64_t budget,
                           unsigned long long* d_hist, unsigned long long* d_stats) {
  if (samples <= 0) return fail(MOCHY_E_INVALID, "samples must be positive");
  MOCHY_TRY(prepare_onthefly(ctx, budget));
  if (ctx->otf_wedges == 0) return fail(MOCHY_E_INVALID, "the hypergraph has no hyperwedge");
  cudaStream_t st = ctx->stream;
  MOCHY_CUDA(cudaMemsetAsync(d_hist, 0, 432 * 8, st));
  MOCHY_CUDA(cudaMemsetAsync(ctx->counters, 0, 16 * sizeof(int32_t), st));
  OtfArgs g{};
  g.n_edges = ctx->n_edges;
  g.W = ctx->otf_words;
  g.eoff = ctx->eoff;
  g.enode = ctx->enode;
  g.esize = ctx->esize;
  g.voff = ctx->voff;
  g.vedge = ctx->vedge;
  g.hidx = ctx->otf_hidx;
  g.hbits = ctx->otf_hbits;
  g.sbits = ctx->otf_sbits;
  g.uprefix = ctx->otf_uprefix;
  g.n_wedges = ctx->otf_wedges;
  g.lut3 = ctx->tables.lut3;
  g.hist = d_hist;
  g.theta = ctx->theta;
  g.seed = seed;
  g.samples = samples;
  g.queue = ctx->counters + 4;   // 64-bit counter over words 4 and 5
  g.stats = d_stats;
  if (d_stats) MOCHY_CUDA(cudaMemsetAsync(d_stats, 0, 4 * 8, st));
  if (ctx->otf_by_size) {
    g.Wp = ctx->otf_pwords;
    g.pbits = ctx->otf_pbits;
    g.cls = ctx->otf_cls;
    g.id_of = ctx->otf_id_of;
    g.draws = (int2*)ctx->otf_draws;
    int per_sm = 0;
    MOCHY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_otf_classify,
                                                             kOtfScanThreads, 0));
    const int64_t warps = (int64_t)ctx->num_sms * std::max(per_sm, 1) * (kOtfScanThreads / 32);
    const int64_t steps = std::max<int64_t>(g.W / kOtfDrawWords, 1);
    for (int64_t first = 0; first < samples; first += ctx->otf_max_draws) {
      g.first = first;
      g.n_draws = std::min(samples - first, ctx->otf_max_draws);
      // a scan is cut when there are fewer than kOtfItems draws to a warp,
      // into parts of kOtfMinSteps steps at least
      g.n_seg = std::max<int64_t>(
          1, std::min((kOtfItems * warps + g.n_draws - 1) / g.n_draws, steps / kOtfMinSteps));
      if (first > 0) MOCHY_CUDA(cudaMemsetAsync(g.queue, 0, 8, st));
      k_otf_draw<<<(unsigned)std::min<int64_t>(ceil_div(g.n_draws, kOtfScanThreads / 32),
                                               (int64_t)ctx->num_sms * 8),
                   kOtfScanThreads, 0, st>>>(g);
      k_otf_classify<<<(unsigned)std::min<int64_t>(
                           ceil_div(g.n_draws * g.n_seg, kOtfScanThreads / 32),
                           (int64_t)ctx->num_sms * std::max(per_sm, 1)),
                       kOtfScanThreads, 0, st>>>(g);
      note_launch();
      MOCHY_LAUNCHED();
    }
    return MOCHY_OK;
  }
  const size_t smem = otf_smem_bytes();
  MOCHY_TRY(ensure_dynamic_smem((const void*)k_otf_sample, smem));
  int per_sm = 0;
  MOCHY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_otf_sample, kOtfThreads,
                                                           smem));
  const int64_t grid = std::min<int64_t>((int64_t)ctx->num_sms * std::max(per_sm, 1),
                                         (samples + kOtfWarps - 1) / kOtfWarps);
  k_otf_sample<<<(unsigned)grid, kOtfThreads, smem, st>>>(g);
  MOCHY_LAUNCHED();
  return MOCHY_OK;
}

}  // namespace mochy

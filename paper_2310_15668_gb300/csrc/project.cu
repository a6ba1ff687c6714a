// Line-graph construction (Section 2.1 "Line Graph"; Algorithm
// "hyperwedge_counting", Section 3.1).
//
// The paper visits, for each e_i and each v in e_i, every e_j in E_v and
// increments omega(e_i, e_j) in a hash map.  Here one warp builds row e_i, a
// chunk of 1,024 neighbour ids at a time (one 32-bit word of ids a lane): the
// union of the incidence lists E_v of its nodes as bits, then, at the place
// that the bits before it give, the mask of the nodes that hold each
// neighbour (bit p: the p-th node of e_i).  Two passes: row lengths (and how
// many neighbours share two nodes or more), then entries.  Nodes of high
// degree have their list as a bitmap too, so that the first step costs them
// one word per 32 ids; rows without such a node skip the chunks that none of
// their lists reaches.
// Issue and shared-memory latency bound it (4.7 warp instructions an entry, 42 %
// of the issue slots, 20 warps an SM): 100,001 Zipf(1.0) hyperedges, 9.9 GB of
// line graph: loading and projecting 62.7 ms with windows of list entries, 14
// here (4 or 6 blocks an SM instead of 8: 21 and 18, blocks of 256 threads 19).
#include "common.cuh"

namespace mochy {
namespace {

constexpr int kProjThreads = 128;
constexpr int kProjWarps = kProjThreads / 32;
constexpr int kChunkBits = 10;                   // ids per chunk: one word a lane
constexpr int kChunk = 1 << kChunkBits;

// A node gets a bitmap when it lies in at least this many hyperedges of its
// unit: four or more per chunk, so that its words are worth reading (a 128th
// and a 512th instead of a 256th: within 2 % at 10,000 and 100,001
// hyperedges).  The bitmaps then take at most 9 words per incidence.
__device__ __forceinline__ int64_t bitmap_degree(int64_t unit_edges) {
  return max((int64_t)32, unit_edges >> 8);
}

struct ProjArgs {
  int64_t n_edges, n_nodes;
  const int64_t* eoff;
  const int32_t* enode;
  const int64_t* voff;
  const int32_t* vedge;
  const uint8_t* esize;
  int n_units;
  const int64_t* nseg;     // [U+1] node and hyperedge ranges (batch)
  const int64_t* eseg;
  int64_t* bitmap;         // [N] first word of a node's bitmap or -1
  uint32_t* bits;          // bitmaps over the hyperedges of a unit, from its first word
  int64_t* deg;            // [E] row length
  int64_t* below;          // [E] neighbours before the row
  int32_t* heavy;          // [E] neighbours that share two nodes or more
  const int64_t* noff;
  uint2* nadj;
};

// warp per node: the bitmap of a node of high degree
__global__ void __launch_bounds__(256)
k_project_bitmaps(ProjArgs g, unsigned long long* __restrict__ cursor) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t v = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < g.n_nodes;
       v += nw) {
    const int64_t b = g.voff[v], e = g.voff[v + 1];
    int64_t e0 = 0, e1 = g.n_edges;
    int64_t at = -1;
    if (e - b >= 32) {
      if (g.n_units > 1) {
        const int u = seg_of(g.nseg, g.n_units, v);
        e0 = g.eseg[u];
        e1 = g.eseg[u + 1];
      }
      if (e - b >= bitmap_degree(e1 - e0)) {
        const int64_t words = ((e1 + 31) >> 5) - (e0 >> 5);
        if (lane == 0) at = (int64_t)atomicAdd(cursor, (unsigned long long)words);
        at = __shfl_sync(0xffffffffu, at, 0);
        for (int64_t p = b + lane; p < e; p += 32) {
          const int32_t k = g.vedge[p];
          atomicOr(&g.bits[at + (k >> 5) - (e0 >> 5)], 1u << (k & 31));
        }
      }
    }
    if (lane == 0) g.bitmap[v] = at;
  }
}

// BITS: some node may have a bitmap
template <bool FILL, bool BITS>
__global__ void __launch_bounds__(kProjThreads) k_project_rows(ProjArgs g) {
  __shared__ uint2 s_word[kProjWarps][32];      // neighbour bits, entries before the word
  __shared__ uint32_t s_twice[kProjWarps][32];  // ids met twice or more
  __shared__ uint32_t s_mask[FILL ? kProjWarps : 1][FILL ? kChunk : 1];
  __shared__ uint16_t s_id[FILL ? kProjWarps : 1][FILL ? kChunk : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint2* word = s_word[warp];
  uint32_t* twice = s_twice[warp];
  uint32_t* mask = s_mask[FILL ? warp : 0];
  uint16_t* id = s_id[FILL ? warp : 0];
  const int64_t nw = (int64_t)gridDim.x * kProjWarps;
  for (int64_t i = (int64_t)blockIdx.x * kProjWarps + warp; i < g.n_edges; i += nw) {
    const int64_t eb = g.eoff[i];
    const int A = (int)(g.eoff[i + 1] - eb);
    const bool masked = A <= kMaskedMax;
    int64_t e0 = 0, e1 = g.n_edges;
    if (g.n_units > 1) {
      const int u = seg_of(g.nseg, g.n_units, g.enode[eb]);
      e0 = g.eseg[u];
      e1 = g.eseg[u + 1];
    }
    // node p = lane + 32 s: its list, the next entry of it and its bitmap
    int64_t cur[2], last[2], bm[2];
    int32_t next[2];
    int cnt[2] = {0, 0};
    unsigned hubs[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int p = lane + 32 * s;
      cur[s] = last[s] = 0;
      bm[s] = -1;
      next[s] = 0x7fffffff;
      if (p < A) {
        const int32_t v = g.enode[eb + p];
        cur[s] = g.voff[v];
        last[s] = g.voff[v + 1];
        if (BITS) bm[s] = g.bitmap[v];
        if (bm[s] < 0) next[s] = g.vedge[cur[s]];
      }
      hubs[s] = __ballot_sync(0xffffffffu, bm[s] >= 0);
    }
    const bool any_hub = (hubs[0] | hubs[1]) != 0u;
    const int w0 = (int)(e0 >> 5), w1 = (int)((e1 + 31) >> 5);   // words of the unit
    const int self_w = (int)(i >> 5);
    const uint32_t self = 1u << (i & 31);
    int n_deg = 0, n_below = 0, n_heavy = 0;   // of this lane's words
    int64_t out = FILL ? g.noff[i] : 0;
    int c = w0 >> 5;
    while (true) {
      if (!any_hub) {
        const int32_t nx = (int32_t)__reduce_min_sync(0xffffffffu, (unsigned)min(next[0], next[1]));
        if (nx == 0x7fffffff) break;
        c = nx >> kChunkBits;
      } else if (32 * c >= w1) {
        break;
      }
      const int32_t end = (int32_t)min((int64_t)0x7fffffff, ((int64_t)c + 1) << kChunkBits);
      const int w = 32 * c + lane;
      uint32_t U = 0u, T = 0u;
#pragma unroll
      for (int s = 0; s < 2; ++s)
        for (unsigned h = hubs[s]; h; h &= h - 1u) {
          const int l = __ffs(h) - 1;
          const int64_t b = __shfl_sync(0xffffffffu, bm[s], l);
          uint32_t v = w >= w0 && w < w1 ? __ldg(&g.bits[b + (w - w0)]) : 0u;
          if (FILL) {
            const int n = __reduce_add_sync(0xffffffffu, __popc(v));
            if (lane == l) cnt[s] = n;
          }
          if (w == self_w) v &= ~self;
          T |= U & v;
          U |= v;
        }
      const unsigned near0 = __ballot_sync(0xffffffffu, next[0] < end);
      const unsigned near1 = A > 32 ? __ballot_sync(0xffffffffu, next[1] < end) : 0u;
      if (near0 | near1) {
        word[lane].x = U;
        twice[lane] = 0u;
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 2; ++s)
          for (unsigned m = s ? near1 : near0; m; m &= m - 1u) {
            const int l = __ffs(m) - 1;
            const int64_t b = __shfl_sync(0xffffffffu, cur[s], l);
            const int64_t e = __shfl_sync(0xffffffffu, last[s], l);
            int total = 0;
            while (true) {
              const int64_t q = b + total + lane;
              const int32_t k = q < e ? g.vedge[q] : 0x7fffffff;
              const bool in = k < end;
              if (in && k != (int32_t)i) {
                const uint32_t bit = 1u << (k & 31);
                const uint32_t old = atomicOr(&word[(k >> 5) & 31].x, bit);
                if (!FILL && (old & bit)) atomicOr(&twice[(k >> 5) & 31], bit);
              }
              const int n = __popc(__ballot_sync(0xffffffffu, in));
              total += n;
              if (n < 32) break;
            }
            if (lane == l) cnt[s] = total;
          }
        __syncwarp();
        U = word[lane].x;
        T |= twice[lane];
      }
      if (!FILL) {
        n_deg += __popc(U);
        n_heavy += __popc(T);
        n_below += w < self_w ? __popc(U) : w == self_w ? __popc(U & (self - 1u)) : 0;
      } else {
        const int n = __popc(U);
        int incl = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += o;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        word[lane] = make_uint2(U, (uint32_t)(incl - n));
        for (int q = lane; q < total; q += 32) mask[q] = 0u;
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 2; ++s)
          for (unsigned m = __ballot_sync(0xffffffffu, cnt[s] > 0); m; m &= m - 1u) {
            const int l = __ffs(m) - 1;
            const int64_t b = __shfl_sync(0xffffffffu, cur[s], l);
            const int nl = __shfl_sync(0xffffffffu, cnt[s], l);
            for (int q = lane; q < nl; q += 32) {
              const int32_t k = g.vedge[b + q];
              if (k == (int32_t)i) continue;
              const uint2 wd = word[(k >> 5) & 31];
              const int at = (int)wd.y + __popc(wd.x & ((1u << (k & 31)) - 1u));
              if (masked) mask[at] |= 1u << l;
              else mask[at] += 1u;
              id[at] = (uint16_t)(k & (kChunk - 1));
            }
            __syncwarp();
          }
        const uint32_t k0 = (uint32_t)c << kChunkBits;
        for (int q = lane; q < total; q += 32) {
          const uint32_t k = k0 + id[q];
          g.nadj[out + q] = make_uint2(k | (uint32_t)g.esize[k] << kIdBits, mask[q]);
        }
        out += total;
        __syncwarp();
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if (cnt[s]) {
          cur[s] += cnt[s];
          if (bm[s] < 0) next[s] = cur[s] < last[s] ? g.vedge[cur[s]] : 0x7fffffff;
          cnt[s] = 0;
        }
      }
      ++c;
    }
    if (!FILL) {
      n_deg = __reduce_add_sync(0xffffffffu, n_deg);
      n_below = __reduce_add_sync(0xffffffffu, n_below);
      n_heavy = __reduce_add_sync(0xffffffffu, n_heavy);
      if (lane == 0) {
        g.deg[i] = n_deg;
        g.below[i] = n_below;
        g.heavy[i] = n_heavy;
      }
    }
  }
}

__global__ void k_upper(int64_t n_edges, const int64_t* __restrict__ noff,
                        const int64_t* __restrict__ deg, const int64_t* __restrict__ below,
                        int64_t* __restrict__ ustart, int64_t* __restrict__ uplen,
                        int* __restrict__ maxdeg) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_edges) return;
  ustart[i] = noff[i] + below[i];
  uplen[i] = deg[i] - below[i];
  atomicMax(maxdeg, (int)deg[i]);
}

// Estimated work of staging row a in the exact count: the neighbours' row
// lengths it will scan.  Keys sort rows by decreasing work.
__global__ void k_row_cost(int64_t n_edges, const int64_t* __restrict__ noff,
                           const uint2* __restrict__ nadj, uint32_t* __restrict__ key,
                           uint32_t* __restrict__ val) {
  const int64_t a = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (a >= n_edges) return;
  double c = 0.0;
  for (int64_t p = noff[a] + lane; p < noff[a + 1]; p += 32) {
    const uint32_t b = ent_id(nadj[p]);
    c += (double)(noff[b + 1] - noff[b]);
  }
  for (int d = 16; d; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
  c += (double)(noff[a + 1] - noff[a]);
  if (lane == 0) {
    key[a] = ~__float_as_uint((float)c);
    val[a] = (uint32_t)a;
  }
}

// unit of each row of an order (rows of a batch)
__global__ void k_row_units(int64_t n, const uint32_t* __restrict__ row,
                            const int64_t* __restrict__ eoff, const int32_t* __restrict__ enode,
                            const int64_t* __restrict__ nseg, int n_units,
                            uint32_t* __restrict__ unit) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) unit[i] = (uint32_t)seg_of(nseg, n_units, enode[eoff[row[i]]]);
}

}  // namespace

int project_graph(mochy_ctx* ctx) {
  release_projection(ctx);
  const int64_t E = ctx->n_edges;
  cudaStream_t st = ctx->stream;
  void* p;
  MOCHY_TRY(dev_alloc(ctx, &p, sizeof(int64_t) * (size_t)(E + 1)));
  ctx->noff = (int64_t*)p;
  MOCHY_TRY(dev_alloc(ctx, &p, sizeof(int64_t) * (size_t)std::max<int64_t>(E, 1)));
  ctx->ustart = (int64_t*)p;
  MOCHY_TRY(dev_alloc(ctx, &p, sizeof(int64_t) * (size_t)(E + 1)));
  ctx->uprefix = (int64_t*)p;
  MOCHY_TRY(dev_alloc(ctx, &p, sizeof(int32_t) * (size_t)std::max<int64_t>(E, 1)));
  ctx->heavy_deg = (int32_t*)p;
  if (E == 0) {
    MOCHY_CUDA(cudaMemsetAsync(ctx->noff, 0, 8, st));
    MOCHY_CUDA(cudaMemsetAsync(ctx->uprefix, 0, 8, st));
    ctx->n_wedges = 0;
    ctx->max_deg = 0;
    ctx->projected = true;
    return MOCHY_OK;
  }
  void* t;
  MOCHY_TRY(scratch(ctx, 0, (size_t)(E + 1) * 8 * 3, &t));
  int64_t* deg = (int64_t*)t;
  int64_t* below = deg + (E + 1);
  int64_t* uplen = below + (E + 1);
  MOCHY_CUDA(cudaMemsetAsync(deg, 0, (size_t)(E + 1) * 8 * 3, st));
  // Bitmaps of the nodes of high degree (at most 9 words per incidence).  The
  // rows come out the same without them, so they do not take memory that the
  // line graph needs.
  const size_t b_nodes = (size_t)ctx->n_nodes * 8, b_bits = (size_t)ctx->n_inc * 36 + 256;
  void* t2 = nullptr;
  const int rc2 = room_for(ctx, scratch_growth(ctx, 2, b_nodes + 8 + b_bits))
                      ? scratch(ctx, 2, b_nodes + 8 + b_bits, &t2) : MOCHY_E_NOMEM;
  if (rc2 < 0 && rc2 != MOCHY_E_NOMEM) return rc2;
  if (rc2 < 0) t2 = nullptr;
  ProjArgs g;
  g.n_edges = E;
  g.n_nodes = ctx->n_nodes;
  g.eoff = ctx->eoff;
  g.enode = ctx->enode;
  g.voff = ctx->voff;
  g.vedge = ctx->vedge;
  g.esize = ctx->esize;
  g.n_units = ctx->n_units;
  g.nseg = ctx->d_nseg;
  g.eseg = ctx->d_nseg ? ctx->d_nseg + ctx->n_units + 1 : nullptr;
  g.bitmap = (int64_t*)t2;
  g.bits = t2 ? (uint32_t*)((char*)t2 + b_nodes + 8) : nullptr;
  g.deg = deg;
  g.below = below;
  g.heavy = ctx->heavy_deg;
  g.noff = ctx->noff;
  g.nadj = nullptr;
  if (t2) {
    MOCHY_CUDA(cudaMemsetAsync((char*)t2 + b_nodes, 0, 8 + b_bits, st));
    k_project_bitmaps<<<(unsigned)std::min<int64_t>(ceil_div(ctx->n_nodes, 8),
                                                   (int64_t)ctx->num_sms * 8),
                        256, 0, st>>>(g, (unsigned long long*)((char*)t2 + b_nodes));
    MOCHY_LAUNCHED();
  }
  const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(E, kProjWarps),
                                                    (int64_t)ctx->num_sms * 16);
  auto lengths = t2 ? k_project_rows<false, true> : k_project_rows<false, false>;
  lengths<<<grid, kProjThreads, 0, st>>>(g);
  MOCHY_LAUNCHED();
  MOCHY_TRY(scan_exclusive_i64(ctx, deg, ctx->noff, E + 1));
  int64_t total = 0;
  MOCHY_CUDA(cudaMemcpyAsync(&total, ctx->noff + E, 8, cudaMemcpyDeviceToHost, st));
  MOCHY_CUDA(cudaStreamSynchronize(st));
  const size_t bytes = (size_t)std::max<int64_t>(total, 1) * sizeof(uint2);
  int rc = dev_alloc(ctx, &p, bytes);
  if (rc == MOCHY_E_NOMEM && t2) {
    MOCHY_TRY(drop_scratch(ctx, 2));
    t2 = nullptr;
    rc = dev_alloc(ctx, &p, bytes);
  }
  if (rc < 0) {
    release_projection(ctx);
    return fail(MOCHY_E_NOMEM, "line graph needs " + std::to_string(bytes) +
                                   " bytes of device memory");
  }
  ctx->nadj = (uint2*)p;
  g.nadj = ctx->nadj;
  auto entries = t2 ? k_project_rows<true, true> : k_project_rows<true, false>;
  entries<<<(unsigned)std::min<int64_t>(ceil_div(E, kProjWarps), (int64_t)ctx->num_sms * 8),
            kProjThreads, 0, st>>>(g);
  MOCHY_LAUNCHED();
  int* maxdeg = ctx->counters + 2;
  MOCHY_CUDA(cudaMemsetAsync(maxdeg, 0, 4, st));
  k_upper<<<ceil_div(E, 256), 256, 0, st>>>(E, ctx->noff, deg, below, ctx->ustart, uplen, maxdeg);
  MOCHY_LAUNCHED();
  MOCHY_TRY(scan_exclusive_i64(ctx, uplen, ctx->uprefix, E + 1));
  int32_t md = 0;
  MOCHY_CUDA(cudaMemcpyAsync(&md, maxdeg, 4, cudaMemcpyDeviceToHost, st));
  MOCHY_CUDA(cudaStreamSynchronize(st));
  ctx->n_wedges = total / 2;
  ctx->max_deg = md;
  ctx->projected = true;
  if (ctx->budget > 0) MOCHY_TRY(drop_scratch(ctx, 2));   // a budget counts what is held
  return MOCHY_OK;
}

// Rows by decreasing estimated work, for the kernels that take rows from a work
// queue (built on first use, released with the line graph).
int ensure_row_order(mochy_ctx* ctx) {
  if (ctx->row_order || ctx->n_edges == 0) return MOCHY_OK;
  const int64_t E = ctx->n_edges;
  cudaStream_t st = ctx->stream;
  void* t2;
  MOCHY_TRY(scratch(ctx, 2, (size_t)E * 8, &t2));
  uint32_t* key = (uint32_t*)t2;
  uint32_t* val = key + E;
  k_row_cost<<<ceil_div(E, 8), 256, 0, st>>>(E, ctx->noff, ctx->nadj, key, val);
  MOCHY_LAUNCHED();
  MOCHY_TRY(radix_sort_pairs_u32(ctx, key, val, E, 32));
  if (ctx->n_units > 1) {
    // a batch: rows grouped by hypergraph (stable), so that a block's
    // consecutive rows mostly belong to one of them
    k_row_units<<<ceil_div(E, 256), 256, 0, st>>>(E, val, ctx->eoff, ctx->enode, ctx->d_nseg,
                                                  ctx->n_units, key);
    MOCHY_LAUNCHED();
    MOCHY_TRY(radix_sort_pairs_u32(ctx, key, val, E, bits_for(ctx->n_units)));
  }
  void* p;
  const int rc = dev_alloc(ctx, &p, sizeof(int32_t) * (size_t)E);
  if (rc == MOCHY_E_NOMEM && ctx->heavy_deg) {
    // no room for both: the order takes the place of the heavy degrees, which
    // only the levels read
    release_levels(ctx);
    p = ctx->heavy_deg;
    ctx->heavy_deg = nullptr;
  } else if (rc < 0) {
    return rc;
  }
  ctx->row_order = (int32_t*)p;
  MOCHY_CUDA(cudaMemcpyAsync(ctx->row_order, val, (size_t)E * 4, cudaMemcpyDeviceToDevice, st));
  return MOCHY_OK;
}

}  // namespace mochy

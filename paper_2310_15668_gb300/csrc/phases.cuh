// Phase timing of the exact counts.
#pragma once

#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "common.cuh"

namespace mochy {

// Phase timing when tracing is on (mochy_trace or MOCHY_TRACE=1): events
// around each kernel on the context's stream, kept in the context and, with
// MOCHY_TRACE set, printed to stderr.
struct PhaseTimer {
  bool on = false, print = false;
  cudaStream_t st;
  cudaEvent_t ev[kMaxPhases];
  const char* name[kMaxPhases];
  int n = 0;
  bool stats = false;
  PhaseTimer(const mochy_ctx* c) : st(c->stream) {
    const char* e = getenv("MOCHY_TRACE");
    print = e && e[0] && e[0] != '0';
    on = c->trace > 0 || print;
    stats = c->trace > 1 || print;
  }
  void mark(const char* what) {
    if (!on || n >= kMaxPhases) return;
    cudaEventCreate(&ev[n]);
    cudaEventRecord(ev[n], st);
    name[n++] = what;
  }
  void restart() {
    for (int i = 0; i < n; ++i) cudaEventDestroy(ev[i]);
    n = 0;
  }
  void report(mochy_ctx* c) {
    if (!on || n < 2) return;
    if (!stats) memset(c->last_stats, 0, sizeof(c->last_stats));
    cudaEventSynchronize(ev[n - 1]);
    c->n_phases = 0;
    for (int i = 1; i < n; ++i) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[i - 1], ev[i]);
      snprintf(c->phase_name[c->n_phases], sizeof(c->phase_name[0]), "%s", name[i]);
      c->phase_ms[c->n_phases++] = ms;
    }
    if (stats)
    {
      cudaMemcpy(c->last_stats, c->stats, 8 * sizeof(unsigned long long), cudaMemcpyDeviceToHost);
      cudaMemcpy(c->last_stats + 8, c->stats + 72, 8 * sizeof(unsigned long long),
                 cudaMemcpyDeviceToHost);
      cudaMemcpy(c->last_stats + 16, c->stats + 80, 8 * sizeof(unsigned long long),
                 cudaMemcpyDeviceToHost);
    }
    if (stats && print) {
      unsigned long long combo[64];
      cudaMemcpy(combo, c->stats + 8, sizeof(combo), cudaMemcpyDeviceToHost);
      fprintf(stderr, "[mochy]   rest combinations (xa,xb,xt): ");
      for (int q = 0; q < 64; ++q)
        if (combo[q]) fprintf(stderr, "(%d,%d,%d)=%llu ", q >> 4, (q >> 2) & 3, q & 3, combo[q]);
      fprintf(stderr, "\n");
    }

    if (print) {
      fprintf(stderr, "[mochy] split exact: E=%lld dense=%lld (threshold %d, %lld words) heavy=%lld\n",
              (long long)c->n_edges, (long long)c->n_dense, c->dense_thr_used,
              (long long)c->wwords, (long long)c->n_heavy);
      for (int i = 0; i < c->n_phases; ++i)
        fprintf(stderr, "[mochy]   %-18s %10.3f ms\n", c->phase_name[i], c->phase_ms[i]);
      if (stats)
        fprintf(stderr, "[mochy]   words %llu  candidates %llu  table %llu  exact %llu  light %llu\n",
                c->last_stats[0], c->last_stats[1], c->last_stats[2], c->last_stats[3],
                c->last_stats[4]);
    }
    for (int i = 0; i < n; ++i) cudaEventDestroy(ev[i]);
    n = 0;
  }
};

}  // namespace mochy

// wave.cuh -- launch interface of the wavefront solver (wave.cu).
#pragma once

#include "common.cuh"
#include "kernels.cuh"

namespace pc {

// One query as the wavefront kernels see it (device pointers; byte offsets of
// a group's shared-memory region and of its device scratch).
struct WaveQuery {
  int W, L, A, P, TW;
  int s_begin, n_strips;
  int divS; uint32_t divM;   // i / A = (i * divM) >> (31 + divS) for i < 2^31
  const int16_t* strip_row;
  const int32_t* row_off;
  const int32_t* ppos;
  OccStream occ;
  const uint32_t* occ_bits;
  int64_t words_per_cfg;
  uint32_t cfg0;
  Outputs out;
  int want_mass;
  long long item0, n_cfg;    // the query's work items
  int NR;                    // word rows of the unvisited map held in shared memory
  int nr_mask;               // row w has slot w & nr_mask
  int cap;                   // frontier entries held in shared memory (two levels)
  int ring_mask;             // layers of the mass rings - 1, or -1: every layer has its own plane
  int o_win, o_queue;        // shared memory: window, queues (row offsets at a fixed place)
  long long a_back, a_over, a_occ, a_nu;  // scratch: evicted rows, overflow maps, occupancy, mass rings
};

// Queries of one launch and where its groups find their work.
struct WaveArgs {
  WaveQuery q0;              // the query, if nq == 1
  const WaveQuery* qs;       // [nq] by increasing item0
  int nq;
  long long n_items;
  unsigned long long* work;     // next work item (or entry of list)
  unsigned long long* list;     // percolating items whose mass is wanted
  unsigned long long* list_n;
  unsigned long long* hard;     // items whose frontier outgrew the mass rings
  unsigned long long* hard_n;
  int group_smem;
  char* scratch;
  long long scratch_stride;
};

// Inspects the queries (stream-ordered, no host synchronisation).
pc_status run_wave(const StreamQuery* qs, int nq, cudaStream_t st);
// Threads that work on one configuration of an A-column lattice when n_all
// configurations are inspected together on the current device.
int wave_threads(int A, long long n_all);

}  // namespace pc

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
  float density, density_most;  // of metallic sites: as levels, and as the start layer, are sized for
  long long item0, n_cfg;    // the query's work items
  int NR;                    // word rows of the unvisited map held in shared memory
  int nr_mask;               // row w has slot w & nr_mask
  int cap;                   // frontier entries held in shared memory (two levels)
  int ring_mask;             // layers of the mass rings - 1, or -1: every layer has its own plane
  int o_win, o_queue;        // shared memory: window, queues (row offsets at a fixed place)
  int o_occ, o_tab, tab_bits;  // occupancy (-1: in scratch), hash tables and their size
  long long a_back, a_over, a_occ, a_nu;  // scratch: evicted rows, overflow maps, occupancy, mass rings
};

// A configuration between two launches over drawn rows.
struct WaveState {
  int phase;  // 0: not begun, 1: waits for rows, 2: done
  int m, wb, G, olo, ohi;
  unsigned total, n0;
};

// Queries of one launch and where its groups find their work.
struct WaveArgs {
  WaveQuery q0;              // the query, if nq == 1
  const WaveQuery* qs;       // [nq] by increasing item0
  int nq;
  long long n_items;
  unsigned long long* work;  // next work item
  unsigned long long* count; // percolating items whose mass is wanted; items left to planes
  int hard;                  // mass launches: only the items marked by the first one
  int full;                  // verdicts and masses in one launch
  unsigned long long min_count, max_count;  // mass launches: run for so many percolating items
  int group_smem;
  Gate gate;
  WaveState* state;          // [n_items]: configurations over drawn rows
  int rows_ready;            // word rows drawn
  char* scratch;
  long long scratch_stride;
};

// Device memory that a caller holds for one query's run.
struct WaveMemory {
  unsigned long long* ctr;   // 8 zeroed counters
  char* scratch;
  size_t bytes;              // for one configuration at least (a streamed solver's slot is larger:
                             // its two FP32 planes of L + 4 layers and its bytes of degrees exceed
                             // this solver's two of L layers and four bit maps)
  long long max_groups;      // configurations in work at once
  bool warps = false;        // groups of one warp too (else a configuration is a CTA's)
};
// Whether m holds at least a third of the groups that the device would take at
// once (fewer leave SMs idle).
bool wave_memory_suffices(const StreamQuery& q, const WaveMemory& m);

// Inspects the queries (stream-ordered, no host synchronisation).  Without m
// the scratch is allocated on st, at most `limit` bytes where that is enough
// for one configuration; with m (one query) nothing is allocated.
constexpr size_t kWaveLimit = 24ull << 30;
pc_status run_wave(const StreamQuery* qs, int nq, cudaStream_t st, const WaveMemory* m = nullptr,
                   size_t limit = kWaveLimit);
// Threads that work on one configuration of q (its levels) when n_all
// configurations are inspected together on nsm SMs.
int wave_threads(const StreamQuery& q, long long n_all, int nsm);
// Whether the streamed and blocked solvers, which work on a configuration with
// the whole device, are the faster ones for n configurations: each of this
// solver's is one SM's, so that few of them with large levels leave the device
// idle; and a cross-section beyond one SM's shared memory (W >= 129), or levels
// beyond its queue, are walked in device memory.  Where the line lies, in sites
// of a level (us of this solver / of the others): W = 64, L = 32, one
// configuration, p = 0.3 (2,700 sites a level) 1,370 / 1,530, p = 0.4 (4,200)
// 1,750 / 1,400, p = 0.95 4,690 / 1,240; 16 of them, p = 0.4 1,860 / 1,900, p =
// 0.55 (6,300) 2,480 / 1,780; 64 of them, p = 0.75 as fast.  Beyond the queue:
// W = 90, L = 128, verdicts, one configuration, p = 0.18 (930 sites) 1,900 /
// 7,800, p = 0.21 (2,200) 12,000 / 5,140; W = 128, L = 512, p = 0.165 (820)
// 127,000 / 57,100, 16 of them, L = 128, 19,900 / 18,300.  Verdicts of one: W =
// 30, L = 180, p = 0.95 (2,580) 881 / 764, p = 0.7 (1,850) 700 / 775; W = 52, L =
// 312, p = 0.35 (2,290) 1,841 / 1,675, p = 0.25 (1,220) 1,498 / 1,857.
bool wave_is_slower(const Lattice& lat, double density, long long n, bool bits_only);
void release_wave();  // pc_shutdown

}  // namespace pc

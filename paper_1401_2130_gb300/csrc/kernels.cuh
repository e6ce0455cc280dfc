// kernels.cuh -- launch interfaces between the C-ABI layer and the kernels.
#pragma once

#include "common.cuh"

namespace pc {

// Outputs of one inspection call (device pointers; optional ones may be null).
struct Outputs {
  uint8_t* verdict;
  int32_t* first_hit;
  float* mass;
  int32_t* m_stop;
  unsigned long long* n_perc;  // atomically incremented per percolating config
};

// Work that runs only where a density sampled on the device (65,536ths of the
// sites) lies in [lo, hi).  Open if at is null.
struct Gate {
  const unsigned* at = nullptr;
  unsigned lo = 0, hi = ~0u;
  __device__ bool closed() const { return at && (*at < lo || *at >= hi); }
};

// Resident (shared-memory) solver, resident.cu.
struct ResidentArgs {
  Lattice lat;
  OccStream occ;             // occupancy stream (cfg field set per config)
  const uint32_t* occ_bits;  // caller occupancy [n_cfg][words_per_cfg] or null
  int64_t words_per_cfg;
  int64_t n_cfg;
  uint32_t cfg0;
  uint8_t* verdict;
  int32_t* first_hit;
  float* mass;
  int32_t* m_stop;
  unsigned long long* n_perc;
  unsigned long long* work;  // zeroed work counter
  int prep_chunk;            // layers prepared per lazy chunk (>= 3)
  int bits_only = 0;         // reached set only: no FP32 sweep, mass written 0
  int verdict_first = 0;     // reached set first, FP32 recursion only where it percolates
  Gate gate;
};
constexpr int kResidentMaxThreads = 640;  // resident CTA size limit: 20 warps at <= 96 registers
size_t resident_smem(const Lattice& lat);
pc_status launch_resident(const ResidentArgs& args, int threads, cudaStream_t st);
// CTA size of the resident solver for n configurations (route.h)
int resident_threads(const Lattice& lat, long long n);
// CTA size picked by the autotuner for (W, L, p bin) (batch.cu); times
// candidates on a miss, outside any stream capture
int tuned_threads(const Lattice& lat, double p, uint64_t seed, cudaStream_t st);
bool resident_fits(int W, int L);
void release_static();  // noalloc.cu: forget the static array's cached addresses

// Streamed solver for lattices beyond shared memory, stream.cu.
struct StreamQuery {
  Lattice lat;
  OccStream occ;
  const uint32_t* occ_bits;
  int64_t words_per_cfg;
  int64_t n_cfg;
  uint32_t cfg0;
  Outputs out;
  int bits_only = 0;  // reached set only: no FP units, mass written 0
  int verdict_first = 0;  // the caller asks for verdicts first (a hint: the outputs are the same)
  // device list of n_cfg configurations (indices from 0 within the query) to
  // solve, outputs written at those indices; null = configurations 0..n_cfg-1
  const int64_t* sel = nullptr;
  // caller occupancies: what the launches are sized for (levels, start layer),
  // and the sampled densities that they are for
  double density = 0.2, density_most = 0.25;
  Gate gate;
};
// q on the resident solver, in CTAs of resident_threads; work: a zeroed counter.
pc_status run_resident(const StreamQuery& q, unsigned long long* work, cudaStream_t st);
ResidentArgs resident_args(const StreamQuery& q);  // without a work counter
// The queries in one launch for each class of shared memory; work: three zeroed
// counters; threads[q]: the CTA size that query q ran with.
pc_status run_residents(const StreamQuery* qs, int nq, unsigned long long* work, int* threads, cudaStream_t st);
// The solver that a call without a PC_MODE flag takes for n configurations of
// occupancy stream occ.
enum class Route { kWave, kResident, kDevice };  // one SM a configuration, .., the whole device (stream.cu, blocked.cu)
Route route_of(const Lattice& lat, const OccStream& occ, long long n, bool bits_only);
struct StreamJob : StreamQuery {
  int* error_out = nullptr;  // device int: 1 if the tick bound was hit (verdict first without a wait: two ints)
  const unsigned long long* n_dev = nullptr;  // device count of configurations (at most n_cfg; null: n_cfg)
  char* pool = nullptr;      // the caller's memory for the slots (else allocated)
  size_t pool_bytes = 0;
};
struct StreamPlan;
// Device resources for a set of queries (stream-ordered allocation on st).
pc_status stream_plan_create(const StreamQuery* qs, int nq, cudaStream_t st, StreamPlan** out,
                             char* pool = nullptr, size_t pool_bytes = 0,
                             const unsigned long long* n_dev = nullptr);
// Adds [init -> WHILE(sweep, control)] to g.
pc_status stream_plan_add(StreamPlan* P, cudaGraph_t g);
void stream_plan_release(StreamPlan* P, cudaStream_t st);
size_t stream_slot_bytes(int W, int L);
pc_status run_stream(const StreamJob& job, cudaStream_t st);
// The queries in one pool of slots that refill as configurations finish (job:
// the run's error flag, pool and count).
pc_status run_streams(const StreamQuery* qs, int nq, const StreamJob& job, cudaStream_t st);
// PC_VERDICT_FIRST on the streamed path: a verdict-only solve of every
// configuration, then the full solve of the percolating ones.  wait: the host
// waits for the first to count them, and takes slots for so many; else they are
// counted on the device, and the slots are those that the scratch pool keeps.
pc_status run_stream_verdict_first(const StreamJob& job, bool wait, cudaStream_t st);
// Verdict-only solver with temporal blocking (blocked.cu): runs a PC_BITS_ONLY
// job when a thread-block cluster holds the lattice's cross-section
// (*handled = true), else leaves it to the step-synchronous solver.
pc_status run_blocked(const StreamJob& job, cudaStream_t st, bool* handled);
// Whether run_blocked takes PC_BITS_ONLY jobs of this lattice on this device.
bool blocked_takes(const Lattice& lat);

// Largest density of a sample of caller occupancies (runs of at least 1,024
// sites), in 65,536ths: to the first of three zeroed words at, and to mail
// (occupancy.cu).
struct Mail;  // pool.cuh
pc_status launch_bits_density(const Lattice& lat, const uint32_t* occ_bits, int64_t words_per_cfg, int64_t n_cfg,
                              unsigned* at, const Mail& mail, cudaStream_t st);
// Standalone occupancy draw, occupancy.cu.
pc_status launch_occupancy(const Lattice& lat, const OccStream& os, uint32_t cfg0,
                           int64_t n_cfg, uint32_t* occ_bits, cudaStream_t st);
// Fixed-count occupancy (exactly n_metallic sites per configuration); waits
// for its own work on st (a convergence check).
pc_status launch_occupancy_fixed(const Lattice& lat, const OccStream& os, uint32_t cfg0, int64_t n_cfg,
                                 int64_t n_metallic, uint32_t* occ_bits, cudaStream_t st);

}  // namespace pc

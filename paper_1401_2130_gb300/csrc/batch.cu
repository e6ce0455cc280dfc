// batch.cu -- pc_batch_run (one GPU submission for many queries of mixed
// lattice sizes) and the autotuner of the forced resident solver's CTA size.
//
// A batch is the launches of run_wave: one for the levels and one for the
// masses of each group size its lattices take, each over the configurations of
// all its queries in decreasing lattice size.  Short, thin or dense lattices of
// resident size go to the resident solver, together, and wide dense ones to the
// device-wide solvers.  Nothing is kept between calls.
// (8 sizes x 400 configurations near the threshold: 1.2 ms; 42 ms as a CUDA
// graph of the full recursion, of which the W = 32 slots' ticks were most.)
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "pool.cuh"
#include "route.h"
#include "tune_file.h"
#include "wave.cuh"

namespace pc {

// ---------------------------------------------------------------------------
// Autotuner: per (W, L, p bin), the resident CTA size with the lowest
// measured time on a sample of configurations; kept in memory and in
// PC_TUNE_FILE.  p matters: below the threshold configurations stop after a
// few short steps, above it they sweep the whole fibre, and the best CTA
// size differs between the two regimes.
// ---------------------------------------------------------------------------
namespace {

constexpr double kTunePBins = 40.0;  // p bins of width 0.025

std::mutex g_tune_mu;
std::map<TuneKey, int> g_tune;
bool g_tune_loaded = false;

int p_bin(double p) { return (int)std::lround(p * kTunePBins); }

void tune_load() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const char* path = std::getenv("PC_TUNE_FILE");
  if (!path) return;
  FILE* f = std::fopen(path, "r");
  if (!f) return;
  tune_read(f, kResidentMaxThreads, g_tune);
  std::fclose(f);
}

void tune_save() {
  const char* path = std::getenv("PC_TUNE_FILE");
  if (!path) return;
  const std::string tmp = std::string(path) + ".tmp";
  FILE* f = std::fopen(tmp.c_str(), "w");
  if (!f) return;
  tune_write(f, g_tune);
  std::fclose(f);
  std::rename(tmp.c_str(), path);
}

}  // namespace

int tuned_threads(const Lattice& lat, double p, uint64_t seed, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  tune_load();
  const std::tuple<int, int, int> key{lat.W, lat.L, p_bin(p)};
  auto it = g_tune.find(key);
  if (it != g_tune.end()) return it->second;
  const int fallback = resident_threads(lat, 2048);
  const int64_t n = 2048;
  char* mem = nullptr;
  if (scratch_alloc((void**)&mem, 64 + n * 13, st) != cudaSuccess) return fallback;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  int best = fallback;
  float best_ms = 1e30f;
  const int cand[] = {128, 256, 384, 512, 640};
  for (int T : cand) {
    ResidentArgs a;
    a.lat = lat;
    a.occ.k0 = (uint32_t)(seed & 0xffffffffu); a.occ.k1 = (uint32_t)(seed >> 32);
    a.occ.cfg = 0; a.occ.wl = (uint32_t)lat.W | ((uint32_t)lat.L << 8); a.occ.T = threshold_of(p);
    a.occ_bits = nullptr; a.words_per_cfg = (lat.N + 31) / 32;
    a.n_cfg = n; a.cfg0 = 0x80000000u;  // a sample away from ordinary ranges
    a.verdict = (uint8_t*)(mem + 64); a.first_hit = (int32_t*)(mem + 64 + n);
    a.mass = (float*)(mem + 64 + 5 * n); a.m_stop = (int32_t*)(mem + 64 + 9 * n);
    a.n_perc = (unsigned long long*)(mem + 8); a.work = (unsigned long long*)mem;
    a.prep_chunk = 8;
    float ms = 0.f;
    bool ok = true;
    for (int rep = 0; rep < 2 && ok; ++rep) {
      cudaMemsetAsync(mem, 0, 64, st);
      cudaEventRecord(e0, st);
      ok = launch_resident(a, T, st) == PC_OK;
      cudaEventRecord(e1, st);
      if (ok) ok = cudaEventSynchronize(e1) == cudaSuccess;
      if (ok) cudaEventElapsedTime(&ms, e0, e1);
    }
    if (ok && ms < best_ms) { best_ms = ms; best = T; }
    cudaGetLastError();  // a candidate that does not fit is simply skipped
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFreeAsync(mem, st);
  cudaStreamSynchronize(st);
  g_tune[key] = best;
  tune_save();
  return best;
}

// ---------------------------------------------------------------------------
// Batches
// ---------------------------------------------------------------------------
namespace {

// The percolating counts of a batch to the queries' own device counters
// (pointers through kernel parameters: no copy per query).
constexpr int kCounts = 256;
struct CountChunk {
  int n;
  int64_t* to[kCounts];
};
__global__ void batch_counts_kernel(const unsigned long long* counts, const __grid_constant__ CountChunk c) {
  const int i = threadIdx.x;
  if (i < c.n && c.to[i]) *c.to[i] = (int64_t)counts[i];
}

// The size class of a query (pc_result.solver): 0 where its state fits one
// CTA's shared memory, 2 where a thread-block cluster holds the cross-section
// of a synchronous verdict-only query, else 1.
int size_class(const Lattice& lat, bool fits, int32_t flags) {
  if (fits) return 0;
  return (flags & PC_BITS_ONLY) && blocked_takes(lat) ? 2 : 1;
}

// Whether the queries, all of resident size, are the resident solver's: by the
// line for their configurations together, each query with the weight of its
// sites (so that they stay together: one launch, or a few, for all of them).
// W = 6, 10 and 12, L = W, 10 configurations each: p = 0.25 126 us on the
// resident solver, 158 on the wavefront solver.
// Never beside as many sites on the wavefront solver: its launch takes them along
// (W = 3, 23 and 32, L = 3 W and 4 W, p = 0.137, 34 configurations each 261 us, with
// W = 3 on the resident solver 314).
bool residents_are_faster(const std::vector<StreamQuery>& res, const std::vector<StreamQuery>& wave, int nsm) {
  long long n = 0;
  double sites = 0.0;
  for (const StreamQuery& s : res) {
    n += s.n_cfg;
    sites += (double)s.lat.N * (double)s.n_cfg;
  }
  for (const StreamQuery& s : wave) sites -= (double)s.lat.N * (double)s.n_cfg;
  if (sites <= 0.0) return false;
  double score = 0.0;
  for (const StreamQuery& s : res) {
    const double p = std::max((double)s.occ.T / 4294967296.0, 1e-3);
    const double over = std::log(p / resident_from(s.lat.W, s.lat.A, s.lat.L, n, nsm));
    score += (double)s.lat.N * (double)s.n_cfg * std::min(std::max(over, -1.0), 1.0);
  }
  return score > 0.0;
}

// The queries of the solvers that work on a configuration with the whole
// device: verdicts alone one after the other where a cluster holds the
// cross-section, the others in one pool of slots, larger lattices first (their
// steps overlap: W = 36 and 64, L = W, p = 0.9, 10 configurations each 2,590 us,
// one query after the other 3,618).
pc_status run_device(std::vector<StreamQuery>& qs, int* error, cudaStream_t st) {
  std::vector<StreamQuery> together;
  together.reserve(qs.size());
  int flags = 0;  // error flags used (one of each query at most)
  for (const StreamQuery& s : qs) {
    if (!s.bits_only || !blocked_takes(s.lat)) { together.push_back(s); continue; }
    StreamJob j;
    static_cast<StreamQuery&>(j) = s;
    j.error_out = error + 2 * flags++;
    const pc_status rc = run_stream(j, st);
    if (rc) return rc;
  }
  if (together.empty()) return PC_OK;
  std::stable_sort(together.begin(), together.end(),
                   [](const StreamQuery& x, const StreamQuery& y) { return x.lat.N > y.lat.N; });
  StreamJob j;
  j.error_out = error + 2 * flags;
  return run_streams(together.data(), (int)together.size(), j, st);
}

// A batch on its device scratch: counters in the first ctr_b bytes, then the
// staging of host outputs.
pc_status batch_run(const pc_query* q, int64_t nq, pc_result* out, int32_t flags, cudaStream_t st, char* mem, size_t ctr_b,
                    size_t bytes) {
  const bool dev_out = (flags & PC_OUT_DEVICE) != 0, async = (flags & PC_ASYNC) != 0;
  unsigned long long* counts = (unsigned long long*)mem;
  pc_status rc = PC_OK;
  std::vector<StreamQuery> sq, res, streamed;  // wavefront, resident (candidates at first), device-wide solvers
  std::vector<int64_t> sq_i, res_i;            // their places in q
  std::vector<Lattice> lats((size_t)nq);
  std::vector<int> threads((size_t)nq);
  std::vector<char> fits((size_t)nq);  // of resident size
  // (what the device says once: asked for each query it is a microsecond of each)
  int dev = 0, nsm = 1, optin = 0;
  PC_CUDA(cudaGetDevice(&dev));
  PC_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  PC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  do {
    cudaError_t e = cudaMemsetAsync(mem, 0, ctr_b, st);
    if (e != cudaSuccess) { rc = cuda_fail(e, "batch counters"); break; }
    char* stage = mem + ctr_b;
    for (int64_t i = 0; i < nq && rc == PC_OK; ++i) {
      const size_t n = (size_t)q[i].n_configs;
      if ((rc = get_lattice(q[i].W, q[i].L, &lats[(size_t)i]))) break;
      if (n == 0) continue;
      StreamQuery s;
      s.lat = lats[(size_t)i];
      s.occ.k0 = (uint32_t)(q[i].seed & 0xffffffffu); s.occ.k1 = (uint32_t)(q[i].seed >> 32);
      s.occ.cfg = 0; s.occ.wl = (uint32_t)q[i].W | ((uint32_t)q[i].L << 8); s.occ.T = threshold_of(q[i].p);
      s.occ_bits = nullptr; s.words_per_cfg = (s.lat.N + 31) / 32;
      s.n_cfg = q[i].n_configs; s.cfg0 = (uint32_t)q[i].config_begin;
      s.bits_only = (flags & PC_BITS_ONLY) ? 1 : 0;
      s.verdict_first = (flags & PC_VERDICT_FIRST) ? 1 : 0;
      s.out.n_perc = counts + i;
      if (dev_out) {
        s.out.verdict = q[i].verdicts; s.out.first_hit = q[i].first_hit;
        s.out.mass = q[i].mass; s.out.m_stop = q[i].m_stop;
      } else {
        s.out.first_hit = (int32_t*)stage; s.out.mass = (float*)(stage + 4 * n);
        s.out.m_stop = (int32_t*)(stage + 8 * n); s.out.verdict = (uint8_t*)(stage + 12 * n);
        stage += (n * 13 + 255) & ~(size_t)255;
      }
      fits[(size_t)i] = s.lat.A <= 32767 && resident_smem(s.lat) <= (size_t)optin;
      if (!s.bits_only && fits[(size_t)i]) { res.push_back(s); res_i.push_back(i); }
      else if (!fits[(size_t)i] && wave_is_slower(s.lat, q[i].p, s.n_cfg, s.bits_only != 0)) streamed.push_back(s);
      else { sq.push_back(s); sq_i.push_back(i); }
    }
    if (rc) break;
    if (!residents_are_faster(res, sq, nsm)) {
      sq.insert(sq.end(), res.begin(), res.end());
      sq_i.insert(sq_i.end(), res_i.begin(), res_i.end());
      res.clear();
      res_i.clear();
    }
    long long n_wave = 0;
    for (const StreamQuery& s : sq) n_wave += s.n_cfg;
    for (size_t k = 0; k < sq.size(); ++k) threads[(size_t)sq_i[k]] = wave_threads(sq[k], n_wave, nsm);
    if (!res.empty()) {
      std::vector<int> t(res.size());
      rc = run_residents(res.data(), (int)res.size(), counts + 2 * nq, t.data(), st);
      for (size_t k = 0; k < res.size(); ++k) threads[(size_t)res_i[k]] = t[k];
    }
    if (rc == PC_OK) rc = run_wave(sq.data(), (int)sq.size(), st);
    if (rc == PC_OK && !streamed.empty()) rc = run_device(streamed, (int*)(counts + nq), st);
    if (rc) break;
    if (dev_out)
      for (int64_t b = 0; b < nq && e == cudaSuccess; b += kCounts) {
        CountChunk c = {};
        c.n = (int)std::min<int64_t>(kCounts, nq - b);
        for (int i = 0; i < c.n; ++i) c.to[i] = q[b + i].n_percolating;
        batch_counts_kernel<<<1, kCounts, 0, st>>>(counts + b, c);
        e = cudaGetLastError();
      }
    if (e != cudaSuccess) { rc = cuda_fail(e, "batch counts"); break; }
    if (async) break;
    // one copy of the counts and, for host queries, of every output; where that
    // is more than the pinned buffer holds, of the counts, and each output to the
    // caller's own array
    HostStage pinned(dev_out ? (size_t)nq * 16 : bytes);
    std::vector<char> plain(pinned.data() ? 0 : (size_t)nq * 16);
    const char* host = pinned.data() ? pinned.data() : plain.data();
    e = cudaMemcpyAsync((void*)host, mem, pinned.data() && !dev_out ? bytes : (size_t)nq * 16, cudaMemcpyDeviceToHost, st);
    if (!pinned.data() && !dev_out) {
      const char* from = mem + ctr_b;
      for (int64_t i = 0; i < nq && e == cudaSuccess; ++i) {
        const size_t n = (size_t)q[i].n_configs;
        auto copy = [&](void* to, size_t off, size_t b) {
          if (to && b && e == cudaSuccess) e = cudaMemcpyAsync(to, from + off, b, cudaMemcpyDeviceToHost, st);
        };
        copy(q[i].first_hit, 0, 4 * n);
        copy(q[i].mass, 4 * n, 4 * n);
        copy(q[i].m_stop, 8 * n, 4 * n);
        copy(q[i].verdicts, 12 * n, n);
        from += (n * 13 + 255) & ~(size_t)255;
      }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { rc = cuda_fail(e, "batch outputs"); break; }
    const unsigned long long* cnt = (const unsigned long long*)host;
    int err = 0;
    for (int64_t i = 0; i < nq; ++i) err |= *(const int*)(cnt + nq + i);
    if (err & 2) { set_error("streamed solver: a bulk-copy wait timed out"); rc = PC_ERR_TIMEOUT; break; }
    if (err) { set_error("streamed solver: tick bound or segment check failed"); rc = PC_ERR_INTERNAL; break; }
    const char* at = host + ctr_b;
    for (int64_t i = 0; i < nq; ++i) {
      const size_t n = (size_t)q[i].n_configs;
      if (!dev_out) {
        if (n > 0 && pinned.data()) {
          if (q[i].first_hit) std::memcpy(q[i].first_hit, at, 4 * n);
          if (q[i].mass) std::memcpy(q[i].mass, at + 4 * n, 4 * n);
          if (q[i].m_stop) std::memcpy(q[i].m_stop, at + 8 * n, 4 * n);
          std::memcpy(q[i].verdicts, at + 12 * n, n);
          at += (n * 13 + 255) & ~(size_t)255;
        }
        if (q[i].n_percolating) *q[i].n_percolating = (int64_t)cnt[i];
      }
      if (out) {
        out[i].n_percolating = (int64_t)cnt[i];
        out[i].Pi = n ? (double)cnt[i] / (double)n : 0.0;
        out[i].solver = n ? size_class(lats[(size_t)i], fits[(size_t)i] != 0, flags) : 0;
        out[i].threads = out[i].solver == 0 && n ? threads[(size_t)i] : 0;
      }
    }
  } while (0);
  return rc;
}

}  // namespace

}  // namespace pc

using namespace pc;

extern "C" pc_status pc_batch_run(const pc_query* q, int64_t nq, pc_result* out, int32_t flags,
                                  void* cuda_stream) {
  NvtxRange nvtx_("pc_batch_run");
  if (nq < 0 || (nq > 0 && !q)) { set_error("pc_batch_run: bad query array"); return PC_ERR_ARG; }
  if (flags & ~(PC_OUT_DEVICE | PC_ASYNC | PC_BITS_ONLY | PC_VERDICT_FIRST)) { set_error("pc_batch_run: unknown flag bits"); return PC_ERR_ARG; }
  const bool dev_out = (flags & PC_OUT_DEVICE) != 0, async = (flags & PC_ASYNC) != 0;
  if (async && (!dev_out || out)) { set_error("PC_ASYNC needs PC_OUT_DEVICE and out == NULL"); return PC_ERR_ARG; }
  for (int64_t i = 0; i < nq; ++i) {
    const pc_query& x = q[i];
    if (x.W < 0 || x.W > 255 || x.L < 1 || x.L >= (1 << 24)) { set_error("pc_batch_run: bad W or L"); return PC_ERR_ARG; }
    if ((n_columns(x.W) + 1) * ((int64_t)x.L + 2) >= ((int64_t)1 << 31)) { set_error("pc_batch_run: lattice too large"); return PC_ERR_ARG; }
    if (!(x.p >= 0.0 && x.p <= 1.0)) { set_error("pc_batch_run: p must be in [0, 1]"); return PC_ERR_ARG; }
    if (x.n_configs < 0 || x.config_begin < 0 || x.config_begin + x.n_configs > ((int64_t)1 << 32)) {
      set_error("pc_batch_run: bad configuration range"); return PC_ERR_ARG;
    }
    if (x.n_configs > 0 && !x.verdicts) { set_error("pc_batch_run: verdicts must not be NULL"); return PC_ERR_ARG; }
  }
  if (nq == 0) return PC_OK;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // device scratch: a counter per query, the streamed solver's error flags, the
  // resident launches' counters, and the outputs of host queries
  const size_t ctr_b = ((size_t)nq * 16 + 24 + 255) & ~(size_t)255;
  size_t bytes = ctr_b;
  if (!dev_out)
    for (int64_t i = 0; i < nq; ++i) bytes += ((size_t)q[i].n_configs * 13 + 255) & ~(size_t)255;
  char* mem = nullptr;
  PC_CUDA(scratch_alloc((void**)&mem, bytes, st));
  pc_status rc = PC_OK;
  try {
    rc = batch_run(q, nq, out, flags, st, mem, ctr_b, bytes);
  } catch (const std::bad_alloc&) {
    set_error("pc_batch_run: no host memory");
    rc = PC_ERR_OOM;
  }
  const cudaError_t fe = cudaFreeAsync(mem, st);
  if (rc == PC_OK && fe != cudaSuccess) rc = cuda_fail(fe, "batch: free");
  return rc;
}

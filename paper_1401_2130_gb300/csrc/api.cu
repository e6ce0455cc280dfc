// api.cu -- the extern "C" entry points of libpercol (include/percol.h).
//
// Validates arguments, chooses the solver (route_of), allocates the call's
// stream-ordered scratch and marshals host or device outputs.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>

#include "common.cuh"
#include "kernels.cuh"
#include "pool.cuh"
#include "route.h"
#include "wave.cuh"

namespace pc {

namespace {
thread_local std::string g_err;
}

void set_error(const std::string& msg) { g_err = msg; }

pc_status cuda_fail(cudaError_t e, const char* what) {
  g_err = std::string(what) + ": " + cudaGetErrorString(e);
  return PC_ERR_CUDA;
}

namespace {

pc_status check_lattice(int32_t W, int32_t L) {
  if (W < 0 || W > 255) { set_error("W must be in [0, 255]"); return PC_ERR_ARG; }
  if (L < 1 || L >= (1 << 24)) { set_error("L must be in [1, 2^24)"); return PC_ERR_ARG; }
  // per-layer arrays of the solvers have (L + 2) rows of A + 1 entries,
  // indexed with 32-bit integers
  const int64_t rows = (n_columns(W) + 1) * ((int64_t)L + 2);
  if (rows >= (int64_t)1 << 31) { set_error("lattice too large: (A + 1)(L + 2) >= 2^31"); return PC_ERR_ARG; }
  return PC_OK;
}

pc_status check_range(int64_t config_begin, int64_t n_configs) {
  if (n_configs < 0 || config_begin < 0 || config_begin + n_configs > ((int64_t)1 << 32)) {
    set_error("configurations must satisfy 0 <= begin, n >= 0, begin + n <= 2^32");
    return PC_ERR_ARG;
  }
  return PC_OK;
}

}  // namespace

bool resident_fits(int W, int L) {
  int dev = 0, max_smem = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int64_t A = n_columns(W);
  if (A > 32767) return false;
  Lattice lat = {};
  lat.W = W; lat.L = L; lat.A = (int)A;
  layout_fill(W, &lat.P, &lat.s_begin, &lat.n_strips, nullptr, nullptr, nullptr, nullptr);
  return resident_smem(lat) <= (size_t)max_smem;
}

int resident_threads(const Lattice& lat, long long n) {
  int dev = 0, nsm = 1, sm_smem = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  return resident_cta(lat.A, lat.L, n, nsm, resident_smem(lat), (size_t)sm_smem);
}

ResidentArgs resident_args(const StreamQuery& q) {
  ResidentArgs a;
  a.lat = q.lat; a.occ = q.occ; a.occ_bits = q.occ_bits; a.words_per_cfg = q.words_per_cfg;
  a.n_cfg = q.n_cfg; a.cfg0 = q.cfg0;
  a.verdict = q.out.verdict; a.first_hit = q.out.first_hit; a.mass = q.out.mass; a.m_stop = q.out.m_stop;
  a.n_perc = q.out.n_perc; a.work = nullptr; a.prep_chunk = 8;
  a.bits_only = q.bits_only;
  a.verdict_first = q.verdict_first;
  a.gate = q.gate;
  return a;
}

pc_status run_resident(const StreamQuery& q, unsigned long long* work, cudaStream_t st) {
  ResidentArgs a = resident_args(q);
  a.work = work;
  return launch_resident(a, resident_threads(q.lat, q.n_cfg), st);
}

Route route_of(const Lattice& lat, const OccStream& occ, long long n, bool bits_only) {
  if (!resident_fits(lat.W, lat.L)) return wave_is_slower(lat, (double)occ.T / 4294967296.0, n, bits_only) ? Route::kDevice : Route::kWave;
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const double p = (double)occ.T / 4294967296.0;
  return !bits_only && p >= resident_from(lat.W, lat.A, lat.L, n, nsm) ? Route::kResident : Route::kWave;
}

namespace {

// Caller occupancies.  The host does not know how dense they are, and waiting
// for the answer would make an asynchronous call wait for its stream: a sample
// on the device opens the launches that are for its density and closes the
// others (each an empty launch, about 2 us).  Sparse: the wavefront solver,
// queues and tables sized for up to a quarter of the sites.  Denser: sized for
// all of them (near 0.2 that costs occupancy).  Denser still: the solver that
// route_of gives such a stream.  Verdicts first: masses in a pass of their own.
// us per call, all launches sized for a density of 0.2 and now: W = 8, L = 48,
// p = 0.7, 16 configurations 1,664 and 212; W = 64, L = 128, p = 0.95, verdicts
// of one 6,218 and 503.
// Beyond resident size what stands behind a closed gate is not cheap: planes of
// hundreds of MB to map, or a graph to build, 100 to 200 us of the host and 50 of
// the device.  There the host looks for the sample for 0.3 ms at most (in a call
// that waits for its stream anyway, until it comes) and leaves the rest out, or
// opens it, if it has come.
// ctr: counters of the call, zeroed; ctr[0] is the resident solver's, ctr[3] and
// ctr[4] are the sample's.
pc_status inspect_bits(StreamJob j, unsigned long long* ctr, bool waits, cudaStream_t st) {
  constexpr double kSparse = 0.25;
  // scratch of launches that may never run: within what the pool keeps
  constexpr size_t kUnsure = 768ull << 20;
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const Lattice& lat = j.lat;
  const bool res = resident_fits(lat.W, lat.L);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) cudaGetLastError();
  const bool captured = capture != cudaStreamCaptureStatusNone;
  double top = 2.0;  // density from which the resident, or the device-wide, solver takes over
  if (res) {
    if (!j.bits_only) top = resident_from(lat.W, lat.A, lat.L, j.n_cfg, nsm);
    if (top <= 0.15) return run_resident(j, ctr, st);
  } else {
    if (wave_is_slower(lat, 0.2, j.n_cfg, j.bits_only != 0))
      return !j.bits_only && j.verdict_first ? run_stream_verdict_first(j, false, st) : run_stream(j, st);
    // (a small lattice is done before the device-wide solvers' graph is built)
    if (lat.N >= 100000 && !captured)
      for (int d = 5; d <= 20 && top > 1.0; ++d)
        if (wave_is_slower(lat, 0.05 * d, j.n_cfg, j.bits_only != 0)) top = 0.05 * d;
  }
  // (what is sized for a quarter of few columns holds more; and where the
  // resident solver takes over soon, it takes all that is not sparse: two
  // launches fewer)
  const double sparse = lat.A <= 2200 ? 0.3 : kSparse;
  if (res && top <= 0.5) top = std::min(top, sparse);
  const double split = std::min(sparse, top);
  const Mail mail = !res && !captured ? take_mail() : Mail();
  pc_status rc = launch_bits_density(lat, j.occ_bits, j.words_per_cfg, j.n_cfg, (unsigned*)(ctr + 3), mail, st);
  if (rc) return rc;
  auto of = [](double d) { return d > 1.0 ? ~0u : (unsigned)(d * 65536.0); };
  auto between = [&](double lo, double hi, double density, double most) {
    j.gate.at = (const unsigned*)(ctr + 3);
    j.gate.lo = of(lo); j.gate.hi = of(hi);
    j.density = density; j.density_most = most;
  };
  between(0.0, split, 0.2, kSparse);
  if ((rc = run_wave(&j, 1, st))) return rc;
  unsigned g = 0;
  bool known = false;
  if (mail.at) {
    const auto until = std::chrono::steady_clock::now() + std::chrono::microseconds(300);
    while (!(known = mail.answer(&g)) && std::chrono::steady_clock::now() < until) {}
    if (!known && waits) {
      PC_CUDA(cudaStreamSynchronize(st));
      known = mail.answer(&g);
    }
  }
  if (known && g < of(split)) return PC_OK;
  if (top <= 1.0 && (!known || g >= of(top))) {
    between(top, 2.0, 0.6, 1.0);
    if (known) j.gate = Gate();
    rc = res ? run_resident(j, ctr, st) : run_stream(j, st);
    // no memory for it: the wavefront solver needs less
    if (rc != PC_ERR_OOM || res) {
      if (rc || known) return rc;
    } else {
      top = 2.0;
      rc = PC_OK;
    }
  }
  if (top > split) {
    between(split, top, 0.6, 1.0);
    if (known) j.gate = Gate();
    rc = run_wave(&j, 1, st, nullptr, known ? kWaveLimit : kUnsure);
  }
  return rc;
}

struct Scratch {
  unsigned long long* work = nullptr;
  unsigned long long* n_perc = nullptr;
  uint8_t* verdict = nullptr;
  int32_t* first_hit = nullptr;
  float* mass = nullptr;
  int32_t* m_stop = nullptr;
  char* base = nullptr;
};

// Shared implementation of pc_inspect / pc_inspect_occupancy.
pc_status inspect_impl(int32_t W, int32_t L, double p, uint64_t seed, int64_t cfg0,
                       const uint32_t* occ_bits, int64_t n, uint8_t* verdicts,
                       int32_t* first_hit, float* mass, int32_t* m_stop,
                       int64_t* n_percolating, double* Pi, int32_t flags, void* stream) {
  const bool dev_out = (flags & PC_OUT_DEVICE) != 0;
  if (flags & ~(PC_OUT_DEVICE | PC_MODE_RESIDENT | PC_MODE_STREAM | PC_BITS_ONLY | PC_VERDICT_FIRST)) {
    set_error("unknown flag bits"); return PC_ERR_ARG;
  }
  if (!verdicts && n > 0) { set_error("verdicts must not be NULL"); return PC_ERR_ARG; }
  if (dev_out && Pi) { set_error("Pi must be NULL with PC_OUT_DEVICE"); return PC_ERR_ARG; }
  if ((flags & PC_MODE_RESIDENT) && (flags & PC_MODE_STREAM)) { set_error("conflicting mode flags"); return PC_ERR_ARG; }
  cudaStream_t st = (cudaStream_t)stream;
  if (n == 0) {
    if (n_percolating) {
      if (dev_out) PC_CUDA(cudaMemsetAsync(n_percolating, 0, sizeof(int64_t), st));
      else *n_percolating = 0;
    }
    if (Pi) *Pi = 0.0;
    return PC_OK;
  }
  Lattice lat;
  pc_status rc = get_lattice(W, L, &lat);
  if (rc) return rc;

  // call scratch: counters (+ device copies of host outputs)
  size_t bytes = 64;  // work counter, percolating counter, streamed-solver error flag
  if (!dev_out) bytes += (size_t)n * (1 + 4 + 4 + 4) + 64;
  Scratch s;
  PC_CUDA(scratch_alloc((void**)&s.base, bytes, st));
  s.work = (unsigned long long*)s.base;
  s.n_perc = s.work + 1;
  if (dev_out) {
    s.verdict = verdicts; s.first_hit = first_hit; s.mass = mass; s.m_stop = m_stop;
    if (n_percolating) s.n_perc = (unsigned long long*)n_percolating;
  } else {
    char* q = s.base + 64;
    s.first_hit = (int32_t*)q; q += (size_t)n * 4;
    s.mass = (float*)q; q += (size_t)n * 4;
    s.m_stop = (int32_t*)q; q += (size_t)n * 4;
    s.verdict = (uint8_t*)q;
    if (!first_hit) s.first_hit = nullptr;
    if (!mass) s.mass = nullptr;
    if (!m_stop) s.m_stop = nullptr;
  }
  rc = PC_OK;
  do {
    if (cudaMemsetAsync(s.base, 0, 64, st) != cudaSuccess) { rc = cuda_fail(cudaGetLastError(), "memset"); break; }
    if (dev_out && n_percolating &&
        cudaMemsetAsync(n_percolating, 0, sizeof(int64_t), st) != cudaSuccess) {
      rc = cuda_fail(cudaGetLastError(), "memset"); break;
    }
    OccStream os;
    os.k0 = (uint32_t)(seed & 0xffffffffu);
    os.k1 = (uint32_t)(seed >> 32);
    os.cfg = 0;
    os.wl = (uint32_t)W | ((uint32_t)L << 8);
    os.T = occ_bits ? 0 : threshold_of(p);
    const int64_t wpc = (lat.N + 31) / 32;

    const bool first = (flags & PC_VERDICT_FIRST) != 0;
    StreamJob j;
    j.lat = lat; j.occ = os; j.occ_bits = occ_bits; j.words_per_cfg = wpc;
    j.n_cfg = n; j.cfg0 = (uint32_t)cfg0;
    j.out.verdict = s.verdict; j.out.first_hit = s.first_hit; j.out.mass = s.mass;
    j.out.m_stop = s.m_stop; j.out.n_perc = s.n_perc;
    j.bits_only = (flags & PC_BITS_ONLY) ? 1 : 0;
    j.verdict_first = first ? 1 : 0;
    j.error_out = (int*)(s.work + 2);
    if (flags & PC_MODE_RESIDENT) {
      if (!resident_fits(W, L)) {
        set_error("PC_MODE_RESIDENT: lattice state exceeds shared memory"); rc = PC_ERR_OOM; break;
      }
      ResidentArgs a;
      a.lat = lat; a.occ = os; a.occ_bits = occ_bits; a.words_per_cfg = wpc;
      a.n_cfg = n; a.cfg0 = (uint32_t)cfg0;
      a.verdict = s.verdict; a.first_hit = s.first_hit; a.mass = s.mass; a.m_stop = s.m_stop;
      a.n_perc = s.n_perc; a.work = s.work; a.prep_chunk = 8;
      a.bits_only = j.bits_only;
      a.verdict_first = first ? 1 : 0;
      rc = launch_resident(a, tuned_threads(lat, occ_bits ? 0.2 : p, seed, st), st);
    } else {
      const Route route = (flags & PC_MODE_STREAM) ? Route::kDevice : route_of(lat, os, n, j.bits_only != 0);
      if (occ_bits && !(flags & PC_MODE_STREAM)) rc = inspect_bits(j, s.work, !dev_out, st);
      else if (route == Route::kWave) rc = run_wave(&j, 1, st);
      else if (route == Route::kResident) rc = run_resident(j, s.work, st);
      else if (j.bits_only || !first) rc = run_stream(j, st);
      // (without PC_MODE_STREAM no call waits for its stream; where most
      // percolate, one pass is the faster way)
      else if (!(flags & PC_MODE_STREAM) && p >= fibre_threshold(W, L)) rc = run_stream(j, st);
      else rc = run_stream_verdict_first(j, (flags & PC_MODE_STREAM) != 0, st);
    }
    if (rc) break;
    if (!dev_out) {
      // counters, first hits, masses, step counts and verdicts lie in a row
      unsigned long long cnt = 0;
      int errs[2] = {0, 0};  // of the streamed solver, two passes with verdicts first
      const size_t all = 64 + (size_t)n * 13;
      HostStage stage(all);
      cudaError_t e = cudaSuccess;
      if (stage.data()) {
        e = cudaMemcpyAsync(stage.data(), s.base, all, cudaMemcpyDeviceToHost, st);
      } else {
        e = cudaMemcpyAsync(verdicts, s.verdict, (size_t)n, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && first_hit) e = cudaMemcpyAsync(first_hit, s.first_hit, (size_t)n * 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && mass) e = cudaMemcpyAsync(mass, s.mass, (size_t)n * 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && m_stop) e = cudaMemcpyAsync(m_stop, s.m_stop, (size_t)n * 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&cnt, s.n_perc, 8, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(errs, s.work + 2, sizeof(errs), cudaMemcpyDeviceToHost, st);
      }
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) { rc = cuda_fail(e, "copy outputs"); break; }
      if (const char* h = stage.data()) {
        std::memcpy(&cnt, h + 8, 8);
        std::memcpy(errs, h + 16, sizeof(errs));
        h += 64;
        if (first_hit) std::memcpy(first_hit, h, (size_t)n * 4);
        if (mass) std::memcpy(mass, h + (size_t)n * 4, (size_t)n * 4);
        if (m_stop) std::memcpy(m_stop, h + (size_t)n * 8, (size_t)n * 4);
        std::memcpy(verdicts, h + (size_t)n * 12, (size_t)n);
      }
      const int err = errs[0] | errs[1];
      if (err & 2) { set_error("streamed solver: a bulk-copy wait timed out"); rc = PC_ERR_TIMEOUT; break; }
      if (err) { set_error("streamed solver: tick bound or device check failed"); rc = PC_ERR_INTERNAL; break; }
      if (n_percolating) *n_percolating = (int64_t)cnt;
      if (Pi) *Pi = (double)cnt / (double)n;
    }
  } while (0);
  cudaError_t fe = cudaFreeAsync(s.base, st);
  if (rc == PC_OK && fe != cudaSuccess) rc = cuda_fail(fe, "free scratch");
  if (rc == PC_OK) {
    cudaError_t le = cudaGetLastError();
    if (le != cudaSuccess) rc = cuda_fail(le, "launch");
  }
  return rc;
}

}  // namespace
}  // namespace pc

using namespace pc;

extern "C" {

pc_status pc_lattice_info(int32_t W, int32_t L, int64_t* n_columns_out, int64_t* n_sites) {
  pc_status rc = check_lattice(W, L);
  if (rc) return rc;
  const int64_t A = n_columns(W);
  if (n_columns_out) *n_columns_out = A;
  if (n_sites) *n_sites = A * (int64_t)L;
  return PC_OK;
}

pc_status pc_occupancy(int32_t W, int32_t L, double p, uint64_t seed, int64_t config_begin,
                       int64_t n_configs, uint32_t* occ_bits, void* cuda_stream) {
  NvtxRange nvtx_("pc_occupancy");
  pc_status rc = check_lattice(W, L);
  if (rc) return rc;
  if (!(p >= 0.0 && p <= 1.0)) { set_error("p must be in [0, 1]"); return PC_ERR_ARG; }
  if ((rc = check_range(config_begin, n_configs))) return rc;
  if (n_configs == 0) return PC_OK;
  if (!occ_bits) { set_error("occ_bits must not be NULL"); return PC_ERR_ARG; }
  Lattice lat;
  if ((rc = get_lattice(W, L, &lat))) return rc;
  OccStream os;
  os.k0 = (uint32_t)(seed & 0xffffffffu);
  os.k1 = (uint32_t)(seed >> 32);
  os.cfg = 0;
  os.wl = (uint32_t)W | ((uint32_t)L << 8);
  os.T = threshold_of(p);
  return launch_occupancy(lat, os, (uint32_t)config_begin, n_configs, occ_bits,
                          (cudaStream_t)cuda_stream);
}

pc_status pc_occupancy_fixed(int32_t W, int32_t L, int64_t n_metallic, uint64_t seed,
                             int64_t config_begin, int64_t n_configs, uint32_t* occ_bits,
                             void* cuda_stream) {
  NvtxRange nvtx_("pc_occupancy_fixed");
  pc_status rc = check_lattice(W, L);
  if (rc) return rc;
  const int64_t N = n_columns(W) * (int64_t)L;
  if (n_metallic < 0 || n_metallic > N) { set_error("n_metallic must be in [0, N]"); return PC_ERR_ARG; }
  if ((rc = check_range(config_begin, n_configs))) return rc;
  if (n_configs == 0) return PC_OK;
  if (!occ_bits) { set_error("occ_bits must not be NULL"); return PC_ERR_ARG; }
  Lattice lat;
  if ((rc = get_lattice(W, L, &lat))) return rc;
  OccStream os;
  os.k0 = (uint32_t)(seed & 0xffffffffu);
  os.k1 = (uint32_t)(seed >> 32);
  os.cfg = 0;
  os.wl = (uint32_t)W | ((uint32_t)L << 8);
  os.T = 0;
  return launch_occupancy_fixed(lat, os, (uint32_t)config_begin, n_configs, n_metallic, occ_bits,
                                (cudaStream_t)cuda_stream);
}

pc_status pc_inspect(int32_t W, int32_t L, double p, uint64_t seed, int64_t config_begin,
                     int64_t n_configs, uint8_t* verdicts, int32_t* first_hit, float* mass,
                     int32_t* m_stop, int64_t* n_percolating, double* Pi, int32_t flags,
                     void* cuda_stream) {
  NvtxRange nvtx_("pc_inspect");
  pc_status rc = check_lattice(W, L);
  if (rc) return rc;
  if (!(p >= 0.0 && p <= 1.0)) { set_error("p must be in [0, 1]"); return PC_ERR_ARG; }
  if ((rc = check_range(config_begin, n_configs))) return rc;
  return inspect_impl(W, L, p, seed, config_begin, nullptr, n_configs, verdicts, first_hit,
                      mass, m_stop, n_percolating, Pi, flags, cuda_stream);
}

pc_status pc_inspect_occupancy(int32_t W, int32_t L, const uint32_t* occ_bits, int64_t n_configs,
                               uint8_t* verdicts, int32_t* first_hit, float* mass,
                               int32_t* m_stop, int64_t* n_percolating, double* Pi,
                               int32_t flags, void* cuda_stream) {
  NvtxRange nvtx_("pc_inspect_occupancy");
  pc_status rc = check_lattice(W, L);
  if (rc) return rc;
  if ((rc = check_range(0, n_configs))) return rc;
  if (n_configs > 0 && !occ_bits) { set_error("occ_bits must not be NULL"); return PC_ERR_ARG; }
  return inspect_impl(W, L, 0.0, 0, 0, occ_bits, n_configs, verdicts, first_hit, mass, m_stop,
                      n_percolating, Pi, flags, cuda_stream);
}

pc_status pc_shutdown(void) {
  release_pools();
  release_wave();
  release_lattices();
  release_static();
  return PC_OK;
}

const char* pc_last_error(void) { return g_err.c_str(); }

}  // extern "C"

// noalloc.cu -- pc_inspect_static: the inspection without any device-memory
// allocation.
//
// Some callers cannot allocate device memory at the point where they need an
// inspection: a process whose framework has reserved the whole device for
// its own pool allocator (a cudaMalloc there fails or fragments the pool),
// and latency-critical loops for which cudaMalloc / cudaFree are off limits
// because they can synchronise the whole device.  This entry point serves
// them: every piece of device scratch it needs -- the work and percolation
// counters, the lattice tables of the requested W, the wavefront solver's
// scratch and the device staging of the per-configuration outputs -- lives in
// one file-scope static device array, g_static_scratch, of kStaticBytes bytes.
// Every GPU that loads the library holds that array until the process exits.
//
// Solvers: the resident one, which needs no scratch, unless the wavefront
// solver is the faster one (route_of) and has room in the array for as many
// configurations at once as the device takes.  (Masses in device planes with a
// few dozen configurations in work: W = 16, L = 16, p = 0.95, 10,000
// configurations 93,700 us, on the resident solver 6,800.)
//
// Limits: the lattice must fit the resident (shared-memory) solver and have
// at most kStaticMaxColumns columns; at most kStaticMaxConfigs configurations
// per call.  Larger requests are rejected with PC_ERR_ARG before any work.
//
// Sharing: all calls on a device use the same array and it keeps the last
// call's contents.  The counters are cleared at the start of every call and
// the tables rewritten, but two calls whose work overlaps on the GPU (for
// example on two streams) race on the array and corrupt each other's
// results; callers must serialise them.
//
// Set-up: the first call on a device looks up the array's device address
// with cudaGetSymbolAddress while that device is current, and caches it.
// Make that first call before any stream capture begins.  A device reset
// (cudaDeviceReset) invalidates the cached address; pc_shutdown() forgets it
// (with every other cached device object), and the next call looks it up
// again.
//
// Limits in practice: the resident solver holds the whole configuration in
// one CTA's shared memory (227 KB on GB300), which bounds the lattice long
// before the tables do: W <= 26 (at L = 1), W = 20 up to L = 8, W = 8 up to
// L = 74.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "kernels.cuh"
#include "pool.cuh"
#include "wave.cuh"

namespace pc {

namespace {

constexpr int kStaticMaxColumns = 8192;       // W <= 51
constexpr int kStaticMaxW = 51;
constexpr int kStaticMaxP = 9216;             // plane entries of the widest allowed lattice
constexpr int kStaticMaxStrips = kStaticMaxP / 3 + 2;
constexpr int kStaticMaxRows = 2 * kStaticMaxW + 1;
constexpr int64_t kStaticMaxConfigs = 1 << 18;
constexpr size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t kPposBytes = up256(sizeof(int32_t) * (kStaticMaxColumns + 4));  // read in fours
constexpr size_t kRoffBytes = up256(sizeof(int32_t) * 4 * kStaticMaxRows);
constexpr size_t kSrowBytes = up256(sizeof(int16_t) * kStaticMaxStrips);
constexpr size_t kPcolBytes = up256(sizeof(int32_t) * kStaticMaxP);
constexpr size_t kNbrBytes = up256(sizeof(int32_t) * kStaticMaxColumns * kLateral);
constexpr size_t kSigBytes = up256(kStaticMaxColumns);
// scratch of the configurations in work (the solver takes as many as it holds;
// a resident-size lattice needs at most 232 KB for one)
constexpr size_t kWaveBytes = 4u << 20;
constexpr size_t kCtrBytes = 256;
constexpr size_t kOutBytes = up256((size_t)kStaticMaxConfigs * (1 + 4 + 4 + 4));
constexpr size_t kStaticBytes = kPposBytes + kRoffBytes + kSrowBytes + kPcolBytes + kNbrBytes + kSigBytes + kWaveBytes +
                                kCtrBytes + kOutBytes;

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
unsigned char* g_addr[kMaxDevices] = {};

// Address of g_static_scratch on the current device (set-up on first use).
pc_status static_scratch(unsigned char** out) {
  int dev = 0;
  PC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("pc_inspect_static: device ordinal out of range");
    return PC_ERR_ARG;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_static_scratch)");
    g_addr[dev] = (unsigned char*)p;
  }
  *out = g_addr[dev];
  return PC_OK;
}

// The rows of a layout, through kernel parameters (no host copy): first plane
// position, row offsets.
struct LayoutRows {
  int W, s_begin, n_strips;
  int16_t start[kStaticMaxRows];
  int16_t off[4 * kStaticMaxRows];
};

// Tables of the compact layout (the same content as the host-built cache):
// position of each column, row of each strip, row offsets; for the resident
// solver (pcol not null) also the column at each position and each column's
// sublattice and neighbours.  Zeroed counters.
__global__ void static_tables_kernel(const __grid_constant__ LayoutRows l, int A, int P, int32_t* ppos, int16_t* strip_row,
                                     int32_t* row_off, int32_t* pcol, int8_t* sigma, int32_t* nbr,
                                     unsigned long long* ctr) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, W = l.W, nr = 2 * W + 1;
  if (k < (int)(kCtrBytes / 8)) ctr[k] = 0ull;
  if (k < 4 * nr) row_off[k] = l.off[k];
  // columns before row i: rows W + 1, .., 2W + 1, .., W + 1 columns long
  auto before = [W](int i) {
    const int j = i <= W ? i : 2 * W + 1 - i, s = j * (W + 1) + j * (j - 1) / 2;
    return i <= W ? s : 3 * W * (W + 1) + 1 - s;
  };
  if (k < A) {
    int lo = 0, hi = nr - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (before(mid) <= k) lo = mid; else hi = mid - 1;
    }
    ppos[k] = l.start[lo] + (k - before(lo));
    if (pcol) {
      const int r = lo - W, q = (r < 0 ? -W - r : -W) + (k - before(lo));
      sigma[k] = (int8_t)(((q - r) % 3 + 3) % 3);
      for (int d = 0; d < kLateral; ++d) {
        const int qq = q + dir_dq(d), rr = r + dir_dr(d), qlo = rr < 0 ? -W - rr : -W, qhi = rr < 0 ? W : W - rr;
        nbr[k * kLateral + d] = rr >= -W && rr <= W && qq >= qlo && qq <= qhi ? before(rr + W) + (qq - qlo) : A;
      }
    }
  }
  if (pcol && k < P) {
    int lo = 0, hi = nr - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (l.start[mid] <= k) lo = mid; else hi = mid - 1;
    }
    const int j = k - l.start[lo];
    pcol[k] = j >= 0 && j < before(lo + 1) - before(lo) ? before(lo) + j : -1;
  }
  if (k < l.n_strips) {  // the row holding one of the strip's positions, else the row before it
    const int p2 = 3 * (l.s_begin + k) + 2;
    int lo = 0, hi = nr - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (l.start[mid] <= p2) lo = mid; else hi = mid - 1;
    }
    strip_row[k] = (int16_t)lo;
  }
}

}  // namespace

// Forget the cached device addresses of the static array (pc_shutdown).
void release_static() {
  std::lock_guard<std::mutex> lk(g_mu);
  for (int d = 0; d < kMaxDevices; ++d) g_addr[d] = nullptr;
}

}  // namespace pc

using namespace pc;

extern "C" pc_status pc_inspect_static(int32_t W, int32_t L, double p, uint64_t seed,
                                       int64_t config_begin, int64_t n_configs,
                                       uint8_t* verdicts, int32_t* first_hit, float* mass,
                                       int32_t* m_stop, int64_t* n_percolating, double* Pi,
                                       void* cuda_stream) {
  NvtxRange nvtx_("pc_inspect_static");
  if (W < 0 || W > 255 || L < 1 || L >= (1 << 24)) { set_error("pc_inspect_static: bad W or L"); return PC_ERR_ARG; }
  if (!(p >= 0.0 && p <= 1.0)) { set_error("pc_inspect_static: p must be in [0, 1]"); return PC_ERR_ARG; }
  if (n_configs < 0 || config_begin < 0 || config_begin + n_configs > ((int64_t)1 << 32)) {
    set_error("pc_inspect_static: bad configuration range"); return PC_ERR_ARG;
  }
  if (n_configs > kStaticMaxConfigs) {
    set_error("pc_inspect_static: at most 262144 configurations per call"); return PC_ERR_ARG;
  }
  const int64_t A64 = n_columns(W);
  if (A64 > kStaticMaxColumns) {
    set_error("pc_inspect_static: at most 8192 columns (W <= 51)"); return PC_ERR_ARG;
  }
  const int A = (int)A64;
  if (!resident_fits(W, L)) {
    set_error("pc_inspect_static: lattice state exceeds one CTA's shared memory"); return PC_ERR_ARG;
  }
  if (n_configs > 0 && !verdicts) { set_error("pc_inspect_static: verdicts must not be NULL"); return PC_ERR_ARG; }
  // the layout's sizes are checked against the static tables before any
  // work is enqueued
  int P = 0, s_begin = 0, n_strips = 0;
  layout_fill(W, &P, &s_begin, &n_strips, nullptr, nullptr, nullptr, nullptr);
  if (P > kStaticMaxP || n_strips > kStaticMaxStrips) {
    set_error("pc_inspect_static: layout exceeds the static tables"); return PC_ERR_ARG;
  }
  unsigned char* base = nullptr;
  pc_status rc = static_scratch(&base);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (n_configs == 0) {
    if (n_percolating) *n_percolating = 0;
    if (Pi) *Pi = 0.0;
    return PC_OK;
  }
  const size_t n = (size_t)n_configs;
  unsigned char* at = base;
  int32_t* d_ppos = (int32_t*)at; at += kPposBytes;
  int32_t* d_roff = (int32_t*)at; at += kRoffBytes;
  int16_t* d_srow = (int16_t*)at; at += kSrowBytes;
  int32_t* d_pcol = (int32_t*)at; at += kPcolBytes;
  int32_t* d_nbr = (int32_t*)at; at += kNbrBytes;
  int8_t* d_sig = (int8_t*)at; at += kSigBytes;
  char* d_wave = (char*)at; at += kWaveBytes;
  unsigned long long* ctr = (unsigned long long*)at;  // then the outputs, in a row
  unsigned char* o = at + kCtrBytes;
  StreamQuery q;
  q.out.n_perc = ctr;
  q.out.first_hit = (int32_t*)o; q.out.mass = (float*)(o + 4 * n);
  q.out.m_stop = (int32_t*)(o + 8 * n); q.out.verdict = o + 12 * n;
  LayoutRows rows;
  rows.W = W; rows.s_begin = s_begin; rows.n_strips = n_strips;
  {
    int32_t off[4 * kStaticMaxRows], pp[kStaticMaxColumns];
    layout_fill(W, nullptr, nullptr, nullptr, nullptr, off, pp, nullptr);
    for (int i = 0; i < 4 * (2 * W + 1); ++i) rows.off[i] = (int16_t)off[i];
    for (int i = 0, c = 0; i <= 2 * W; ++i) {
      rows.start[i] = (int16_t)pp[c];
      c += 2 * W + 1 - (i < W ? W - i : i - W);
    }
  }
  q.lat = Lattice{};
  q.lat.W = W; q.lat.L = L; q.lat.A = A; q.lat.N = (int64_t)A * L; q.lat.S = A + 1;
  q.lat.TW = (L + 31) / 32; q.lat.TWP = q.lat.TW + 2;
  q.lat.P = P; q.lat.s_begin = s_begin; q.lat.n_strips = n_strips;
  q.lat.strip_row = d_srow; q.lat.row_off = d_roff; q.lat.ppos = d_ppos; q.lat.pcol = d_pcol;
  q.lat.nbr = d_nbr; q.lat.sigma = d_sig;
  q.occ.k0 = (uint32_t)(seed & 0xffffffffu); q.occ.k1 = (uint32_t)(seed >> 32);
  q.occ.cfg = 0; q.occ.wl = (uint32_t)W | ((uint32_t)L << 8); q.occ.T = threshold_of(p);
  q.occ_bits = nullptr; q.words_per_cfg = (q.lat.N + 31) / 32;
  q.n_cfg = n_configs; q.cfg0 = (uint32_t)config_begin;
  WaveMemory m;
  m.ctr = ctr + 8; m.scratch = d_wave; m.bytes = kWaveBytes; m.max_groups = n_configs;
  bool wave = route_of(q.lat, q.occ, n_configs, false) == Route::kWave;
  if (wave) {  // groups of one warp where the array holds enough of them, else of a CTA
    m.warps = true;
    if (!wave_memory_suffices(q, m)) {
      m.warps = false;
      wave = wave_memory_suffices(q, m);
    }
  }
  static_tables_kernel<<<(std::max(A, P) + 127) / 128 + 4, 128, 0, st>>>(rows, A, P, d_ppos, d_srow, d_roff,
                                                                         wave ? nullptr : d_pcol, d_sig, d_nbr, ctr);
  PC_CUDA(cudaGetLastError());
  rc = wave ? run_wave(&q, 1, st, &m) : run_resident(q, ctr + 8, st);
  if (rc) return rc;

  const size_t all = kCtrBytes + 13 * n;
  HostStage stage(all);  // pinned host memory, kept after the first call
  unsigned long long cnt = 0;
  if (stage.data()) {
    PC_CUDA(cudaMemcpyAsync(stage.data(), ctr, all, cudaMemcpyDeviceToHost, st));
    PC_CUDA(cudaStreamSynchronize(st));
    const char* h = stage.data();
    std::memcpy(&cnt, h, 8);
    h += kCtrBytes;
    if (first_hit) std::memcpy(first_hit, h, 4 * n);
    if (mass) std::memcpy(mass, h + 4 * n, 4 * n);
    if (m_stop) std::memcpy(m_stop, h + 8 * n, 4 * n);
    std::memcpy(verdicts, h + 12 * n, n);
  } else {
    PC_CUDA(cudaMemcpyAsync(verdicts, q.out.verdict, n, cudaMemcpyDeviceToHost, st));
    if (first_hit) PC_CUDA(cudaMemcpyAsync(first_hit, q.out.first_hit, n * 4, cudaMemcpyDeviceToHost, st));
    if (mass) PC_CUDA(cudaMemcpyAsync(mass, q.out.mass, n * 4, cudaMemcpyDeviceToHost, st));
    if (m_stop) PC_CUDA(cudaMemcpyAsync(m_stop, q.out.m_stop, n * 4, cudaMemcpyDeviceToHost, st));
    PC_CUDA(cudaMemcpyAsync(&cnt, ctr, 8, cudaMemcpyDeviceToHost, st));
    PC_CUDA(cudaStreamSynchronize(st));
  }
  if (n_percolating) *n_percolating = (int64_t)cnt;
  if (Pi) *Pi = (double)cnt / (double)n_configs;
  return PC_OK;
}

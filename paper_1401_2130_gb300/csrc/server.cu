// server.cu -- pc_server_*: continuous-batching request loop.
//
// Queries (W, L, p, seed, configuration range) arrive at any time through
// pc_server_submit.  A worker thread admits them in arrival order as soon as
// their HBM footprint fits a device arena (first-fit allocator): output
// buffers, and for a lattice beyond one CTA's shared memory k slots of state
// (k <= free slots, bounded by what the arena holds).  An admitted query is
// one run of the wavefront solver on one of several side streams, its groups'
// scratch in its slots (k configurations in work at once; the device takes the
// next configuration without the host), so queries run beside each other.  A
// host callback behind each run wakes the worker, which copies the outputs out
// on a stream of their own, returns memory and slots, and admits more queries.
// Latency = completion time - submission time.
// Results equal pc_inspect's: the occupancy stream is counter based and the
// per-configuration solve does not depend on what runs beside it.
//
// The queries beyond shared memory used to share the streamed solver's slots,
// advanced in chunks of ticks with a status read between chunks: a burst of 8
// queries (W <= 32, L/W <= 16, 50 - 600 configurations) took 467 ms.
#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#include "arena.h"
#include "common.cuh"
#include "kernels.cuh"
#include "pool.cuh"
#include "wave.cuh"

namespace pc {
namespace {

using Clock = std::chrono::steady_clock;

// Run streams.  A query has one of its own while it runs, and admission waits
// for an idle one.  With the copies' stream they are fewer than the device's
// hardware queues by default (eight): further streams share a queue, and a run's
// later launches then wait behind another query's (a burst of 100 queries, W <=
// 32, L <= 12 W, 50 to 500 configurations: 20 ms with 6 or 7, 94 with 16, 208 with
// 32; 8 given out in turn whether idle or not 189).  50 bursts of 3 to 9 queries:
// 6 are 3 % faster than 7 or 8, and 6 % than 10.
constexpr int kStreams = 6;
// scratch of a query whose state fits shared memory: stream-ordered, and at most this
constexpr size_t kSmallScratch = 64ull << 20;

enum TicketState { T_PENDING, T_RUNNING, T_DONE, T_FAILED, T_CANCELLED };

struct Ticket {
  pc_query q;
  TicketState state = T_PENDING;
  pc_status status = PC_OK;
  Clock::time_point t_submit, t_done;
  pc_result result = {};
  // running state
  int kind = 0;                 // 0: fits shared memory, 1: state in arena slots
  int stream_idx = -1;          // its run stream
  size_t off_out = 0, bytes_out = 0, off_slots = 0, bytes_slots = 0;
  int nslots = 0;               // slots held until the query finishes
  cudaEvent_t ev = nullptr;
  unsigned long long* n_perc = nullptr;
  uint8_t* v = nullptr; int32_t* fh = nullptr; float* mass = nullptr; int32_t* ms = nullptr;
};

}  // namespace
}  // namespace pc

struct pc_server {
  pc_server_opts opts;
  int device = 0;
  cudaStream_t streams[pc::kStreams] = {};
  cudaStream_t copy = nullptr;     // outputs of finished queries
  bool busy[pc::kStreams] = {};    // (worker)
  char* arena_mem = nullptr;
  pc::Arena arena;
  int free_slots = 0;
  std::thread worker;
  std::mutex mu;
  std::condition_variable cv_work, cv_done;
  std::deque<uint64_t> pending;
  std::map<uint64_t, pc::Ticket> tickets;
  uint64_t next_ticket = 1;
  bool stop = false;
  bool woken = false;  // an arrival or the end of a run since the worker last looked
  // statistics
  std::vector<double> lat_ms;
  int64_t submitted = 0, completed = 0, configs_done = 0;
  pc::Clock::time_point t_first, t_last;
  bool any = false;
};

namespace pc {
namespace {

size_t out_bytes(int64_t n) { return 256 + (size_t)n * 13 + 256; }

// Host callback behind a query's run.
void CUDART_CB wake_worker(void* p) {
  pc_server* s = (pc_server*)p;
  std::lock_guard<std::mutex> lk(s->mu);
  s->woken = true;
  s->cv_work.notify_one();
}

// Enqueues an admitted query (worker thread; s->mu not held: the callback of a
// run that ends meanwhile takes it).
pc_status start_query(pc_server* s, Ticket& t) {
  const pc_query& q = t.q;
  Lattice lat;
  pc_status rc = get_lattice(q.W, q.L, &lat);
  if (rc) return rc;
  const int64_t n = q.n_configs;
  char* o = s->arena.base + t.off_out;
  t.n_perc = (unsigned long long*)o;
  char* d = o + 256;
  t.fh = (int32_t*)d; t.mass = (float*)(d + 4 * n); t.ms = (int32_t*)(d + 8 * n);
  t.v = (uint8_t*)(d + 12 * n);
  cudaStream_t st = s->streams[t.stream_idx];
  PC_CUDA(cudaMemsetAsync(o, 0, 256, st));
  StreamQuery sq;  // (counters in the first 256 bytes: percolating, the solvers' from 64 and, error flag, 128 on)
  sq.lat = lat;
  sq.occ.k0 = (uint32_t)(q.seed & 0xffffffffu); sq.occ.k1 = (uint32_t)(q.seed >> 32);
  sq.occ.cfg = 0; sq.occ.wl = (uint32_t)q.W | ((uint32_t)q.L << 8); sq.occ.T = threshold_of(q.p);
  sq.occ_bits = nullptr; sq.words_per_cfg = (lat.N + 31) / 32;
  sq.n_cfg = n; sq.cfg0 = (uint32_t)q.config_begin;
  sq.out.verdict = t.v; sq.out.first_hit = t.fh; sq.out.mass = t.mass; sq.out.m_stop = t.ms;
  sq.out.n_perc = t.n_perc;
  if (t.kind == 1 && wave_is_slower(lat, q.p, n, false)) {
    StreamJob j;
    static_cast<StreamQuery&>(j) = sq;
    j.error_out = (int*)(t.n_perc + 16);
    j.pool = s->arena.base + t.off_slots;
    j.pool_bytes = t.bytes_slots;
    rc = run_stream(j, st);
  } else if (t.kind == 0) {
    rc = route_of(lat, sq.occ, n, false) == Route::kResident ? PC_ERR_OOM : run_wave(&sq, 1, st, nullptr, kSmallScratch);
    if (rc == PC_ERR_OOM) rc = run_resident(sq, t.n_perc + 8, st);  // needs no scratch
  } else {
    WaveMemory m;
    m.ctr = t.n_perc + 8;
    m.scratch = s->arena.base + t.off_slots;
    m.bytes = t.bytes_slots;
    m.max_groups = t.nslots;
    rc = run_wave(&sq, 1, st, &m);
  }
  if (rc) return rc;
  PC_CUDA(cudaEventCreateWithFlags(&t.ev, cudaEventDisableTiming));
  PC_CUDA(cudaEventRecord(t.ev, st));
  PC_CUDA(cudaLaunchHostFunc(st, wake_worker, s));
  return PC_OK;
}

// Copy a finished query's outputs to the caller, release its resources.  On a
// stream of its own: the run stream may hold the next query's run by then.
void finish_query(pc_server* s, Ticket& t) {
  const int64_t n = t.q.n_configs;
  // one copy: the count, then first hits, masses, step counts, verdicts; large
  // outputs each to the caller's array
  const size_t all = 256 + 13 * (size_t)n;
  HostStage stage(all);
  char head[256] = {};
  const char* h = stage.data() ? stage.data() : head;
  const char* o = (const char*)t.n_perc;
  cudaError_t e = cudaMemcpyAsync((void*)h, o, stage.data() ? all : sizeof(head), cudaMemcpyDeviceToHost, s->copy);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->copy);
  unsigned long long cnt = 0;
  int err = 0;  // of the streamed solver
  if (e == cudaSuccess) {
    std::memcpy(&cnt, h, 8);
    std::memcpy(&err, h + 128, sizeof(int));
  }
  if (e == cudaSuccess && !err) {
    auto give = [&](void* to, size_t off, size_t b) {
      if (!to || e != cudaSuccess) return;
      if (stage.data()) std::memcpy(to, h + 256 + off, b);
      else e = cudaMemcpyAsync(to, o + 256 + off, b, cudaMemcpyDeviceToHost, s->copy);
    };
    give(t.q.first_hit, 0, 4 * (size_t)n);
    give(t.q.mass, 4 * (size_t)n, 4 * (size_t)n);
    give(t.q.m_stop, 8 * (size_t)n, 4 * (size_t)n);
    give(t.q.verdicts, 12 * (size_t)n, (size_t)n);
    if (e == cudaSuccess && !stage.data()) e = cudaStreamSynchronize(s->copy);
  }
  // (no CUDA call under s->mu, which the host callbacks take)
  if (t.ev) { cudaEventDestroy(t.ev); t.ev = nullptr; }
  std::lock_guard<std::mutex> lk(s->mu);
  if (e != cudaSuccess) {
    t.state = T_FAILED;
    t.status = cuda_fail(e, "server: copy outputs");
  } else if (err) {
    set_error("server: streamed solver: device bound reached");
    t.state = T_FAILED;
    t.status = (err & 2) ? PC_ERR_TIMEOUT : PC_ERR_INTERNAL;
  } else {
    t.state = T_DONE;
    t.result.n_percolating = (int64_t)cnt;
    t.result.Pi = n ? (double)cnt / (double)n : 0.0;
    t.result.solver = t.kind;
    t.result.threads = 0;
    if (t.q.n_percolating) *t.q.n_percolating = (int64_t)cnt;
  }
  t.t_done = Clock::now();
  const double ms = std::chrono::duration<double, std::milli>(t.t_done - t.t_submit).count();
  s->lat_ms.push_back(ms);
  s->completed += 1;
  s->configs_done += n;
  s->t_last = t.t_done;
  s->arena.release(t.off_out, t.bytes_out);
  if (t.bytes_slots) s->arena.release(t.off_slots, t.bytes_slots);
  s->free_slots += t.nslots;
  s->cv_done.notify_all();
}

void worker_main(pc_server* s) {
  cudaSetDevice(s->device);
  std::vector<uint64_t> running;
  for (;;) {
    // ---- admission (arrival order; stops at the first query that does not fit)
    std::vector<Ticket*> to_start;
    std::vector<uint64_t> started;
    {
      std::unique_lock<std::mutex> lk(s->mu);
      if (s->stop) break;
      s->woken = false;
      while (!s->pending.empty()) {
        const uint64_t id = s->pending.front();
        auto found = s->tickets.find(id);  // a cancelled ticket may already be polled away
        if (found == s->tickets.end() || found->second.state == T_CANCELLED) { s->pending.pop_front(); continue; }
        int idle = 0;
        while (idle < kStreams && s->busy[idle]) ++idle;
        if (idle == kStreams) break;
        Ticket& t = found->second;
        const pc_query& q = t.q;
        size_t off = 0;
        const size_t ob = out_bytes(q.n_configs);
        if (t.kind == 0) {
          if (!s->arena.alloc(ob, &off)) break;
          t.off_out = off; t.bytes_out = ob;
        } else {
          if (s->free_slots == 0) break;
          const size_t sb = stream_slot_bytes(q.W, q.L);
          if (!s->arena.alloc(ob, &off)) break;
          const size_t room = s->arena.largest();
          // not more than half of the free slots while other queries run or
          // wait: the next one in a burst would be left with a handful for
          // its whole run (burst of 8: 5.1 - 6.1 ms without this)
          const bool alone = running.empty() && to_start.empty() && s->pending.size() == 1;
          long long k = std::min<long long>(q.n_configs, alone ? s->free_slots : (s->free_slots + 1) / 2);
          k = std::min<long long>(k, std::max(1, s->opts.max_slots_per_query));
          k = std::min<long long>(k, (long long)(room / (sb + 256)));
          size_t soff = 0;
          if (k < 1 || !s->arena.alloc((size_t)k * sb, &soff)) { s->arena.release(off, ob); break; }
          t.off_out = off; t.bytes_out = ob;
          t.off_slots = soff; t.bytes_slots = (size_t)k * sb; t.nslots = (int)k;
          s->free_slots -= t.nslots;
        }
        t.stream_idx = idle;
        s->busy[idle] = true;
        t.state = T_RUNNING;
        s->pending.pop_front();
        to_start.push_back(&t);  // a running ticket stays in the map (and in place) until it is polled when done
        started.push_back(id);
      }
    }
    for (size_t i = 0; i < to_start.size(); ++i) {
      Ticket& t = *to_start[i];
      const pc_status rc = start_query(s, t);
      if (rc) {
        cudaStreamSynchronize(s->streams[t.stream_idx]);  // nothing of it runs on in memory given back
        if (t.ev) { cudaEventDestroy(t.ev); t.ev = nullptr; }
        s->busy[t.stream_idx] = false;
        std::lock_guard<std::mutex> lk(s->mu);
        t.state = T_FAILED; t.status = rc;
        s->arena.release(t.off_out, t.bytes_out);
        if (t.bytes_slots) s->arena.release(t.off_slots, t.bytes_slots);
        s->free_slots += t.nslots;
        s->cv_done.notify_all();
      } else {
        running.push_back(started[i]);
      }
    }
    // ---- completions (a failed run's event returns its error: finished too,
    // and the copy reports it)
    std::vector<uint64_t> still;
    for (uint64_t id : running) {
      Ticket* tp;
      {
        std::lock_guard<std::mutex> lk(s->mu);
        tp = &s->tickets[id];
      }
      if (cudaEventQuery(tp->ev) != cudaErrorNotReady) {
        s->busy[tp->stream_idx] = false;
        finish_query(s, *tp);
      } else {
        still.push_back(id);
      }
    }
    const bool freed = still.size() < running.size();
    running.swap(still);
    std::unique_lock<std::mutex> lk(s->mu);
    if (s->stop) break;
    if (!freed && !s->woken)  // an arrival or the end of a run wakes it
      s->cv_work.wait_for(lk, std::chrono::milliseconds(running.empty() ? 5 : 1));
  }
  for (auto r : s->streams) cudaStreamSynchronize(r);  // running work is drained
}

}  // namespace
}  // namespace pc

using namespace pc;

extern "C" {

pc_status pc_server_create(const pc_server_opts* opts, pc_server** out) {
  if (!out) { set_error("pc_server_create: out is NULL"); return PC_ERR_ARG; }
  *out = nullptr;
  pc_server_opts o;
  o.hbm_budget_bytes = 8ull << 30;
  o.max_slots = 256;
  o.max_slots_per_query = 64;
  o.ticks_per_poll = 8;
  o.max_pending = 1 << 16;
  o.max_W = 255;
  if (opts) o = *opts;
  if (o.max_W == 0) o.max_W = 255;
  if (o.hbm_budget_bytes < (1u << 20) || o.max_slots < 1 || o.max_slots > 4096 || o.ticks_per_poll < 1 ||
      o.max_pending < 1 || o.max_slots_per_query < 1 || o.max_W < 0 || o.max_W > 255) {
    set_error("pc_server_create: bad options"); return PC_ERR_ARG;
  }
  pc_server* s = new pc_server();
  s->opts = o;
  cudaGetDevice(&s->device);
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < kStreams && e == cudaSuccess; ++i) e = cudaStreamCreateWithFlags(&s->streams[i], cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s->copy, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaMalloc((void**)&s->arena_mem, o.hbm_budget_bytes);
  if (e != cudaSuccess) {
    pc_status rc = cuda_fail(e, "pc_server_create");
    if (s->arena_mem) cudaFree(s->arena_mem);
    for (auto r : s->streams) if (r) cudaStreamDestroy(r);
    if (s->copy) cudaStreamDestroy(s->copy);
    delete s;
    return rc == PC_ERR_CUDA && e == cudaErrorMemoryAllocation ? PC_ERR_OOM : rc;
  }
  s->arena.init(s->arena_mem, o.hbm_budget_bytes);
  s->free_slots = o.max_slots;
  s->worker = std::thread(worker_main, s);
  *out = s;
  return PC_OK;
}

pc_status pc_server_submit(pc_server* s, const pc_query* q, uint64_t* ticket) {
  if (!s || !q || !ticket) { set_error("pc_server_submit: NULL argument"); return PC_ERR_ARG; }
  if (q->W < 0 || q->W > 255 || q->L < 1 || q->L >= (1 << 24) ||
      (n_columns(q->W) + 1) * ((int64_t)q->L + 2) >= ((int64_t)1 << 31)) {
    set_error("pc_server_submit: bad W or L"); return PC_ERR_ARG;
  }
  if (!(q->p >= 0.0 && q->p <= 1.0) || q->n_configs < 1 || q->config_begin < 0 ||
      q->config_begin + q->n_configs > ((int64_t)1 << 32)) {
    set_error("pc_server_submit: bad p or configuration range"); return PC_ERR_ARG;
  }
  size_t need = out_bytes(q->n_configs);
  const bool small = resident_fits(q->W, q->L);
  if (!small) {
    if (q->W > s->opts.max_W) { set_error("pc_server_submit: lattice wider than the server's max_W"); return PC_ERR_ARG; }
    need += stream_slot_bytes(q->W, q->L) + 256;
  }
  if (need > s->opts.hbm_budget_bytes) {
    set_error("pc_server_submit: footprint exceeds the server's HBM budget"); return PC_ERR_OOM;
  }
  std::lock_guard<std::mutex> lk(s->mu);
  if (s->stop) { set_error("pc_server_submit: server is shutting down"); return PC_ERR_CANCELLED; }
  if ((int64_t)s->pending.size() >= s->opts.max_pending) { set_error("pc_server_submit: queue full"); return PC_ERR_BUSY; }
  const uint64_t id = s->next_ticket++;
  Ticket& t = s->tickets[id];
  t.q = *q;
  t.kind = small ? 0 : 1;
  t.t_submit = Clock::now();
  if (!s->any) { s->any = true; s->t_first = t.t_submit; }
  s->submitted += 1;
  s->pending.push_back(id);
  *ticket = id;
  s->woken = true;
  s->cv_work.notify_one();
  return PC_OK;
}

pc_status pc_server_poll(pc_server* s, uint64_t ticket, pc_result* out, int64_t timeout_ns) {
  if (!s) { set_error("pc_server_poll: NULL server"); return PC_ERR_ARG; }
  std::unique_lock<std::mutex> lk(s->mu);
  auto it = s->tickets.find(ticket);
  if (it == s->tickets.end()) { set_error("pc_server_poll: unknown ticket"); return PC_ERR_ARG; }
  auto ready = [&] {
    const TicketState st = s->tickets[ticket].state;
    return st == T_DONE || st == T_FAILED || st == T_CANCELLED;
  };
  if (!ready()) {
    if (timeout_ns > 0) s->cv_done.wait_for(lk, std::chrono::nanoseconds(timeout_ns), ready);
    if (!ready()) { set_error("pc_server_poll: not finished"); return PC_ERR_BUSY; }
  }
  Ticket& t = s->tickets[ticket];
  const pc_status st = t.state == T_DONE ? PC_OK : t.state == T_CANCELLED ? PC_ERR_CANCELLED : t.status;
  if (st == PC_ERR_CANCELLED) set_error("pc_server_poll: query cancelled");
  if (out && t.state == T_DONE) *out = t.result;
  s->tickets.erase(ticket);
  return st;
}

pc_status pc_server_cancel(pc_server* s, uint64_t ticket) {
  if (!s) { set_error("pc_server_cancel: NULL server"); return PC_ERR_ARG; }
  std::lock_guard<std::mutex> lk(s->mu);
  auto it = s->tickets.find(ticket);
  if (it == s->tickets.end()) { set_error("pc_server_cancel: unknown ticket"); return PC_ERR_ARG; }
  if (it->second.state != T_PENDING) { set_error("pc_server_cancel: query already running"); return PC_ERR_BUSY; }
  it->second.state = T_CANCELLED;
  s->cv_done.notify_all();
  return PC_OK;
}

pc_status pc_server_get_stats(pc_server* s, pc_server_stats* out) {
  if (!s || !out) { set_error("pc_server_get_stats: NULL argument"); return PC_ERR_ARG; }
  std::lock_guard<std::mutex> lk(s->mu);
  out->submitted = s->submitted;
  out->completed = s->completed;
  out->configs_completed = s->configs_done;
  std::vector<double> l = s->lat_ms;
  std::sort(l.begin(), l.end());
  auto pct = [&](double f) -> double {
    if (l.empty()) return 0.0;
    size_t i = (size_t)(f * (double)(l.size() - 1) + 0.5);
    return l[std::min(i, l.size() - 1)];
  };
  out->p50_ms = pct(0.50);
  out->p99_ms = pct(0.99);
  double sum = 0;
  for (double v : l) sum += v;
  out->mean_ms = l.empty() ? 0.0 : sum / (double)l.size();
  const double span = s->completed ? std::chrono::duration<double>(s->t_last - s->t_first).count() : 0.0;
  out->configs_per_s = span > 0 ? (double)s->configs_done / span : 0.0;
  return PC_OK;
}

pc_status pc_server_destroy(pc_server* s) {
  if (!s) return PC_OK;
  {
    std::lock_guard<std::mutex> lk(s->mu);
    s->stop = true;
    for (uint64_t id : s->pending) {
      auto& t = s->tickets[id];
      if (t.state == T_PENDING) t.state = T_CANCELLED;
    }
    s->pending.clear();
    s->cv_work.notify_all();
    s->cv_done.notify_all();
  }
  if (s->worker.joinable()) s->worker.join();
  cudaSetDevice(s->device);
  for (auto r : s->streams) cudaStreamSynchronize(r);
  for (auto& kv : s->tickets) if (kv.second.ev) cudaEventDestroy(kv.second.ev);
  cudaFree(s->arena_mem);
  for (auto r : s->streams) cudaStreamDestroy(r);
  cudaStreamDestroy(s->copy);
  delete s;
  return PC_OK;
}

}  // extern "C"

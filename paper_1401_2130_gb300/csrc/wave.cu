// wave.cu -- wavefront solver: every reached site is updated once, at the
// step at which mass first arrives there (Sec. II.B, Eqs. (2)-(4)).
//
// Why once is enough.  The outputs are the first step with non-zero detector
// probability, whether there is one, the step at which the reached set stops
// growing, and the detector probability at the first hit.  That probability is
// a sum over the walks that reach the detector in exactly first_hit moves; none
// is shorter, so after k moves each of them stands on a site at distance k
// from the start layer.  Of the vector nu_k only the entries of the sites whose
// distance is k ("level" k, the sites that enter the reached set at step k)
// ever reach the detector, and for such a site the sum over its 14 contacts is
// the sum over its contacts of level k - 1: contacts at distance k and k + 1
// hold nothing at step k - 1.  The terms and their additions are those of the
// full recursion with zeros in the other places, so that the sums are equal
// to it to the bit.  Once every entry of a level has underflowed to 0 all
// later ones are 0, as in the full FP32 recursion.
//
// wave_kernel, by its mode:
//   M_LEVELS, M_PRE  levels of every configuration (verdict, first_hit, m_stop;
//                    mass 0); M_PRE: over word rows drawn by a launch before.
//   M_HASH, M_PLANES levels with nu, until the end layer is reached or nu has
//                    vanished: of the percolating ones after a launch for the
//                    levels, or of all ("full", verdicts too).  nu of two levels
//                    lives in a hash table in shared memory or in planes in
//                    device scratch.
//
// A "group" (one warp, or one CTA) takes configurations from a counter.  It
// keeps
//   U      bits: metallic and not yet reached, word [w][pos] = tubes 32w ..
//          32w + 31 at plane position pos (layout in lattice.cu: contacts lie
//          at fixed offsets from the position, and positions outside the
//          hexagon are zero).  Word rows [wb, wb + NR) live in shared memory
//          (a ring), the others in device scratch, where the few sites whose
//          contacts lie outside the window are handled with global atomics.
//   queues the sites of the current and of the next level, each as the site it
//          was claimed from (position and hexagon row; tube) and the direction.
//          Sites beyond the queue's capacity are kept as bits of an overflow
//          map in device scratch, so that no level is too large.
// A level: each site of the current one claims its 14 contacts in U, one
// atomicAnd each without a look at the word first; whoever finds the bit still
// set appends the contact to the next level.  One barrier per level.  Occupancy
// is drawn a few layers ahead of the frontier from the same Philox stream as
// every other path.
//
// What bounds it: a level is a chain of dependent shared-memory accesses and
// integer instructions of one or a few warps (a warp issues one every 4.8
// cycles), and there are first_hit - 1 of them; HBM traffic is nil.  Against
// the full recursion, which updates every site of the window at every step
// (us per call): W = 8, L = 64, p = 0.185, 10^4 configurations 7,230 -> 498;
// W = 46, L = 400, p = 0.165, 32 configurations 258,000 -> 2,280; W = 64,
// L = 4096, p = 0.17, one configuration 1,250,000 -> 17,600.  Where it is not
// the faster one: route.h, wave_is_slower.
#include <algorithm>
#include <cstddef>
#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "pool.cuh"
#include "route.h"
#include "wave.cuh"

namespace pc {

namespace {

constexpr int kPosBits = 18;  // plane position of a frontier entry; its hexagon row above
constexpr uint32_t kPosMask = (1u << kPosBits) - 1u;
constexpr uint32_t kNone = 0xffffffffu;  // empty hash entry (no site packs to it)
constexpr int kDrawLayers = 8;  // layers drawn at a time (divides 32)

// Contact directions (order of common.cuh, then the end contacts): offset
// along the row, row offset index (0: r-2, 1: r-1, 2: r+1, 3: r+2, 4: own
// row), tube offset: fixed (end contacts), +1 from sublattice 2 (up), -1 from
// sublattice 0 (down).
__host__ __device__ constexpr int c_dq(int d) { return d < 12 ? dir_dq(d) : 0; }
__host__ __device__ constexpr int c_row(int d) {
  return d >= 12 ? 4 : dir_dr(d) == -2 ? 0 : dir_dr(d) == -1 ? 1 : dir_dr(d) == 0 ? 4 : dir_dr(d) == 1 ? 2 : 3;
}
__host__ __device__ constexpr int c_drow(int d) { return d < 12 ? dir_dr(d) : 0; }
__host__ __device__ constexpr int c_end(int d) { return d == 12 ? -1 : d == 13 ? 1 : 0; }
__host__ __device__ constexpr int c_up(int d) { return d >= 6 && d < 9; }
__host__ __device__ constexpr int c_dn(int d) { return d >= 9 && d < 12; }

// Direction d for the claims: c_ent is added to a frontier entry (hexagon row
// and offset along the row; the row offset comes on top); c_cls = byte of the
// row offset in a row's table | tube offset + 1 at sublattice s in bits
// 8 + 2s.
__host__ __device__ constexpr uint32_t c_ent(int d) { return (uint32_t)(c_drow(d) * (1 << kPosBits) + c_dq(d)); }
__host__ __device__ constexpr uint32_t c_cls(int d) {
  return (uint32_t)(4 * c_row(d)) | (uint32_t)(1 + c_end(d) - c_dn(d)) << 8 | (uint32_t)(1 + c_end(d)) << 10 |
         (uint32_t)(1 + c_end(d) + c_up(d)) << 12;
}

// What the claims of a level report (rare: tested by one comparison a site)
enum : unsigned { F_NEED = 1u, F_HIT = 2u, F_OUT = 4u };

// Scalars of a group, rotated over three levels: a level reads the previous
// one's, writes its own and clears the next one's.
struct GroupShared {
  unsigned cf[3][2];      // sites of the level, flags
  int olo[3], ohi[3];     // word rows of the level's overflow bits (ohi < 0: none)
  int span[2];            // tubes of a level (level_span)
  unsigned nz[2];
  long long item;
  uint2 dir[16];          // c_ent, c_cls of the 14 directions
};
constexpr int kSharedHead = 224;
static_assert(sizeof(GroupShared) <= kSharedHead && offsetof(GroupShared, dir) % 8 == 0, "group scalars");

template <bool kWarp>
__device__ __forceinline__ void group_sync() {
  if (kWarp) __syncwarp();
  else __syncthreads();
}

// ld.shared at a 32-bit shared address plus an immediate
template <int OFF>
__device__ __forceinline__ uint32_t lds_u(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
  return v;
}

// Shared-memory atomics at 32-bit shared addresses.
__device__ __forceinline__ uint32_t atoms_add(uint32_t a, uint32_t v) {
  uint32_t r;
  asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(r) : "r"(a), "r"(v) : "memory");
  return r;
}
template <int OFF>
__device__ __forceinline__ uint32_t atoms_and_at(uint32_t a, uint32_t m) {
  uint32_t r;
  asm volatile("atom.shared.and.b32 %0, [%1+%3], %2;" : "=r"(r) : "r"(a), "r"(m), "n"(OFF) : "memory");
  return r;
}
// the same under a condition: a predicated instruction, no branch
__device__ __forceinline__ void sts_u2_if(bool c, uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.v2.u32 [%1], {%2, %3};\n\t}"
               :: "r"((uint32_t)c), "r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts_u2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" :: "r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void reds_min(uint32_t a, int v) {
  asm volatile("red.shared.min.s32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void reds_max(uint32_t a, int v) {
  asm volatile("red.shared.max.s32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void reds_or(uint32_t a, uint32_t v) {
  asm volatile("red.shared.or.b32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
// or bit into the word at a if u <= last (predicated, no branch)
__device__ __forceinline__ void reds_or_le(uint32_t u, uint32_t last, uint32_t a, uint32_t bit) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %0, %1;\n\t@p red.shared.or.b32 [%2], %3;\n\t}"
               :: "r"(u), "r"(last), "r"(a), "r"(bit) : "memory");
}
__device__ __forceinline__ uint2 lds_u2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t smem_at(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Occupancy of layers [G, Gn) of configuration rel, by `size` threads: sets bit
// t & t_mask of the word of each metallic site's position, in shared memory at
// row_s (shared) or through set_site(t, position).
template <class F>
__device__ __forceinline__ void draw_layers(const WaveQuery& Q, long long rel, int G, int Gn, int tid, int size,
                                            bool shared, uint32_t row_s, int t_mask, F&& set_site) {
  const int A = Q.A;
  const int32_t* ppos = Q.ppos;
  const uint32_t i0 = (uint32_t)G * (uint32_t)A, i1 = (uint32_t)Gn * (uint32_t)A;
  const uint32_t divM = Q.divM;
  const int divS = 31 + Q.divS;
  if (Q.occ_bits) {
    const uint32_t* cb = Q.occ_bits + (size_t)rel * Q.words_per_cfg;
    for (uint32_t wi = (i0 >> 5) + tid; wi <= (i1 - 1) >> 5; wi += size) {
      uint32_t bits = cb[wi];
      while (bits) {
        const uint32_t i = (wi << 5) + __ffs(bits) - 1;
        bits &= bits - 1;
        if (i < i0 || i >= i1) continue;
        const int t = (int)(((uint64_t)i * divM) >> divS), c = (int)(i - (uint32_t)t * A);
        set_site(t, __ldg(ppos + c));
      }
    }
    return;
  }
  // a word u is metallic iff u < T, i.e. u <= T - 1
  const uint64_t T = Q.occ.T;
  if (T == 0) return;
  const uint32_t last = (uint32_t)(T - 1ull), k0 = Q.occ.k0, k1 = Q.occ.k1, wl = Q.occ.wl, cfg = Q.cfg0 + (uint32_t)rel;
  const uint32_t b_first = i0 >> 2, b_end = (i1 - 1) >> 2;
  uint32_t bi = b_first + tid;
  int t = (int)(((uint64_t)(bi << 2) * divM) >> divS), c = (int)((bi << 2) - (uint32_t)t * A);
  const int dt = (int)(((uint64_t)(4 * size) * divM) >> divS), dc = 4 * size - dt * A;  // one round further
  for (; bi <= b_end; bi += size) {
    // a block's four columns (the table is padded by four entries)
    const int q0 = __ldg(ppos + c), q1 = __ldg(ppos + c + 1), q2 = __ldg(ppos + c + 2), q3 = __ldg(ppos + c + 3);
    const u32x4 r = philox4x32_10(u32x4{bi, cfg, wl, 0u}, k0, k1);
    if (shared && c + 3 < A && bi != b_first && bi != b_end) {  // four sites of one layer to draw
      const uint32_t bit = 1u << (t & t_mask);
      reds_or_le(r.x, last, row_s + 4u * (uint32_t)q0, bit);
      reds_or_le(r.y, last, row_s + 4u * (uint32_t)q1, bit);
      reds_or_le(r.z, last, row_s + 4u * (uint32_t)q2, bit);
      reds_or_le(r.w, last, row_s + 4u * (uint32_t)q3, bit);
    } else {  // the chunk's ends, two layers in a block, or no window
      const uint32_t u[4] = {r.x, r.y, r.z, r.w};
      int t1 = t, c1 = c;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (u[j] <= last && t1 >= G && t1 < Gn) set_site(t1, __ldg(ppos + c1));
        if (++c1 == A) { c1 = 0; ++t1; }
      }
    }
    t += dt;
    c += dc;
    if (c >= A) { c -= A; ++t; }
  }
}

// kMode: levels only, or levels with nu -- in shared memory (a hash table of
// the level's sites) or in planes in device scratch
// M_PRE: levels, of configurations whose word rows were drawn by a launch
// before (see run_wave)
enum : int { M_LEVELS = 0, M_HASH = 1, M_PLANES = 2, M_PRE = 3 };

template <bool kWarp, bool kPart, int kMode>
__device__ __forceinline__ void wave_body(const WaveArgs& a, unsigned char* sm, char* scratch) {
  constexpr bool kMass = kMode == M_HASH || kMode == M_PLANES;
  constexpr bool kPre = kMode == M_PRE;
  const int tid = kWarp ? (threadIdx.x & 31) : threadIdx.x;
  const int size = kWarp ? 32 : blockDim.x;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  GroupShared* gs = reinterpret_cast<GroupShared*>(sm);
  int* roff = reinterpret_cast<int*>(sm + kSharedHead);  // [row][8]: offsets to rows r-2, r-1, r+1, r+2, then 0
  const uint32_t gs_s = smem_at(gs), roff_s = smem_at(roff);
  int cur_q = -1;
#pragma unroll
  for (int d = 0; d < 14; ++d)
    if (tid == d) gs->dir[d] = make_uint2(c_ent(d), c_cls(d));
  if (tid == 14 || tid == 15) gs->dir[tid] = make_uint2(0u, 16u | 0x1500u);
  const uint32_t dir_s = gs_s + (uint32_t)offsetof(GroupShared, dir);
  // this lane's contact when sixteen lanes share a site (lanes 14 and 15 idle)
  const bool has16 = (lane & 15) < 14;
  const uint32_t e16 = has16 ? c_ent(lane & 15) : 0u, y16 = has16 ? c_cls(lane & 15) : 16u | 0x1500u;

  if (kMass && !(a.full && !a.hard)) {  // nothing to do here?
    const unsigned long long n = a.count[a.hard ? 1 : 0];
    if (n < a.min_count || n > a.max_count) return;
  }
  for (bool once = false;; once = true) {
    long long item;
    if (kPre) {  // a CTA per configuration, with its own scratch
      if (once) break;
      item = blockIdx.x;
    } else {
      unsigned long long v = 0;
      if (tid == 0) v = atomicAdd(a.work, 1ull);
      if (kWarp) {
        item = (long long)__shfl_sync(0xffffffffu, v, 0);
      } else {
        if (tid == 0) gs->item = (long long)v;
        __syncthreads();
        item = gs->item;
      }
    }
    if (item >= a.n_items) break;
    int qi = 0;
    if (a.nq > 1) {  // items come in order: mostly the previous one's query
      if (cur_q >= 0 && item >= a.qs[cur_q].item0 && item < a.qs[cur_q].item0 + a.qs[cur_q].n_cfg) {
        qi = cur_q;
      } else {
        int hi = a.nq - 1;
        while (qi < hi) {
          const int mid = (qi + hi + 1) >> 1;
          if (a.qs[mid].item0 <= item) qi = mid; else hi = mid - 1;
        }
      }
    }
    const WaveQuery& Q = a.nq > 1 ? a.qs[qi] : a.q0;
    const int L = Q.L, A = Q.A, P = Q.P, NR = Q.NR, cap = Q.cap, sb = Q.s_begin, nr_mask = Q.nr_mask;
    const int32_t* ppos = Q.ppos;
    const int16_t* strip_row = Q.strip_row;
    uint32_t* win = reinterpret_cast<uint32_t*>(sm + Q.o_win);
    uint2* queue = reinterpret_cast<uint2*>(sm + Q.o_queue);
    const uint32_t win_s = smem_at(win), queue_s = smem_at(queue);
    uint32_t* back = reinterpret_cast<uint32_t*>(scratch + Q.a_back);
    uint32_t* over = reinterpret_cast<uint32_t*>(scratch + Q.a_over);  // two maps of TW rows
    const size_t over_n = (size_t)Q.TW * P;
    uint32_t* occ = Q.o_occ >= 0 ? reinterpret_cast<uint32_t*>(sm + Q.o_occ) : reinterpret_cast<uint32_t*>(scratch + Q.a_occ);
    float* nu = reinterpret_cast<float*>(scratch + Q.a_nu);            // two rings of planes
    // hash tables (key, entry) of two levels, then nu of the entries of two levels
    const uint32_t tab_s = smem_at(sm + Q.o_tab), nuq_s = tab_s + 16u * (1u << Q.tab_bits);
    const int tab_bits = Q.tab_bits;
    const uint32_t tab_mask = (1u << tab_bits) - 1u;
    const int ring_mask = Q.ring_mask;
    const size_t nu_n = (size_t)(ring_mask < 0 ? L : ring_mask + 1) * P;
    const long long rel = item - Q.item0;
    if (kMass && (a.hard || !a.full)) {  // percolating, or marked, configurations only (group-uniform)
      const bool skip = !Q.want_mass || (a.hard ? !(Q.out.mass[rel] < 0.f) : !Q.out.verdict[rel]);
      group_sync<kWarp>();  // every thread has read the item
      if (skip) continue;
    }
    if (qi != cur_q) {
      cur_q = qi;
      for (int k = tid; k < 8 * (2 * Q.W + 1); k += size) roff[k] = (k & 7) < 4 ? Q.row_off[(k >> 3) * 4 + (k & 7)] : 0;
    }
    if (tid == 0) {
      gs->nz[0] = 0u;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        gs->cf[k][0] = 0u; gs->cf[k][1] = 0u; gs->olo[k] = 0x7fffffff; gs->ohi[k] = -1;
      }
    }
    if (kMode == M_HASH)
      for (uint32_t k = tid; k < 2u * (tab_mask + 1u); k += size) sts_u2(tab_s + 8u * k, kNone, 0u);
    group_sync<kWarp>();

    int G = 0;   // layers drawn
    int wb = 0;  // lowest word row of the window; row w has slot w & nr_mask
    auto resident = [&](int w) { return !kPart || (unsigned)(w - wb) < (unsigned)NR; };
    auto word_ptr = [&](int w, int pos) -> uint32_t* {  // any row
      return resident(w) ? win + (w & nr_mask) * P + pos : back + (size_t)w * P + pos;
    };
    auto plane = [&](int t) -> size_t { return (size_t)(t & ring_mask) * P; };
    // A frontier entry: the site it was claimed from (position, hexagon row;
    // tube << 4) and the direction, 15 for that site itself.  Its own position,
    // row and tube:
    auto decode = [&](uint2 e, uint32_t& ent, int& t) {
      const uint2 y = lds_u2(dir_s + 8u * (e.y & 15u));
      const int pos = (int)(e.x & kPosMask), sg = pos - 3 * (int)__umulhi((unsigned)pos, 0x55555556u);
      ent = e.x + y.x + lds_u<0>(roff_s + ((e.x >> (kPosBits - 5)) & ~31u) + (y.y & 255u));
      t = (int)(e.y >> 4) + (int)((y.y >> (8 + 2 * sg)) & 3u) - 1;
    };
    auto row_of = [&](int pos) -> int { return strip_row[(int)__umulhi((unsigned)pos, 0x55555556u) - sb]; };
    // Slide the window by one row: the row that leaves is written back if it
    // was drawn, the row that enters (the same slot) read if it was.
    // Group-uniform.
    auto slide = [&](int dir) {
      const int out = dir > 0 ? wb : wb + NR - 1, in = dir > 0 ? wb + NR : wb - 1;
      uint32_t* row = win + (out & nr_mask) * P;
      const bool w_out = 32 * out < G, r_in = 32 * in < G;
      for (int k = tid; k < P; k += size) {
        if (w_out) back[(size_t)out * P + k] = row[k];
        if (r_in) row[k] = back[(size_t)in * P + k];
      }
      wb += dir;
      group_sync<kWarp>();
    };
    // Draw the next layers (within one word row).  Group-uniform.
    auto draw = [&]() {
      if (kPre) {  // the next row was drawn into the scratch
        const int w = G >> 5;
        if (kPart && NR > 0) {
          while (w >= wb + NR) slide(1);
          while (w < wb) slide(-1);
        }
        if (!kPart || NR > 0)
          for (int k = tid; k < P; k += size) win[(w & nr_mask) * P + k] = back[(size_t)w * P + k];
        G = min(32 * (w + 1), L);
        group_sync<kWarp>();
        return;
      }
      const int Gn = min(G + kDrawLayers, L), w = G >> 5;
      if (kPart && NR > 0) {
        while (w >= wb + NR) slide(1);
        while (w < wb) slide(-1);
      }
      uint32_t* row = !kPart || NR > 0 ? win + (w & nr_mask) * P : back + (size_t)w * P;
      const uint32_t row_s = win_s + 4u * (uint32_t)((!kPart || NR > 0 ? w & nr_mask : 0) * P);
      uint32_t* row_g = back + (size_t)w * P;
      if ((G & 31) == 0) {  // first layers of the row
        for (int k = tid; k < P; k += size) {
          row[k] = 0u;
          if (kMode != M_HASH) {
            over[(size_t)w * P + k] = 0u;
            over[over_n + (size_t)w * P + k] = 0u;
          }
        }
        group_sync<kWarp>();
      }
      draw_layers(Q, rel, G, Gn, tid, size, !kPart || NR > 0, row_s, 31, [&](int t, int pos) {
        if (!kPart || NR > 0) reds_or(row_s + 4u * (uint32_t)pos, 1u << (t & 31));
        else atomicOr(row_g + pos, 1u << (t & 31));
      });
      group_sync<kWarp>();
      if (kMass) {  // the degrees need the occupancy itself
        const int nl = Gn - G;
        const uint32_t mask = (nl == 32 ? 0xffffffffu : (1u << nl) - 1u) << (G & 31);
        for (int k = tid; k < P; k += size) {
          uint32_t* o = occ + (size_t)w * P + k;
          *o = ((G & 31) ? *o : 0u) | (row[k] & mask);
        }
        group_sync<kWarp>();
      }
      G = Gn;
    };

    // Hash table of a level: the site's key -> its queue entry.  Levels hold
    // tubes less than 2^14 apart (longer fibres keep nu in planes).
    auto key_of = [&](uint32_t pos, int t) -> uint32_t { return pos | (uint32_t)t << kPosBits; };
    auto hash_add = [&](int level, uint32_t key, uint32_t entry) {
      uint32_t h = (key * 0x9E3779B1u) >> (32 - tab_bits);
      const uint32_t base = tab_s + 8u * (uint32_t)((level & 1) << tab_bits);
      for (;;) {
        uint32_t old;
        asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(old) : "r"(base + 8u * h), "r"(kNone), "r"(key) : "memory");
        if (old == kNone) break;
        h = (h + 1u) & tab_mask;
      }
      asm volatile("st.shared.u32 [%0], %1;" :: "r"(base + 8u * h + 4u), "r"(entry) : "memory");
    };
    // nu of a site if it belongs to the level, else 0
    auto hash_nu = [&](int level, uint32_t key) -> float {
      uint32_t h = (key * 0x9E3779B1u) >> (32 - tab_bits);
      const uint32_t base = tab_s + 8u * (uint32_t)((level & 1) << tab_bits);
      for (;;) {
        const uint2 e = lds_u2(base + 8u * h);
        if (e.x == key) return __uint_as_float(lds_u<0>(nuq_s + 4u * (uint32_t)((level & 1) * cap) + 4u * e.y));
        if (e.x == kNone) return 0.f;
        h = (h + 1u) & tab_mask;
      }
    };

    WaveState* const state = kPre ? a.state + item : nullptr;
    const int phase = kPre ? state->phase : 0;
    unsigned total = 0, n_start = 0;
    int m0 = 0;  // the level the queue holds
    if (kPre && phase == 2) continue;  // done
    if (kPre && phase == 1) {          // resume
      m0 = state->m; total = state->total; wb = state->wb; G = state->G; n_start = state->n0;
      if (tid == 0) { gs->olo[0] = state->olo; gs->ohi[0] = state->ohi; }
      const uint2* saved = reinterpret_cast<const uint2*>(scratch + Q.a_nu);
      for (unsigned k = tid; k < min(total, (unsigned)cap); k += size) queue[(m0 & 1) * cap + k] = saved[k];
      for (int w = wb; w < wb + NR && 32 * w < G; ++w)
        for (int k = tid; k < P; k += size) win[(w & nr_mask) * P + k] = back[(size_t)w * P + k];
      group_sync<kWarp>();
      draw();  // the rows it waited for
    } else {
    draw();
    // level 0: the metallic sites of t = 0
    {
      uint32_t* row = !kPart || NR > 0 ? win : back;
      for (int k0 = tid & ~31; k0 < P; k0 += size) {
        const int pos = k0 + lane;
        bool c = false;
        if (pos < P) {
          const uint32_t w = row[pos];
          c = w & 1u;
          if (c) row[pos] = w & ~1u;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, c);
        if (bal) {
          unsigned base = 0;
          if (kWarp) {
            base = total;
            total += __popc(bal);
          } else {
            if (lane == 0) base = atoms_add(gs_s + (uint32_t)offsetof(GroupShared, cf), (unsigned)__popc(bal));
            base = __shfl_sync(0xffffffffu, base, 0);
          }
          base += __popc(bal & lt);
          if (c) {
            if (base < (unsigned)cap) {
              queue[base] = make_uint2((uint32_t)pos | (uint32_t)row_of(pos) << kPosBits, 15u);
            } else if (kMode != M_HASH) {
              atomicOr(over + pos, 1u);
              gs->olo[0] = 0;
              gs->ohi[0] = 0;
            }
          }
        }
      }
      group_sync<kWarp>();
      if (!kWarp) total = gs->cf[0][0];
    }
    n_start = total;
    }
    const unsigned n0 = n_start;

    // nu of a new site: (1/degree) x the sum over the contacts of the previous
    // level, whose values value_of gives (0 for other contacts); at level 0:
    // (1/degree) x 1/n0
    auto site_value = [&](int t, int pos, int hrow, bool later, auto&& value_of) -> float {
      const int sg = pos - 3 * (int)__umulhi((unsigned)pos, 0x55555556u);
      const int4 o4 = reinterpret_cast<const int4*>(roff)[2 * hrow];
      const int ro[5] = {o4.x, o4.y, o4.z, o4.w, 0};
      float v[14];
      int deg = t == L - 1;  // the detector edge
      uint32_t ow[14];
#pragma unroll
      for (int d = 0; d < 14; ++d) {
        const int tt = t + c_end(d) + (c_up(d) & (sg == 2)) - (c_dn(d) & (sg == 0));
        const int np = pos + c_dq(d) + ro[c_row(d)];
        ow[d] = (unsigned)tt < (unsigned)L ? occ[(size_t)(tt >> 5) * P + np] >> (tt & 31) : 0u;
      }
#pragma unroll
      for (int d = 0; d < 14; ++d) {
        v[d] = 0.f;
        if (ow[d] & 1u) {
          ++deg;
          if (later) v[d] = value_of(t + c_end(d) + (c_up(d) & (sg == 2)) - (c_dn(d) & (sg == 0)), pos + c_dq(d) + ro[c_row(d)]);
        }
      }
      const float inv = deg ? __frcp_rn((float)deg) : 0.f;
      if (!later) return inv * __frcp_rn((float)n0);
      // the addition trees of the full recursion (strip_sums in tiling.cuh)
      const float e = v[6] + v[9], h = v[12] + v[13], g = v[5] + v[2];
      const float pa = v[7] + v[0], pbs = v[8] + v[1], pcs = v[4] + v[11], pd = v[3] + v[10];
      float r;
      if (sg == 0) r = (((pa + pbs) + pcs) + (pd + e)) + (h + g);
      else if (sg == 1) r = ((pcs + pd) + (pa + pbs)) + ((e + h) + g);
      else r = (((pcs + pd) + pa) + (pbs + e)) + (h + g);
      return inv * r;
    };
    // M_HASH: nu of the sites of level m, sixteen lanes to a site, one contact
    // each; true if any is not 0.  The contact values of the previous level
    // come from its table (others are not in it: 0), the additions are those of
    // site_value, between lanes.
    auto level_hash = [&](int m, unsigned n) -> bool {
      const uint32_t q_s = queue_s + 8u * (uint32_t)((m & 1) * cap);
      const int half = lane & 16;
      // the lane whose value the first addition takes: the pairs (0,7) (1,8)
      // (2,5) (3,10) (4,11) (6,9) (12,13), four bits a lane
      const int mate = half | (int)((0xFECD4361092BA587ull >> (4 * (lane & 15))) & 15u);
      bool nz = false;
      // many sites: a lane per site (about 13 instructions a site in full warps
      // against 45 with sixteen lanes, but a chain three times as long)
      const bool lanes = kWarp && n > 6u;  // (in the CTA kernels its registers cost more than it saves)
      for (unsigned i0 = (unsigned)(tid & ~31); lanes && i0 < n; i0 += (unsigned)size) {
        const unsigned i = i0 + (unsigned)lane;
        uint32_t ent;
        int t;
        decode(lds_u2(q_s + 8u * (i < n ? i : i0)), ent, t);
        if (i < n) {
          hash_add(m, key_of(ent & kPosMask, t), i);
          const float val = site_value(t, (int)(ent & kPosMask), (int)(ent >> kPosBits), m != 0,
                                       [&](int tt, int np) { return hash_nu(m - 1, key_of((uint32_t)np, tt)); });
          asm volatile("st.shared.f32 [%0], %1;" :: "r"(nuq_s + 4u * (uint32_t)((m & 1) * cap) + 4u * i), "f"(val) : "memory");
          nz |= val != 0.f;
        }
      }
      for (unsigned i0 = (unsigned)(tid >> 5) * 2u; !lanes && i0 < n; i0 += (unsigned)(size >> 5) * 2u) {
        const unsigned i = i0 + (unsigned)(lane >> 4);
        const bool act = i < n && has16;
        uint32_t ent;
        int t;
        decode(lds_u2(q_s + 8u * (i < n ? i : i0)), ent, t);
        const int pos = (int)(ent & kPosMask), sg = pos - 3 * (int)__umulhi((unsigned)pos, 0x55555556u);
        if (i < n && (lane & 15) == 0) hash_add(m, key_of((uint32_t)pos, t), i);
        const uint32_t np = (ent + e16 + lds_u<0>(roff_s + ((ent >> (kPosBits - 5)) & ~31u) + (y16 & 255u))) & kPosMask;
        const int tt = t + (int)((y16 >> (8 + 2 * sg)) & 3u) - 1;
        const bool on = act && (unsigned)tt < (unsigned)L && ((occ[(size_t)(tt >> 5) * P + np] >> (tt & 31)) & 1u);
        const float v = on && m ? hash_nu(m - 1, key_of(np, tt)) : 0.f;
        const unsigned bal = __ballot_sync(0xffffffffu, on);
        const int deg = __popc(bal & (0x3fffu << half)) + (t == L - 1);  // with the detector edge
        const float x = v + __shfl_sync(0xffffffffu, v, mate);
        const float pa = __shfl_sync(0xffffffffu, x, half), pbs = __shfl_sync(0xffffffffu, x, half | 1),
                    g = __shfl_sync(0xffffffffu, x, half | 2), pd = __shfl_sync(0xffffffffu, x, half | 3),
                    pcs = __shfl_sync(0xffffffffu, x, half | 4), ee = __shfl_sync(0xffffffffu, x, half | 6),
                    h = __shfl_sync(0xffffffffu, x, half | 12);
        float r;
        if (sg == 0) r = (((pa + pbs) + pcs) + (pd + ee)) + (h + g);
        else if (sg == 1) r = ((pcs + pd) + (pa + pbs)) + ((ee + h) + g);
        else r = (((pcs + pd) + pa) + (pbs + ee)) + (h + g);
        const float inv = deg ? __frcp_rn((float)deg) : 0.f;
        const float val = m ? inv * r : inv * __frcp_rn((float)n0);
        if (i < n && (lane & 15) == 0) {
          asm volatile("st.shared.f32 [%0], %1;" :: "r"(nuq_s + 4u * (uint32_t)((m & 1) * cap) + 4u * i), "f"(val) : "memory");
          nz |= val != 0.f;
        }
      }
      if (nz) gs->nz[m & 1] = 1u;
      group_sync<kWarp>();
      // the other table and flag are the next level's, which fills them after
      // the barrier of its claims
      if (tid == 0) gs->nz[(m + 1) & 1] = 0u;
      for (uint32_t k = tid; k <= tab_mask; k += size) sts_u2(tab_s + 8u * ((uint32_t)(((m + 1) & 1) << tab_bits) + k), kNone, 0u);
      return gs->nz[m & 1] != 0u;
    };
    // nu of the sites of level m (queue qn, overflow rows [lo, hi]); true if any is not 0
    auto level_values = [&](int m, unsigned n, const uint2* qn, int lo, int hi) -> bool {
      const float* src = m ? nu + (size_t)((m - 1) & 1) * nu_n : nullptr;
      float* dst = nu + (size_t)(m & 1) * nu_n;
      auto value_of = [&](int tt, int np) {  // reached sites: of the previous level, or zeroed when claimed
        return (*word_ptr(tt >> 5, np) >> (tt & 31)) & 1u ? 0.f : src[plane(tt) + np];
      };
      if (tid == 0) gs->nz[m & 1] = 0u;
      group_sync<kWarp>();
      bool nz = false;
      const unsigned stored = min(n, (unsigned)cap);
      for (unsigned i = tid; i < stored; i += size) {
        uint32_t ent;
        int t;
        decode(qn[i], ent, t);
        const int pos = (int)(ent & kPosMask);
        const float x = site_value(t, pos, (int)(ent >> kPosBits), m != 0, value_of);
        dst[plane(t) + pos] = x;
        nz |= x != 0.f;
      }
      for (int w = lo; w <= hi; ++w)
        for (int pos = tid; pos < P; pos += size) {
          uint32_t word = over[(size_t)(m & 1) * over_n + (size_t)w * P + pos];
          while (word) {
            const int t = 32 * w + __ffs(word) - 1;
            word &= word - 1;
            const float x = site_value(t, pos, row_of(pos), m != 0, value_of);
            dst[plane(t) + pos] = x;
            nz |= x != 0.f;
          }
        }
      if (nz) gs->nz[m & 1] = 1u;
      group_sync<kWarp>();
      return gs->nz[m & 1] != 0u;
    };
    // detector mass: nu over the reached sites of t = L - 1, by the group's
    // first warp in a fixed order (the same for every group size)
    auto detector_mass = [&](int m) -> float {
      const float* dst = nu + (size_t)(m & 1) * nu_n;
      float part_sum = 0.f;
      if (tid < 32)
        for (int c = tid; c < A; c += 32) {
          const int pos = __ldg(ppos + c), w = (L - 1) >> 5;
          const uint32_t bit = (occ[(size_t)w * P + pos] & ~*word_ptr(w, pos)) >> ((L - 1) & 31);
          if (bit & 1u) part_sum += kMode == M_HASH ? hash_nu(m, key_of((uint32_t)pos, L - 1)) : dst[plane(L - 1) + pos];
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part_sum += __shfl_xor_sync(0xffffffffu, part_sum, o);
      return part_sum;  // valid in the first warp
    };

    int verdict = 0, fh = -1, mstop = 0;
    float mass = 0.f;
    bool hard = kMode == M_HASH && total > (unsigned)cap;  // left to the launch with planes
    bool wait = false;
    bool live = true;  // some nu of the level is not 0
    if (kMass && n0 > 0 && !hard) {
      if (kMode == M_HASH) level_hash(0, total);
      else level_values(0, total, queue, 0, gs->ohi[0]);
    }
    if (n0 > 0 && L == 1) {
      verdict = 1; fh = 1; mstop = 1;
      if (kMass && !hard) mass = detector_mass(0);
    } else if (n0 > 0 && !hard) {
      int cu_ = 0;  // rotating index of the current level
      for (int m = m0 + 1;; ++m) {
        const int nx = cu_ == 2 ? 0 : cu_ + 1, nn = nx == 2 ? 0 : nx + 1;
        const uint32_t qc_s = queue_s + 8u * (uint32_t)(((m - 1) & 1) * cap), qn_s = queue_s + 8u * (uint32_t)((m & 1) * cap);
        uint32_t* on = over + (size_t)(m & 1) * over_n;
        const uint32_t cf_s = gs_s + (uint32_t)offsetof(GroupShared, cf) + 8u * (uint32_t)nx;
        float* zero = nu + (size_t)((m - 1) & 1) * nu_n;
        // tubes [t_lo, t_lo + t_span) call for nothing; t_need: contacts in
        // layers not drawn yet
        const int t_need = G < L ? G - 1 : 0x7fffffff;
        const int t_lo = kPart ? 32 * wb : 0;
        const unsigned t_span = (unsigned)(min(min(t_need, L - 1), kPart ? 32 * (wb + NR) : 0x7fffffff) - t_lo);
        unsigned count = 0, f = 0;
        // sites at tubes [e_lo, e_lo + e_n) claim nothing outside those
        const int e_lo = kPart ? t_lo + 1 : 0;
        const unsigned e_n = (unsigned)max(0, t_lo + (int)t_span - 1 - e_lo);
        // n entries of the next level for this warp
        auto reserve = [&](unsigned n) -> unsigned {
          unsigned base = 0;
          if (lane == 0) base = atoms_add(cf_s, n);
          return __shfl_sync(0xffffffffu, base, 0);
        };
        // where the word of (entry, tube) lies in the window
        auto at_of = [&](uint32_t ent, int tt) -> uint32_t {
          return win_s + 4u * (uint32_t)(((tt >> 5) & nr_mask) * P + (int)(ent & kPosMask));
        };
        // Claims the contacts of a site per lane and appends them
        // (warp-collective).  The claim is one atomicAnd per contact, issued
        // without a look at the word first: fourteen in flight, and the old
        // word says both whether the site was free and that this lane has it.
        // (Fourteen loads first and claims of the set bits alone: fewer atomics,
        // one more round of latency.  us per call without and with them: W =
        // 64, L = 4096 17,489 and 22,956; W = 8, L = 64, 10^4 configurations 492
        // and 519 in CTAs, 594 in warps as well.)
        auto expand = [&](bool act, uint32_t ent, int t) {
          const int pos = (int)(ent & kPosMask);
          const int sg = pos - 3 * (int)__umulhi((unsigned)pos, 0x55555556u);
          const uint32_t ro_s = roff_s + 32u * (ent >> kPosBits);
          const int w = t >> 5, b = t & 31;
          const bool s2 = sg == 2, sz = sg == 0;
          uint32_t c = 0u;  // bit d: contact d was free and is this site's
          bool in = act;
          if (kPart) in = act && resident(w) && (b != 31 || resident(w + 1)) && (b != 0 || t == 0 || resident(w - 1));
          if (in) {
            uint4 o;  // offsets to rows r-2, r-1, r+1, r+2
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(o.x), "=r"(o.y), "=r"(o.z), "=r"(o.w) : "r"(ro_s));
            const uint32_t base = at_of(ent, t);
            const uint32_t nb = b == 31 ? at_of(ent, t + 1) : base, pbs = b == 0 && t ? at_of(ent, t - 1) : base;
            const uint32_t ub = s2 ? nb : base, db = sz ? pbs : base;
            const uint32_t o2 = 4u * o.x, o1 = 4u * o.y, p1 = 4u * o.z, p2 = 4u * o.w;
            const int bn = (b + 1) & 31, bp = (b - 1) & 31;
            const uint32_t k0 = ~(1u << b), kn = ~(1u << bn), kp = t ? ~(1u << bp) : 0xffffffffu;
            const uint32_t ku = s2 ? kn : k0, kd = sz ? kp : k0;
            const uint32_t w13 = atoms_and_at<0>(nb, kn), w12 = atoms_and_at<0>(pbs, kp), w11 = atoms_and_at<0>(db + p1, kd),
                           w10 = atoms_and_at<4>(db + o1, kd), w9 = atoms_and_at<-4>(db, kd), w8 = atoms_and_at<0>(ub + o1, ku),
                           w7 = atoms_and_at<-4>(ub + p1, ku), w6 = atoms_and_at<4>(ub, ku), w5 = atoms_and_at<-4>(base + p2, k0),
                           w4 = atoms_and_at<-8>(base + p1, k0), w3 = atoms_and_at<-4>(base + o1, k0),
                           w2 = atoms_and_at<4>(base + o2, k0), w1 = atoms_and_at<8>(base + o1, k0), w0 = atoms_and_at<4>(base + p1, k0);
            // each word is shifted so that the contact's bit comes first and a
            // funnel shift takes it in
            const int xs = 31 - b, xn = 31 - bn, xp = 31 - bp;
            const int xu = s2 ? xn : xs, xd = sz ? xp : xs;
            auto take = [&](uint32_t v, int sh) { c = __funnelshift_l(v << sh, c, 1); };
            take(w13, xn); take(w12, xp); take(w11, xd); take(w10, xd); take(w9, xd); take(w8, xu); take(w7, xu);
            take(w6, xu); take(w5, xs); take(w4, xs); take(w3, xs); take(w2, xs); take(w1, xs); take(w0, xs);
            if (t == 0) c &= sz ? ~((1u << 12) | (7u << 9)) : ~(1u << 12);
          } else if (act) {  // a row outside the window
            const int4 o = *reinterpret_cast<const int4*>(roff + 8 * (ent >> kPosBits));
            const int ro[5] = {o.x, o.y, o.z, o.w, 0};
            uint32_t v[14];
#pragma unroll
            for (int d = 0; d < 14; ++d) {
              const int tt = t + c_end(d) + (c_up(d) & s2) - (c_dn(d) & sz);
              v[d] = tt < 0 ? 0u : *word_ptr(tt >> 5, pos + c_dq(d) + ro[c_row(d)]) >> (tt & 31);
            }
#pragma unroll
            for (int d = 0; d < 14; ++d)
              if (v[d] & 1u) {
                const int tt = t + c_end(d) + (c_up(d) & s2) - (c_dn(d) & sz);
                const uint32_t bit = 1u << (tt & 31);
                if (atomicAnd(word_ptr(tt >> 5, pos + c_dq(d) + ro[c_row(d)]), ~bit) & bit) c |= 1u << d;
              }
          }
          // lane after lane's first, then second, .. claim: independent votes
          // and predicated stores for four (a site rarely claims more), no
          // branches
          const unsigned n_c = (unsigned)__popc(c);
          const unsigned b0 = __ballot_sync(0xffffffffu, n_c > 0u), b1 = __ballot_sync(0xffffffffu, n_c > 1u),
                         b2 = __ballot_sync(0xffffffffu, n_c > 2u), b3 = __ballot_sync(0xffffffffu, n_c > 3u);
          if (!b0) return;
          const uint32_t t4 = (uint32_t)t << 4, claimed = c;
          const unsigned p0 = (unsigned)__popc(b0), p1 = p0 + (unsigned)__popc(b1), p2 = p1 + (unsigned)__popc(b2);
          unsigned n_all = p2 + (unsigned)__popc(b3);
          const bool more = __any_sync(0xffffffffu, n_c > 4u);
          if (more) n_all = __reduce_add_sync(0xffffffffu, n_c);
          const unsigned first = kWarp ? count : reserve(n_all);
          auto append = [&](bool has, unsigned idx) {
            sts_u2_if(has && idx < (unsigned)cap, qn_s + 8u * idx, ent, t4 | (uint32_t)((__ffs(c) - 1) & 15));
            c &= c - 1u;
          };
          append(n_c > 0u, first + (unsigned)__popc(b0 & lt));
          append(n_c > 1u, first + p0 + (unsigned)__popc(b1 & lt));
          append(n_c > 2u, first + p1 + (unsigned)__popc(b2 & lt));
          append(n_c > 3u, first + p2 + (unsigned)__popc(b3 & lt));
          unsigned base = first + p2 + (unsigned)__popc(b3);
          unsigned bal;
          if (more)
            while ((bal = __ballot_sync(0xffffffffu, c != 0u)) != 0u) {
              append(c != 0u, base + (unsigned)__popc(bal & lt));
              base += (unsigned)__popc(bal);
            }
          if (kWarp) count = base;
          // the same once more where a claim needs a look: near layers not
          // drawn, the end layer or the window's edges, beyond the queue, or
          // with nu in planes
          const bool look = claimed && (kMode == M_PLANES || (unsigned)(t - e_lo) >= e_n);
          if (__any_sync(0xffffffffu, look) || base > (unsigned)cap) {
            base = first;
            c = claimed;
            while ((bal = __ballot_sync(0xffffffffu, c != 0u)) != 0u) {
              const unsigned idx = base + (unsigned)__popc(bal & lt);
              if (c) {
                uint32_t en;
                int tt;
                decode(make_uint2(ent, t4 | (uint32_t)(__ffs(c) - 1)), en, tt);
                if (kMode != M_HASH && idx >= (unsigned)cap) {
                  atomicOr(on + (size_t)(tt >> 5) * P + (en & kPosMask), 1u << (tt & 31));
                  reds_min(gs_s + (uint32_t)offsetof(GroupShared, olo) + 4u * (uint32_t)nx, tt >> 5);
                  reds_max(gs_s + (uint32_t)offsetof(GroupShared, ohi) + 4u * (uint32_t)nx, tt >> 5);
                }
                f |= (tt >= t_need ? F_NEED : 0u) | (tt == L - 1 ? F_HIT : 0u) | (resident(tt >> 5) ? 0u : F_OUT);
                if (kMode == M_PLANES) zero[plane(tt) + (en & kPosMask)] = 0.f;  // level m holds nothing at step m - 1
                c &= c - 1u;
              }
              base += (unsigned)__popc(bal);
            }
          }
        };
        const unsigned stored = min(total, (unsigned)cap);
        for (unsigned i0 = (unsigned)(tid & ~31); i0 < stored; i0 += (unsigned)size) {
          const unsigned i = i0 + (unsigned)lane;
          uint32_t ent;
          int t;
          decode(lds_u2(qc_s + 8u * (i < stored ? i : i0)), ent, t);
          expand(i < stored, ent, t);
        }
        if (kMode != M_HASH && total > (unsigned)cap) {  // sites of this level beyond the queue
          uint32_t* oc = over + (size_t)((m - 1) & 1) * over_n;
          const int lo = gs->olo[cu_], hi = gs->ohi[cu_];
          for (int w = lo; w <= hi; ++w)
            for (int p0 = tid & ~31; p0 < P; p0 += size) {
              const int pos = p0 + lane;
              uint32_t word = pos < P ? oc[(size_t)w * P + pos] : 0u;
              if (word) oc[(size_t)w * P + pos] = 0u;
              uint32_t ent = 0u;
              if (word) ent = (uint32_t)pos | (uint32_t)row_of(pos) << kPosBits;
              while (__any_sync(0xffffffffu, word != 0u)) {
                const bool act = word != 0u;
                const int b = act ? __ffs(word) - 1 : 0;
                word &= word - 1u;
                expand(act, ent, 32 * w + b);
              }
            }
        }
        __syncwarp();
        if (kWarp) {
          total = count;
          f = __any_sync(0xffffffffu, f != 0u) ? __reduce_or_sync(0xffffffffu, f) : 0u;
          if (total > (unsigned)cap && lane == 0) { gs->olo[nn] = 0x7fffffff; gs->ohi[nn] = -1; }
          __syncwarp();
        } else {
          if (f) reds_or(cf_s + 4u, f);
          if (tid == 0) { gs->cf[nn][0] = 0u; gs->cf[nn][1] = 0u; gs->olo[nn] = 0x7fffffff; gs->ohi[nn] = -1; }
          __syncthreads();
          const uint2 cf = lds_u2(cf_s);
          total = cf.x;
          f = cf.y;
        }
        cu_ = nx;
        if (total == 0) { mstop = m; break; }
        if (kMode == M_HASH && total > (unsigned)cap) { hard = true; break; }
        if (f & F_NEED) {  // the new sites have contacts in the next layers
          if (kPre && !(f & F_HIT) && (G >> 5) >= a.rows_ready) {  // to be drawn by the next launch: leave
            wait = true;
            uint2* saved = reinterpret_cast<uint2*>(scratch + Q.a_nu);
            for (unsigned k = tid; k < min(total, (unsigned)cap); k += size) saved[k] = queue[(m & 1) * cap + k];
            for (int w = wb; w < wb + NR && 32 * w < G; ++w)
              for (int k = tid; k < P; k += size) back[(size_t)w * P + k] = win[(w & nr_mask) * P + k];
            if (tid == 0) {
              state->phase = 1; state->m = m; state->total = total; state->wb = wb; state->G = G; state->n0 = n0;
              state->olo = gs->olo[nx]; state->ohi = gs->ohi[nx];
            }
            break;
          }
          if (kMass || !(f & F_HIT)) draw();
        }
        if (kMode == M_HASH && live) {
          live = level_hash(m, total);
          if (live && (f & F_HIT)) mass = detector_mass(m);
          if (!live && !a.full) break;  // nu has underflowed everywhere: the mass is 0
        }
        if (kMode == M_PLANES || (kPart && NR > 0 && (f & F_OUT))) {
          int lo = 0, hi = 0;  // tubes of the new level
          if (kMode != M_PLANES || ring_mask >= 0) {
            if (tid == 0) { gs->span[0] = gs->olo[nx] < 0x7fffffff ? 32 * gs->olo[nx] : 0x7fffffff; gs->span[1] = 32 * gs->ohi[nx] + 31; }
            group_sync<kWarp>();
            lo = 0x7fffffff; hi = -1;
            for (unsigned i = tid; i < min(total, (unsigned)cap); i += size) {
              uint32_t ent;
              int t;
              decode(lds_u2(qn_s + 8u * i), ent, t);
              lo = min(lo, t);
              hi = max(hi, t);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0) { atomicMin(&gs->span[0], lo); atomicMax(&gs->span[1], hi); }
            group_sync<kWarp>();
            lo = gs->span[0];
            hi = gs->span[1];
            group_sync<kWarp>();
          }
          if (kMode == M_PLANES) {
            // the rings hold the levels m - 1 and m only while their tubes
            // (a level lies within one tube of the previous one's) and the
            // tubes around them are fewer than the rings' planes
            if (ring_mask >= 0 && hi - lo + 5 > ring_mask + 1) { hard = true; break; }
            if (live) live = level_values(m, total, queue + (m & 1) * cap, gs->olo[nx], gs->ohi[nx]);
            if (live && (f & F_HIT)) mass = detector_mass(m);
            if (!live && !a.full) break;  // nu has underflowed everywhere: the mass is 0
          }
          if (kPart && NR > 0 && (f & F_OUT)) {  // keep the window on the frontier
            if ((lo >> 5) < wb && (hi >> 5) < wb + NR - 1) slide(-1);
            else if ((hi >> 5) >= wb + NR && (lo >> 5) > wb) slide(1);
          }
        }
        if (f & F_HIT) {
          verdict = 1; fh = m + 1; mstop = m + 1;
          break;
        }
      }
    }
    if (tid == 0 && !wait) {
      if (kPre) state->phase = 2;
      if (hard) atomicAdd(a.count + 1, 1ull);
      if (kMass) Q.out.mass[rel] = hard ? -1.f : mass;
      else if (Q.out.mass) Q.out.mass[rel] = 0.f;
      if ((!kMass || a.full) && !hard) {
        Q.out.verdict[rel] = (uint8_t)verdict;
        if (Q.out.first_hit) Q.out.first_hit[rel] = fh;
        if (Q.out.m_stop) Q.out.m_stop[rel] = mstop;
        if (verdict && Q.out.n_perc) atomicAdd(Q.out.n_perc, 1ull);
        if (!kMass && verdict && Q.want_mass) atomicAdd(a.count, 1ull);
      }
    }
    group_sync<kWarp>();
  }
}

// kThreads: threads of a group; 32 = a warp, four to a CTA.  Registers are
// bounded so that 24 to 28 warps (groups of a warp, or of 128 or 256 threads)
// or one CTA of 512 threads fit an SM.  (Seven CTAs of 128 threads instead of
// six, 72 registers: W = 6, L = 96, p = 0.3, 1,024 configurations 734 -> 524
// us; eight, 64 registers, spill: W = 20, L = 301 1,540 -> 1,690 us.)
template <int kThreads, bool kPart, int kMode>
__global__ void __launch_bounds__(kThreads == 32 ? 128 : kThreads, kThreads == 32 ? 6 : kThreads == 128 ? 7 : kThreads == 256 ? 3 : 1)
    wave_kernel(const __grid_constant__ WaveArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (a.gate.closed()) return;
  if (kThreads == 32) {
    const int w = threadIdx.x >> 5;
    wave_body<true, kPart, kMode>(a, smem_raw + (size_t)w * a.group_smem,
                                  a.scratch + ((long long)blockIdx.x * (blockDim.x >> 5) + w) * a.scratch_stride);
  } else {
    wave_body<false, kPart, kMode>(a, smem_raw, a.scratch + (long long)blockIdx.x * a.scratch_stride);
  }
}

template <int kThreads>
const void* wave_fn_of(bool part, int mode) {
  if (mode == M_LEVELS) return part ? (const void*)wave_kernel<kThreads, true, M_LEVELS> : (const void*)wave_kernel<kThreads, false, M_LEVELS>;
  if (mode == M_HASH) return part ? (const void*)wave_kernel<kThreads, true, M_HASH> : (const void*)wave_kernel<kThreads, false, M_HASH>;
  constexpr int T = kThreads == 32 ? 128 : kThreads;  // these: CTAs
  if (mode == M_PRE) return part ? (const void*)wave_kernel<T, true, M_PRE> : (const void*)wave_kernel<T, false, M_PRE>;
  return part ? (const void*)wave_kernel<T, true, M_PLANES> : (const void*)wave_kernel<T, false, M_PLANES>;
}

const void* wave_fn(int threads, bool part, int mode) {
  return threads == 32    ? wave_fn_of<32>(part, mode)
         : threads == 128 ? wave_fn_of<128>(part, mode)
         : threads == 256 ? wave_fn_of<256>(part, mode)
                          : wave_fn_of<512>(part, mode);
}

// Layers drawn ahead of M_PRE launches: a CTA per configuration and chunk of
// eight layers of the word rows [row0, row1), into the byte of the words of the
// row in the configuration's scratch.  The first chunk of a row clears the
// row of the overflow maps.
__global__ void __launch_bounds__(512) wave_draw_kernel(const __grid_constant__ WaveArgs a, int row0, int row1) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* tile = reinterpret_cast<uint32_t*>(smem_raw);
  const int chunks = 4 * (row1 - row0);
  const long long item = blockIdx.x / chunks;
  if (a.gate.closed()) return;
  if (a.state[item].phase == 2) return;
  int qi = 0;
  if (a.nq > 1) {
    int hi = a.nq - 1;
    while (qi < hi) {
      const int mid = (qi + hi + 1) >> 1;
      if (a.qs[mid].item0 <= item) qi = mid; else hi = mid - 1;
    }
  }
  const WaveQuery& Q = a.nq > 1 ? a.qs[qi] : a.q0;
  const int P = Q.P, G = 32 * row0 + 8 * (int)(blockIdx.x % chunks), w = G >> 5, tid = threadIdx.x, size = blockDim.x;
  char* scratch = a.scratch + item * a.scratch_stride;
  uint8_t* to = reinterpret_cast<uint8_t*>(scratch + Q.a_back) + 4 * (size_t)w * P + ((G >> 3) & 3);
  if (w >= Q.TW) return;
  if ((G & 31) == 0) {
    uint32_t* over = reinterpret_cast<uint32_t*>(scratch + Q.a_over);
    for (int k = tid; k < P; k += size) {
      over[(size_t)w * P + k] = 0u;
      over[(size_t)(Q.TW + w) * P + k] = 0u;
    }
  }
  for (int k = tid; k < P; k += size) tile[k] = 0u;
  __syncthreads();
  const uint32_t tile_s = smem_at(tile);
  if (G < Q.L)
    draw_layers(Q, item - Q.item0, G, min(G + 8, Q.L), tid, size, true, tile_s, 7,
                [&](int t, int pos) { reds_or(tile_s + 4u * (uint32_t)pos, 1u << (t & 7)); });
  __syncthreads();
  for (int k = tid; k < P; k += size) to[4 * (size_t)k] = (uint8_t)tile[k];
}

int ceil_log2(long long x) {
  int b = 0;
  while ((1ll << b) < x) ++b;
  return b;
}

inline size_t up(size_t x, size_t m) { return (x + m - 1) / m * m; }

void fill_lattice(WaveQuery& w, const Lattice& lat) {
  w.W = lat.W; w.L = lat.L; w.A = lat.A; w.P = lat.P; w.TW = lat.TW;
  w.s_begin = lat.s_begin; w.n_strips = lat.n_strips;
  w.divS = ceil_log2(lat.A);
  w.divM = (uint32_t)((1ull << (31 + w.divS)) / (unsigned long long)lat.A + 1ull);
  w.strip_row = lat.strip_row; w.row_off = lat.row_off; w.ppos = lat.ppos;
}

}  // namespace

namespace {

// The query table goes through kernel parameters: asynchronous, and no
// pageable host copy.
constexpr int kUpload = 14;
struct UploadChunk {
  int n;
  WaveQuery q[kUpload];
};
static_assert(sizeof(UploadChunk) <= 4000, "kernel parameters");
// a word a thread: the lanes of a warp read the parameters one after the other
// (a query a thread, with all its words one after the other in one warp: 22 us
// for 14 queries)
__global__ void wave_upload_kernel(WaveQuery* dst, const __grid_constant__ UploadChunk c) {
  constexpr int kWords = sizeof(WaveQuery) / 4;
  static_assert(sizeof(WaveQuery) % 4 == 0, "whole words");
  for (int i = threadIdx.x; i < c.n * kWords; i += blockDim.x)
    reinterpret_cast<uint32_t*>(dst)[i] = reinterpret_cast<const uint32_t*>(c.q)[i];
}

// One launch over the queries that run with the same group size.
struct WaveLaunch {
  int mode = M_LEVELS, threads = 0;
  bool part = false, hard = false, full = false;
  int cls = 0;               // launches of one class share the counts
  unsigned long long min_count = 1, max_count = ~0ull;
  std::vector<WaveQuery> q;
  long long items = 0;
  size_t group_smem = 0, stride = 256;
  long long grid = 0;
  size_t per_cta() const { return threads == 32 ? 4 : 1; }
  size_t table_b() const { return q.size() > 1 ? up(sizeof(WaveQuery) * q.size(), 256) : 0; }
};

double density(const WaveQuery& w) { return w.density; }
void fill_density(WaveQuery& w, const StreamQuery& s) {
  const double p = (double)s.occ.T / 4294967296.0;
  w.density = (float)(s.occ_bits ? s.density : p);
  w.density_most = (float)(s.occ_bits ? s.density_most : p);
}
// Sites of a level, on average over a percolating configuration: the start
// layer, p A sites, is also about the largest (measured at W = 24: 85 at p =
// 0.18, 141 at 0.2, 347 at 0.3, 1,576 at 0.9).
double level_sites(const WaveQuery& w) {
  const double p = std::max(density(w), 1e-9), f = 1.0 - 0.0256 / (p * p);
  return p * w.A * std::max(f, 0.1);
}

// Threads of a group.  With more configurations than groups fit the device,
// few (more configurations in flight; a level's fixed cost is paid by every
// warp); else more (a level is a chain of instructions: more warps, fewer
// sites each), and more still where levels are large for their lattice (from 32
// and 100 sites a level on; without that, times what it takes: W = 24, L = 64, p
// = 0.3, 20 configurations 1.49, W = 14, L = 100, p = 0.2, 300 of them 1.33, W =
// 12, L = 200, p = 0.2, 60 of them 1.22; twice or half the sites: no gain in 15
// calls).
int group_threads(int A, long long n, int nsm) {
  if (A <= 640) return n <= 8ll * nsm ? 128 : 32;
  if (A <= 2000) return n <= 2ll * nsm ? 256 : 128;
  if (A <= 5000) return n <= nsm ? 512 : 256;
  return 512;
}
int group_threads(const WaveQuery& w, long long n, int nsm) {
  const int t = group_threads(w.A, n, nsm);
  const double s = 20.0 * level_sites(w);
  if (n <= nsm) return std::max(t, s > 2000.0 ? 512 : s > 640.0 ? 256 : 32);
  return n <= 2ll * nsm && s > 640.0 ? std::max(t, 256) : t;
}

// Shared memory (at most `most` bytes; `share`: of an SM's, per configuration,
// if all of them are resident) and scratch of query w in a launch.
// False: no room for the hash tables.
// The targets leave an SM as many groups as its registers allow; with masses in
// tables twice that, as fewer configurations percolate than have levels.  Half
// of them: W = 20, L = 301, p = 0.172, 500 configurations 1.75 times the time,
// 14 other calls as before, but W = 10, L = 100, p = 0.22, 3,000 of them 0.93.
// Tables of twice or half the size: within 2 % over 15 calls.
bool place(WaveQuery& w, WaveLaunch& l, size_t most, bool full_rings, size_t share) {
  const size_t row_b = sizeof(uint32_t) * (size_t)w.P;
  const bool hash = l.mode == M_HASH;
  size_t target = l.threads == 32 ? 12 * 1024 : l.threads == 128 ? 36 * 1024 : l.threads == 256 ? 72 * 1024 : most;
  if (hash) target = std::min(most, 2 * target);
  target = std::max(target, std::min(most, share));
  w.cap = (int)std::min<long long>(w.A, (long long)(1.1 * w.density_most * w.A) + 64);
  const size_t head = kSharedHead + 32 * (size_t)(2 * w.W + 1);
  w.tab_bits = 0;
  size_t tab = 0;
  bool window = true;
  if (!hash) {
    // near the threshold levels are small after the first few and span up to 90
    // tubes: a window of four rows before room for those few; else room for
    // large levels, of a tube or two, and two rows
    const int least = (int)std::min<long long>(w.A, l.threads == 32 ? 512 : 1200);
    const bool small = 1.5 * level_sites(w) <= least;
    auto with = [&](int n) { return head + 128 + 2 * sizeof(uint2) * (size_t)least + std::min(w.TW, n) * row_b; };
    window = with(1) <= most;  // W <= 128
    const size_t rows = head + 128 + std::min(w.TW, with(2) <= most ? 2 : window ? 1 : 0) * row_b;
    const int room = most > rows ? (int)((most - rows) / (2 * sizeof(uint2))) : 0;
    w.cap = std::min(w.cap, small && window ? least : std::max(least, room));
  } else {
    w.cap = std::min(w.A, w.cap + w.cap / 8 + 32);
    w.tab_bits = ceil_log2(std::max(3 * w.cap / 2, (int)(4.0 * level_sites(w))) + 1);
    tab = (16ull << w.tab_bits) + 8 * (size_t)w.cap;
    if (w.L > 16384) return false;
  }
  const size_t fixed = head + 2 * sizeof(uint2) * (size_t)w.cap + tab + 64;
  // every word row in shared memory if they fit the target, else a power of
  // two of them
  auto fits = [&](int rows, size_t lim) { return fixed + (size_t)rows * row_b <= lim; };
  if (fits(w.TW, target) || (w.TW <= 2 && fits(w.TW, most))) {
    w.NR = w.TW; w.nr_mask = -1;
  } else {
    w.NR = 0;
    for (int r = 1; window && r < w.TW && (fits(r, target) || (r <= 2 && fits(r, most))); r *= 2) w.NR = r;
    w.nr_mask = w.NR - 1;
    if (hash && w.NR < 2) return false;
  }
  size_t o = head;
  w.o_win = (int)o; o += w.NR * row_b;
  w.o_occ = -1;
  if (hash && w.NR == w.TW && fits(2 * w.TW, target)) { w.o_occ = (int)o; o += w.TW * row_b; }
  o = up(o, 16);
  w.o_queue = (int)o; o += 2 * sizeof(uint2) * (size_t)w.cap;
  o = up(o, 16);
  w.o_tab = (int)o; o += tab;
  l.group_smem = std::max(l.group_smem, up(o, 16));
  l.part = l.part || w.NR < w.TW;
  const size_t map_b = up(row_b * w.TW, 256);
  size_t off = 0;
  w.a_over = 0;
  if (!hash) off = up(2 * row_b * w.TW, 256);
  w.a_back = (long long)off;
  if (w.NR < w.TW) off += map_b;
  if (l.mode == M_PRE && w.NR == w.TW) off += map_b;
  w.a_occ = w.a_nu = (long long)off;
  w.ring_mask = -1;
  if (l.mode == M_PRE) off += up(sizeof(uint2) * (size_t)w.cap, 256);  // a queue between launches
  if ((hash || l.mode == M_PLANES) && w.o_occ < 0) off += map_b;
  if (l.mode == M_PLANES) {
    w.a_nu = (long long)off;
    if (!full_rings && w.L > 128) w.ring_mask = 127;
    off += up(2 * row_b * (size_t)(w.ring_mask < 0 ? w.L : 128), 256);
  }
  l.stride = std::max(l.stride, off);
  return true;
}

// Groups of a launch that fit the device at once.  What the driver says is kept
// per device, kernel and shared memory (at most kFits entries): asking took
// several microseconds a launch.
constexpr size_t kFits = 256;
std::mutex g_fit_mu;
std::map<std::tuple<int, const void*, size_t>, int> g_fit;

pc_status resident_groups(const WaveLaunch& l, int nsm, int optin, long long* n) {
  const void* f = wave_fn(l.threads, l.part, l.mode);
  int dev = 0;
  PC_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_fit_mu);
  const auto key = std::make_tuple(dev, f, l.group_smem);
  const auto known = g_fit.find(key);
  if (known != g_fit.end()) {
    *n = (long long)known->second * nsm * (long long)l.per_cta();
    return PC_OK;
  }
  // the same limit on every call: calls from several threads never lower it
  PC_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
  int per_sm = 0;
  PC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, l.threads * (int)l.per_cta(), l.group_smem * l.per_cta()));
  if (per_sm < 1) { set_error("wavefront solver: no block fits an SM"); return PC_ERR_INTERNAL; }
  if (g_fit.size() >= kFits) g_fit.clear();
  g_fit[key] = per_sm;
  *n = (long long)per_sm * nsm * (long long)l.per_cta();
  return PC_OK;
}

// The launches of a class of queries (item0 set).
//  - Verdicts only: the levels.
//  - Masses too, and every configuration resident at once: levels and masses in
//    one pass (the longest configuration's chain of levels is the time, and it
//    usually percolates).  Not where the caller asks for verdicts first and
//    hardly one is expected to percolate (`few`).
//  - Else the levels, then the masses of the percolating ones: in hash tables,
//    by CTAs while these are few, by warps where more percolate than CTAs fit
//    (a level then costs fewer instructions); or in rings of planes where a
//    start layer does not fit the tables, or levels are large: sixteen lanes a
//    site cost most there (W = 24, L = 16, p = 0.95, 1,500 configurations:
//    12,260 -> 2,410 us; L = 64, 4 configurations, 40 sites a level: 410 us in
//    tables, 660 in planes).  The line, 48 sites for 128 threads: a third of it
//    costs 1.2 to 1.3 times the time in four of 15 calls and saves 11 % in one,
//    five times as much 1.5 to 2 times in four.  With planes and nearly every configuration
//    percolating, levels and masses go in one pass again, with one draw (W = 14,
//    L = 14, 1,500 configurations, p = 0.95 770 us in two passes, 588 in one; at p
//    = 0.35 still 1.2 to 1.4 times as fast over 16 lattices) -- where no ring
//    can overflow (W = 30, L = 180, p = 0.35, 200 configurations 2,100 and 2,450).
//  - Last, masses that did not fit (marked -1), with a plane for every layer.
pc_status launches_of(const std::vector<WaveQuery>& qs, long long items, int threads, int nsm, int optin, bool ahead,
                      bool few, long long at_once, std::vector<WaveLaunch>& out) {
  const long long per_sm = (std::min(items, at_once) + nsm - 1) / nsm;
  // (more than 32 to an SM: less than any target; not taken into account or always, 15 calls take the same)
  const size_t share = per_sm > 32 ? 0 : (size_t)optin / (size_t)per_sm - (per_sm > 1 ? 1024 : 64);
  auto make = [&](int mode, int t, bool full_rings, WaveLaunch& l) -> bool {
    l = WaveLaunch();
    l.mode = mode; l.threads = t; l.items = items; l.hard = mode == M_PLANES && full_rings;
    for (WaveQuery w : qs) {
      if (!place(w, l, (size_t)optin / l.per_cta() - 64, full_rings, share)) return false;
      l.q.push_back(w);
    }
    return true;
  };
  bool some = false, all = true, most = true;
  double sites = 0.0;
  for (const WaveQuery& w : qs) {
    some = some || w.want_mass;
    all = all && w.want_mass;
    most = most && density(w) > fibre_threshold(w.W, w.L) + 0.1;
    // in a short fibre the start layer is one of few levels
    sites = std::max({sites, level_sites(w), density(w) * w.A / w.L});
  }
  const int mt = std::max(threads, 128);
  WaveLaunch levels, hash, warps, planes;
  make(ahead ? M_PRE : M_LEVELS, threads, false, levels);
  if (!some) { out.push_back(levels); return PC_OK; }
  const bool has_hash = sites <= 3.0 * mt / 8 && make(M_HASH, mt, false, hash);
  bool left = true;  // something may be left to the last launch
  long long fit = 0;
  if (has_hash) {
    const pc_status rc = resident_groups(hash, nsm, optin, &fit);
    if (rc) return rc;
  }
  bool full = false;
  const bool has_warps = threads == 32 && make(M_HASH, 32, false, warps);
  if (all && !ahead && !few && has_hash && items <= std::min(fit, at_once)) {
    full = true;
    hash.full = true;
    out.push_back(hash);
  } else {
    out.push_back(levels);
    if (has_hash) {
      if (has_warps) {
        hash.max_count = (unsigned long long)fit;
        warps.min_count = (unsigned long long)fit + 1ull;
        out.push_back(warps);
      }
      out.push_back(hash);
    } else {
      make(M_PLANES, mt, false, planes);
      left = false;
      for (const WaveQuery& w : planes.q) left = left || w.ring_mask >= 0;
      if (all && most && !ahead && !left) {
        full = planes.full = true;
        out.back() = planes;
      } else {
        out.push_back(planes);
      }
    }
  }
  if (left) {
    make(M_PLANES, mt, true, planes);
    planes.full = full;
    out.push_back(planes);
  }
  return PC_OK;
}

}  // namespace

bool wave_is_slower(const Lattice& lat, double p, long long n, bool bits_only) {
  if (lat.A < (bits_only ? 2700 : 3000) || resident_fits(lat.W, lat.L)) return false;
  int dev = 0, nsm = 1, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  WaveQuery w = {};
  fill_lattice(w, lat);
  w.density = w.density_most = (float)p;
  WaveLaunch l;
  l.threads = 512;
  if (!place(w, l, (size_t)optin - 64, false, 0) || w.NR == 0) return true;
  const double sites = level_sites(w), k = 152.0 * (double)n / nsm;
  if (w.NR < std::min(w.TW, 2) || sites > 0.8 * w.cap || density(w) * w.A > 4.5 * w.cap) return sites > 760.0 + 20.0 * k;
  return sites > (bits_only ? 2040.0 : 2600.0) + 60.0 * k;
}

bool wave_memory_suffices(const StreamQuery& s, const WaveMemory& m) try {
  int dev = 0, nsm = 1, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  WaveQuery w = {};
  fill_lattice(w, s.lat);
  w.occ = s.occ; w.occ_bits = s.occ_bits;
  fill_density(w, s);
  w.want_mass = (!s.bits_only && s.out.mass) ? 1 : 0;
  w.n_cfg = s.n_cfg;
  const int threads = std::max(group_threads(w, std::min<long long>(s.n_cfg, m.max_groups), nsm), m.warps ? 32 : 128);
  std::vector<WaveLaunch> ls;
  if (launches_of({w}, s.n_cfg, threads, nsm, optin, false, false, m.max_groups, ls)) return false;
  for (const WaveLaunch& l : ls) {
    long long fit = 0;
    if (l.hard) continue;
    if (resident_groups(l, nsm, optin, &fit)) return false;
    if (3 * (m.bytes / l.stride) < (size_t)std::min(fit, l.items)) return false;
  }
  return true;
} catch (const std::bad_alloc&) {
  return false;
}

void release_wave() {
  std::lock_guard<std::mutex> lk(g_fit_mu);
  g_fit.clear();
}

int wave_threads(const StreamQuery& q, long long n_all, int nsm) {
  WaveQuery w = {};
  w.A = q.lat.A;
  fill_density(w, q);
  return group_threads(w, n_all, nsm);
}

pc_status run_wave(const StreamQuery* qs, int nq, cudaStream_t st, const WaveMemory* m, size_t limit) try {
  int dev = 0, nsm = 0, optin = 0;
  PC_CUDA(cudaGetDevice(&dev));
  PC_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  PC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  // classes by group size; within one, larger lattices first (their
  // configurations run longest)
  std::vector<int> order;
  for (int i = 0; i < nq; ++i)
    if (qs[i].n_cfg > 0) order.push_back(i);
  if (order.empty()) return PC_OK;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return qs[x].lat.N > qs[y].lat.N; });
  long long n_all = 0;
  for (int i : order) n_all += qs[i].n_cfg;
  if (m) n_all = std::min(n_all, m->max_groups);
  std::vector<WaveLaunch> ls;
  int classes = 0;
  auto build = [&](size_t most_ahead) -> pc_status {
    ls.clear();
    classes = 0;
    for (int threads : {512, 256, 128, 32}) {
      std::vector<WaveQuery> cq;
      long long items = 0;
      bool few = true;  // most configurations are not expected to percolate, and the caller says so
      for (int i : order) {
        const StreamQuery& s = qs[i];
        WaveQuery w = {};
        fill_lattice(w, s.lat);
        w.occ = s.occ; w.occ_bits = s.occ_bits; w.words_per_cfg = s.words_per_cfg; w.cfg0 = s.cfg0;
        w.out = s.out;
        fill_density(w, s);
        if (std::max(group_threads(w, n_all, nsm), m && !m->warps ? 128 : 32) != threads) continue;
        w.want_mass = (!s.bits_only && s.out.mass) ? 1 : 0;
        few = few && s.verdict_first && (s.occ_bits || density(w) < few_percolate_below(w.W, w.L, s.n_cfg));
        w.item0 = items; w.n_cfg = s.n_cfg;
        items += s.n_cfg;
        cq.push_back(w);
      }
      if (cq.empty()) continue;
      ++classes;
      // Few configurations of large lattices: their rows are drawn by the whole
      // device ahead of the levels, instead of by the one SM that works on them
      // (a third of its time at W = 64).
      bool ahead = !m && items <= nsm && threads >= 256;
      size_t maps = 0;
      for (const WaveQuery& w : cq) {
        ahead = ahead && (long long)w.A * w.L >= (1 << 18) && 4 * (size_t)w.P <= (size_t)optin - 64;
        maps = std::max(maps, 12 * (size_t)w.P * w.TW);
      }
      ahead = ahead && maps * (size_t)items <= most_ahead;
      const size_t first = ls.size();
      const pc_status rc = launches_of(cq, items, threads, nsm, optin, ahead, few, m ? m->max_groups : items, ls);
      if (rc) return rc;
      for (size_t k = first; k < ls.size(); ++k) ls[k].cls = classes - 1;
    }
    return PC_OK;
  };
  pc_status rc = build(std::min<size_t>(limit, 2ull << 30));
  if (rc) return rc;
  // Grids, and one scratch for all launches (they run one after the other) of
  // at most `total` bytes, one group at least.  The launch for what the rings
  // and tables left gets what the others need.
  auto plan = [&](size_t total, size_t* scratch) -> pc_status {
    *scratch = 0;
    for (int pass = 0; pass < 2; ++pass)
      for (WaveLaunch& l : ls) {
        if (l.hard != (pass == 1)) continue;
        long long fit = 0;
        const pc_status rc = resident_groups(l, nsm, optin, &fit);
        if (rc) return rc;
        const long long per_cta = (long long)l.per_cta();
        const size_t cta_b = l.stride * l.per_cta();
        if (l.mode == M_PRE) {
          l.grid = l.items;
          *scratch = std::max(*scratch, cta_b * (size_t)l.grid);
          continue;
        }
        const size_t most = l.hard ? std::min(total, std::max<size_t>(*scratch, 64u << 20)) : total;
        long long n = std::min<long long>(fit / per_cta, (l.items + per_cta - 1) / per_cta);
        n = std::min<long long>(n, (long long)(most / cta_b));
        if (m) n = std::min(n, (m->max_groups + per_cta - 1) / per_cta);
        l.grid = std::max<long long>(n, 1);
        *scratch = std::max(*scratch, cta_b * (size_t)l.grid);
      }
    return PC_OK;
  };
  size_t tables = 0, states = 0, head = 0;
  auto sizes = [&]() {
    tables = states = 0;
    for (const WaveLaunch& l : ls) {
      tables += l.table_b();
      if (l.mode == M_PRE) states += up(sizeof(WaveState) * (size_t)l.items, 256);
    }
    head = 256 * ls.size() + states;
  };
  sizes();
  cudaError_t e = cudaSuccess;
  char* mem = nullptr;
  size_t scratch = 0;
  if (m) {
    if ((rc = plan(m->bytes, &scratch))) return rc;
    if (classes != 1 || tables || scratch > m->bytes || ls.size() > 4) {
      set_error("wavefront solver: the caller's memory does not hold the query");
      return PC_ERR_INTERNAL;
    }
  } else {
    for (size_t total = limit;; total /= 8) {  // fewer groups where the memory for more cannot be had
      if ((rc = plan(total, &scratch))) return rc;
      e = scratch_alloc((void**)&mem, head + tables + scratch, st);
      if (e == cudaSuccess) break;
      if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "wavefront solver: scratch");
      cudaGetLastError();
      if (states) {  // rows drawn ahead need every configuration's at once: drawn by their groups instead
        if ((rc = build(0))) return rc;
        sizes();
      }
      if (total < (1ull << 20)) {
        set_error("wavefront solver: no memory for one configuration's state");
        return PC_ERR_OOM;
      }
    }
    e = cudaMemsetAsync(mem, 0, head, st);
  }
  char* at = m ? nullptr : mem + head;  // query tables
  char* const base = m ? m->scratch : mem + head + tables;
  char* state = m ? nullptr : mem + 256 * ls.size();
  for (size_t k = 0; k < ls.size() && e == cudaSuccess; ++k) {
    WaveLaunch& l = ls[k];
    WaveArgs a = {};
    a.q0 = l.q[0];
    a.nq = (int)l.q.size();
    a.n_items = l.items;
    a.group_smem = (int)l.group_smem;
    a.hard = l.hard ? 1 : 0;
    a.full = l.full ? 1 : 0;
    a.min_count = l.min_count;
    a.max_count = l.max_count;
    if (nq == 1) a.gate = qs[0].gate;
    a.work = m ? m->ctr + k : (unsigned long long*)(mem + 256 * k);
    a.count = m ? m->ctr + 4 : (unsigned long long*)(mem + 256 * l.cls + 64);
    a.scratch = base;
    a.scratch_stride = (long long)l.stride;
    if (l.table_b()) {
      a.qs = (const WaveQuery*)at;
      for (size_t b = 0; b < l.q.size() && e == cudaSuccess; b += kUpload) {
        UploadChunk u = {};
        u.n = (int)std::min<size_t>(kUpload, l.q.size() - b);
        for (int i = 0; i < u.n; ++i) u.q[i] = l.q[b + i];
        wave_upload_kernel<<<1, 512, 0, st>>>((WaveQuery*)at + b, u);
        e = cudaGetLastError();
      }
      at += l.table_b();
    }
    void* args[] = {&a};
    auto launch = [&]() {
      if (e == cudaSuccess)
        e = cudaLaunchKernel(wave_fn(l.threads, l.part, l.mode), dim3((unsigned)l.grid),
                             dim3(l.threads * (unsigned)l.per_cta()), args, l.group_smem * l.per_cta(), st);
    };
    if (l.mode != M_PRE) {
      launch();
      continue;
    }
    // rows drawn ahead in growing steps, so that configurations which end early
    // cost little; those that reach the last drawn row wait for the next step
    a.state = (WaveState*)state;
    state += up(sizeof(WaveState) * (size_t)l.items, 256);
    int rows = 0, most_p = 0;
    for (const WaveQuery& w : l.q) { rows = std::max(rows, w.TW); most_p = std::max(most_p, w.P); }
    if (e == cudaSuccess) e = cudaFuncSetAttribute(wave_draw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    for (int r0 = 0, r1 = std::min(4, rows); r0 < rows && e == cudaSuccess; r0 = r1, r1 = std::min(4 * r1, rows)) {
      wave_draw_kernel<<<(unsigned)(l.items * 4 * (r1 - r0)), 512, 4 * (size_t)most_p, st>>>(a, r0, r1);
      e = cudaGetLastError();
      a.rows_ready = r1;
      launch();
    }
  }
  if (e != cudaSuccess) rc = cuda_fail(e, "wavefront solver");
  if (mem) cudaFreeAsync(mem, st);
  return rc;
} catch (const std::bad_alloc&) {  // of the plan, before any device memory is taken
  set_error("wavefront solver: no host memory for the plan");
  return PC_ERR_OOM;
}

}  // namespace pc

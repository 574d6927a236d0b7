// Per-source path: one BFS per source, run by a persistent cooperative kernel that
// loops over the sources of the call and, per source, over BFS levels.
//
// Forward (shortest-path counting, Alg. 2 / Alg. 3, Sec. 3.2):
//   * top-down levels use active-edge parallelism (Sec. 3.1): the frontier's adjacency
//     lists are treated as one concatenated edge array; each warp takes an equal,
//     contiguous slice and maps edge -> owning frontier vertex by a search in the
//     exclusive degree prefix CD.  CD is not recomputed per level: every append to the
//     queue Q reserves its slot and its edge offset with one packed 64-bit atomicAdd,
//     so CD is produced in Q order as the frontier is built, and the backward sweep
//     reuses it (the scan / search reuse of Sec. 3.1).  A warp keeps a window of 128
//     CD entries in shared memory and has four 32-edge steps in flight at once.
//   * Alg. 3 tests d[w] and adds sigma in one parallel loop, which can drop a term when
//     a thread reads d[w] before another thread has set it.  Here an edge into a vertex not
//     reached at an earlier level (a bitmap test) raises its depth with an atomic maximum,
//     which tells the discoverer, and adds sigma in any case, so every parent edge contributes
//     once.  Depth values carry a base that grows from source to source, so depths of earlier
//     sources read as "not reached" and are not reset.
//   * bottom-up levels (direction switch): each unvisited vertex sums sigma over all its
//     neighbours in the frontier bitmap (all parents at level d-1, no early exit, so
//     sigma stays exact).
//   * the level bitmaps rotate: one is built, one is the frontier, one is cleared; the frontier is
//     merged into the visited bitmap word by word beside the sweep, so a level needs one grid
//     barrier and no pass over its vertices.
//   * sigma is kept modulo 2^64 with a sticky overflow bit; vertices whose count
//     overflows also get an extended-range value (double mantissa, int exponent).
// Backward (dependency accumulation, Alg. 4 / Alg. 5, successor checking):
//   for depth = D-1 .. 1, every edge (w, v) of the depth-level vertices w with
//   d[v] = d[w] + 1 adds sigma[w] * r[v] = sigma[w] / sigma[v] * (1 + delta[v] + omega[v])
//   to acc[w]; then delta[w] = acc[w] (updateDep), BC[w] += (omega[s] + 1) * delta[w]
//   (Eq. 3 / Eq. 4) and r[w] = (1 + delta[w] + omega[w]) / sigma[w].  Each term lies in
//   [0, n] and is added as a 128-bit fixed-point integer (64 fraction bits; per-lane and
//   warp-segmented sums, one pair of 64-bit integer atomics per segment): integer sums do not
//   depend on the order of the additions, so the result repeats bit for bit from run to run,
//   and a level whose successors have few arcs sums over theirs instead.
#include <climits>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "bc_internal.h"

namespace bcl {

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int U = 4;             // 32-edge steps in flight per warp
constexpr int WIN = 32 * U;      // owner window (queue entries) per warp
constexpr int kBaseMax = 1 << 30;  // depth values stay below (base + level)
constexpr int kPushFactor = 2;     // backward: push from a level with at most half of the arcs

struct WarpWin {
  int cd[WIN + 1];  // CD of window entries (INT_MAX past the range), then the next CD
  int v[WIN];       // vertex of each entry
  int bias[WIN];    // row_ptr[v] - CD: col position of edge e is e + bias
  int ex[WIN];      // extended-range exponent of the owner (backward, EXT only)
  double sg[WIN];   // sigma of the owner (backward; EXT: its mantissa)
};
constexpr size_t kSmemBytes = sizeof(WarpWin) * kWarps;

struct PK {
  int32_t n;
  int64_t nnz;
  int32_t max_degree;
  const int32_t *__restrict__ rp;
  const int32_t *__restrict__ ci;
  const int32_t *__restrict__ omega;
  const int32_t *__restrict__ src;
  int32_t nsrc;
  double *bc;
  int leaf_term;
  int32_t *depth, *Q, *CD, *lvl_off, *lvl_eoff;
  unsigned long long *sig;
  uint32_t *ovf, *vis;
  uint32_t *lvb[3];         // bitmap of level l in lvb[l % 3]; 1 and 2 lie in r (idle in the forward sweep)
  int32_t base;             // depth values of the first source start here; below: not reached
  unsigned long long *acc;  // [2n]: per vertex the low and high word of a 64.64 fixed-point sum
  double *r, *xm;
  int32_t *xe;
  PlainCtl *ctl;
  int32_t *out_depth;
  unsigned long long *out_sigma;
  uint8_t *out_ovf;
  float alpha, beta;
  uint64_t limit_ns;
  unsigned long long *trace;  // optional phase trace: (phase << 56 | level << 32, time) pairs
  int trace_cap;
  int no_cd_reuse;            // backward: rescan CD per level (ablation)
  int *bad;                   // plain_solo: set for a source id outside [0, n)
};

// Grid barrier; with tracing on, CTA 0 stamps the time at which every CTA has finished
// the phase (so consecutive stamps give each phase's duration, slowest CTA included).
template <bool SOLO = false>
__device__ __forceinline__ bool phase_sync(const PK &p, GridSync *gs, int phase, int level) {
  if (SOLO) {  // one CTA runs the source: nobody to wait for
    __syncthreads();
    return true;
  }
  const bool ok = grid_sync(gs, p.limit_ns);
  if (p.trace && blockIdx.x == 0 && threadIdx.x == 0) {
    int i = p.ctl->trace_n++;
    if (i < p.trace_cap) {
      p.trace[2 * i] = ((unsigned long long)phase << 56) | ((unsigned long long)(unsigned)level << 24);
      p.trace[2 * i + 1] = globaltimer_ns();
    }
  }
  return ok;
}

// Extended-range sigma: value = m * 2^e.
struct XS {
  double m;
  int e;
};

__device__ __forceinline__ XS xs_from_u64(unsigned long long s) {
  XS x;
  x.m = frexp((double)s, &x.e);
  return x;
}
__device__ __forceinline__ void xs_add(XS &a, XS b) {
  if (b.m == 0.0) return;
  if (a.m == 0.0) { a = b; return; }
  if (b.e > a.e) {
    a.m = ldexp(a.m, a.e - b.e) + b.m;
    a.e = b.e;
  } else {
    a.m += ldexp(b.m, b.e - a.e);
  }
}
__device__ __forceinline__ XS xs_norm(XS a) {
  int de;
  a.m = frexp(a.m, &de);
  a.e += de;
  return a;
}
__device__ __forceinline__ XS get_xs(const PK &p, int v) {
  if (test_bit(p.ovf, v)) {
    XS x;
    x.m = p.xm[v];
    x.e = p.xe[v];
    return x;
  }
  return xs_from_u64(p.sig[v]);
}

// Largest i in [lo, hi) with CD[i] <= x (CD non-decreasing on [lo, hi), CD[lo] <= x).
__device__ __forceinline__ int warp_find_owner(const int32_t *CD, int lo, int hi, int x) {
  const int lane = lane_id();
  while (hi - lo > 32) {
    int stride = (hi - lo + 31) / 32;
    int pos = lo + lane * stride;
    bool ok = pos < hi && CD[pos] <= x;
    unsigned b = __ballot_sync(BC_FULL, ok);
    int k = 31 - __clz(b);
    lo = lo + k * stride;
    hi = min(lo + stride, hi);
  }
  int pos = lo + lane;
  bool ok = pos < hi && CD[pos] <= x;
  unsigned b = __ballot_sync(BC_FULL, ok);
  return lo + (31 - __clz(b));
}

// Warp-aggregated append of up to U flagged vertices per lane to Q (and their degree
// prefix to CD) with one packed atomicAdd per warp.
// (ctr: the level's packed counter; its entries start at queue position q1, edge offset E1).
// The vertices' bits in the level's bitmap are set here too.
__device__ __forceinline__ void warp_append_u(const PK &p, const int (&w)[U], const bool (&isnew)[U],
                                              unsigned long long *ctr, int q1, int E1, uint32_t *lvb) {
  int cnt = 0, dsum = 0;
  int dg[U];
#pragma unroll
  for (int k = 0; k < U; k++) {
    dg[k] = isnew[k] ? (p.rp[w[k] + 1] - p.rp[w[k]]) : 0;
    cnt += isnew[k];
    dsum += dg[k];
  }
  if (__ballot_sync(BC_FULL, cnt > 0) == 0) return;
  int ctot, dtot;
  int cpre = warp_excl_scan(cnt, &ctot);
  int dpre = warp_excl_scan(dsum, &dtot);
  unsigned long long base = 0;
  if (lane_id() == 0) base = atomicAdd(ctr, pack_qe((unsigned)ctot, (unsigned)dtot));
  base = __shfl_sync(BC_FULL, base, 0);
  int pos = q1 + (int)(base >> 32) + cpre;
  int eo = E1 + (int)(base & 0xffffffffull) + dpre;
#pragma unroll
  for (int k = 0; k < U; k++) {
    if (isnew[k]) {
      set_bit_atomic(lvb, w[k]);
      p.Q[pos] = w[k];
      p.CD[pos] = eo;
      pos++;
      eo += dg[k];
    }
  }
}

// What a window holds per entry besides its vertex: nothing (MODE 0), sigma (1; EXT: as m 2^e), or
// r and its exponent (2).
template <int MODE, bool EXT = false>
__device__ __forceinline__ void fill_window(const PK &p, WarpWin &W, int base, int q1, int E1) {
  const int lane = lane_id();
  int vv[U], cc[U];
#pragma unroll
  for (int k = 0; k < U; k++) {
    int idx = base + lane + 32 * k;
    bool in = idx < q1;
    cc[k] = in ? p.CD[idx] : INT_MAX;
    vv[k] = in ? p.Q[idx] : -1;
  }
#pragma unroll
  for (int k = 0; k < U; k++) {
    int j = lane + 32 * k;
    W.cd[j] = cc[k];
    W.v[j] = vv[k];
    W.bias[j] = vv[k] >= 0 ? p.rp[vv[k]] - cc[k] : 0;
    if (MODE == 2) {
      W.sg[j] = vv[k] >= 0 ? p.r[vv[k]] : 0.0;
      if (EXT) W.ex[j] = vv[k] >= 0 ? p.xe[vv[k]] : 0;
    }
    if (MODE == 1) {
      if (EXT) {
        const XS x = vv[k] >= 0 ? get_xs(p, vv[k]) : XS{0.0, 0};
        W.ex[j] = x.e;
        W.sg[j] = x.m;
      } else {
        W.sg[j] = vv[k] >= 0 ? (double)p.sig[vv[k]] : 0.0;
      }
    }
  }
  if (lane == 0) W.cd[WIN] = (base + WIN < q1) ? p.CD[base + WIN] : E1;
  __syncwarp();
}

__device__ __forceinline__ int win_owner(const WarpWin &W, int e) {
  int j = 0;
#pragma unroll
  for (int s = WIN / 2; s >= 1; s >>= 1)
    if (W.cd[j + s] <= e) j += s;
  return j;
}

// Iterate the warp's slice of the edge range [E0, E1) of queue range [q0, q1), U x 32
// edges at a time.  body(e0, ee) is called once per window with the window filled.
template <int MODE, bool EXT = false, typename F>
__device__ __forceinline__ void edge_windows(const PK &p, WarpWin &W, int q0, int q1, int E0,
                                             int E1, int gwarp, int nwarps, F &&body) {
  long long E = (long long)E1 - E0;
  if (E <= 0) return;
  long long per = (E + nwarps - 1) / nwarps;
  per = (per + 31) & ~31ll;
  long long ebl = (long long)E0 + (long long)gwarp * per;
  if (ebl >= E1) return;
  const int eb = (int)ebl;
  const int ee = (int)min(ebl + per, (long long)E1);
  int base = warp_find_owner(p.CD, q0, q1, eb);
  for (int e0 = eb; e0 < ee; e0 += WIN) {
    fill_window<MODE, EXT>(p, W, base, q1, E1);
    body(e0, ee);
    // next window starts at the owner of edge e0 + WIN
    int jl = win_owner(W, e0 + WIN - 1);
    int nb = base + jl + ((e0 + WIN >= W.cd[jl + 1]) ? 1 : 0);
    __syncwarp();
    base = nb;
  }
}

// The level in progress: its number and depth value, its slots and where its entries start.
struct Lvl {
  int level, dv;            // dv = base + level
  int q1, E1;               // queue position and edge offset of its first entry
  unsigned long long *ctr;  // packed append counter
  int *ovf;                 // set when a vertex of the level passes 2^64
  bool povf;                // vertices of earlier levels may have
  uint32_t *cur;            // bitmap of the level (being built)
  const uint32_t *front;    // bitmap of the level before
};

// Reached before this level: vis holds the levels up to level - 2, and is being merged with the
// level before meanwhile.
__device__ __forceinline__ bool reached_before(const PK &p, const Lvl &L, int v) {
  return test_bit(p.vis, v) || test_bit(L.front, v);
}

__device__ void expand_topdown(const PK &p, WarpWin &W, const Lvl &L, int q0, int E0, int gwarp, int nwarps,
                               bool fast) {
  const int lane = lane_id();
  edge_windows<0>(p, W, q0, L.q1, E0, L.E1, gwarp, nwarps, [&](int e0, int ee) {
    int w[U], v[U];
    bool isnew[U], dag[U];
#pragma unroll
    for (int k = 0; k < U; k++) {
      int e = e0 + lane + 32 * k;
      int j = win_owner(W, e);
      v[k] = W.v[j];
      w[k] = e < ee ? p.ci[e + W.bias[j]] : -1;
    }
#pragma unroll
    for (int k = 0; k < U; k++) {
      isnew[k] = false;
      dag[k] = false;
      if (w[k] >= 0 && !reached_before(p, L, w[k])) {
        int old = atomicMax(p.depth + w[k], L.dv);
        isnew[k] = old < L.dv;
        dag[k] = true;  // discovered here or by another parent at this level
      }
    }
#pragma unroll
    for (int k = 0; k < U; k++) {
      if (dag[k]) {
        unsigned long long sv = p.sig[v[k]];
        if (fast) {
          atomicAdd(p.sig + w[k], sv);
        } else {
          unsigned long long old = atomicAdd(p.sig + w[k], sv);
          if (old + sv < old || test_bit(p.ovf, v[k])) {
            set_bit_atomic(p.ovf, w[k]);
            *L.ovf = 1;
            p.ctl->src_ovf = 1;
          }
        }
      }
    }
    warp_append_u(p, w, isnew, L.ctr, L.q1, L.E1, L.cur);
  });
}

// s += v; ov: a carry out of bit 63, or v had passed 2^64 itself.
__device__ __forceinline__ void sum_carry(unsigned long long &s, bool &ov, unsigned long long v, bool o) {
  const unsigned long long t = s + v;
  ov = ov || t < s || o;
  s = t;
}

// Bottom-up level: 32 consecutive vertices per warp, those not reached yet sum sigma over their
// neighbours in the frontier (all of them, no early exit).  A lane takes a row of up to
// kBuLane arcs, four in flight; the warp takes larger rows together, one after another, and
// reduces by shuffles.  Sums stay in registers: 64-bit additions to shared memory are
// compare-and-swap loops, which the arcs of one vertex, next to each other in a step, repeated up
// to 32 times (R-MAT scale 20: 363 us for a level-3 sweep with them).
constexpr int kBuLane = 32;
__device__ void sweep_bottomup(const PK &p, const Lvl &L, int gwarp, int nwarps) {
  const int lane = lane_id();
  for (int g = gwarp; g * 32 < p.n; g += nwarps) {
    const uint32_t seen = p.vis[g] | L.front[g];
    if (seen == BC_FULL) continue;
    const int u = g * 32 + lane;
    int st = 0, c = 0;
    if (u < p.n && !((seen >> lane) & 1u)) {
      st = p.rp[u];
      c = p.rp[u + 1] - st;
    }
    unsigned long long sum = 0ull;
    bool ov = false, found = false;
    if (c <= kBuLane) {
      for (int e = 0; e < c; e += U) {
        int pn[U];
        bool fr[U];
        unsigned long long sv[U];
#pragma unroll
        for (int k = 0; k < U; k++) pn[k] = e + k < c ? p.ci[st + e + k] : -1;
#pragma unroll
        for (int k = 0; k < U; k++) fr[k] = pn[k] >= 0 && test_bit(L.front, pn[k]);
#pragma unroll
        for (int k = 0; k < U; k++) sv[k] = fr[k] ? p.sig[pn[k]] : 0ull;
#pragma unroll
        for (int k = 0; k < U; k++) {
          if (!fr[k]) continue;
          found = true;
          sum_carry(sum, ov, sv[k], L.povf && test_bit(p.ovf, pn[k]));
        }
      }
    }
    __syncwarp();
    unsigned big = __ballot_sync(BC_FULL, c > kBuLane);
    while (big) {
      const int j = __ffs(big) - 1;
      big &= big - 1;
      const int s0 = __shfl_sync(BC_FULL, st, j), cj = __shfl_sync(BC_FULL, c, j);
      unsigned long long s = 0ull;
      bool o = false, f = false;
      for (int e = lane; e < cj; e += 32 * U) {
        int pn[U];
        bool fr[U];
        unsigned long long sv[U];
#pragma unroll
        for (int k = 0; k < U; k++) pn[k] = e + 32 * k < cj ? p.ci[s0 + e + 32 * k] : -1;
#pragma unroll
        for (int k = 0; k < U; k++) fr[k] = pn[k] >= 0 && test_bit(L.front, pn[k]);
#pragma unroll
        for (int k = 0; k < U; k++) sv[k] = fr[k] ? p.sig[pn[k]] : 0ull;
#pragma unroll
        for (int k = 0; k < U; k++) {
          if (!fr[k]) continue;
          f = true;
          sum_carry(s, o, sv[k], L.povf && test_bit(p.ovf, pn[k]));
        }
      }
      __syncwarp();
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) sum_carry(s, o, __shfl_xor_sync(BC_FULL, s, d), false);
      const bool ao = __any_sync(BC_FULL, o), af = __any_sync(BC_FULL, f);
      if (lane == j) {
        sum = s;
        ov = ao;
        found = af;
      }
    }
    if (found) {
      p.depth[u] = L.dv;
      p.sig[u] = sum;
      if (ov) {
        set_bit_atomic(p.ovf, u);
        *L.ovf = 1;
        p.ctl->src_ovf = 1;
      }
    }
    int wv[U] = {u};
    bool nv[U] = {found};
    warp_append_u(p, wv, nv, L.ctr, L.q1, L.E1, L.cur);
  }
}

// Extended-range sigma of an overflowed vertex: sum over its parents (depth value dp).
__device__ void ext_sigma(const PK &p, int w, int dp) {
  XS a;
  a.m = 0.0;
  a.e = 0;
  for (int e = p.rp[w]; e < p.rp[w + 1]; e++) {
    int x = p.ci[e];
    if (p.depth[x] == dp) xs_add(a, get_xs(p, x));
  }
  a = xs_norm(a);
  p.xm[w] = a.m;
  p.xe[w] = a.e;
}

// A term t in [0, 2^63) as a 128-bit fixed-point integer with 64 fraction bits (hi: integer
// part, lo: fraction), truncated below 2^-64; integer operations on the IEEE-754 fields.
__device__ __forceinline__ void fx_from(double t, unsigned long long &hi, unsigned long long &lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(t);
  const int ex = (int)((b >> 52) & 0x7ffull);
  hi = lo = 0ull;
  if (ex == 0 || (b >> 63)) return;  // zero (or below 2^-1022: far below 2^-64)
  const unsigned long long m = (b & 0x000fffffffffffffull) | (1ull << 52);  // t = m 2^(ex - 1075)
  const int sh = ex - 1075 + 64;                                           // fixed = m 2^sh
  if (sh >= 64) {
    hi = m << (sh - 64);
  } else if (sh > 0) {
    hi = m >> (64 - sh);
    lo = m << sh;
  } else if (sh > -64) {
    lo = m >> (-sh);
  }
}

// acc[o] += (hi, lo): integer additions, so their order does not matter.
__device__ __forceinline__ void acc_add(const PK &p, int o, unsigned hi, unsigned long long lo) {
  if (!(hi | lo)) return;
  unsigned long long *a = p.acc + 2 * (size_t)o;
  const unsigned long long old = lo ? atomicAdd(a, lo) : 0ull;
  const unsigned long long c = (lo && old + lo < old) ? 1ull : 0ull;  // the low word wrapped
  if (hi + c) atomicAdd(a + 1, hi + c);
}

// Level d's sums over the arcs (w, v) of its own entries w (pull).  A lane takes four consecutive
// arcs of a window and adds up the terms of one owner as it goes; where the owner changes
// inside its four arcs it writes the finished sum out, and only its last owner's sum goes
// through the warp-segmented reduction, so that runs once per 128 arcs and not at all where no
// arc leads to a successor.  hi: a sum of one owner's terms stays below n < 2^31.
template <bool EXT>
__device__ void accumulate_level(const PK &p, WarpWin &W, int dn, int q0, int q1, int E0, int E1,
                                 int gwarp, int nwarps) {
  const int lane = lane_id();
  edge_windows<1, EXT>(p, W, q0, q1, E0, E1, gwarp, nwarps, [&](int e0, int ee) {
    const int e = e0 + U * lane;
    int j = win_owner(W, min(e, ee - 1));
    int ow[U], nb[U];
#pragma unroll
    for (int k = 0; k < U; k++) {
      while (j < WIN - 1 && W.cd[j + 1] <= e + k) j++;
      ow[k] = j;
      nb[k] = e + k < ee ? p.ci[e + k + W.bias[j]] : -1;
    }
    int dv[U];
#pragma unroll
    for (int k = 0; k < U; k++) dv[k] = nb[k] >= 0 ? p.depth[nb[k]] : -1;
    double val[U];
    bool any = false;
#pragma unroll
    for (int k = 0; k < U; k++) {
      val[k] = 0.0;
      if (nb[k] >= 0 && dv[k] == dn) {
        val[k] = p.r[nb[k]];
        if (EXT) val[k] = ldexp(val[k], W.ex[ow[k]] - p.xe[nb[k]]);
        val[k] *= W.sg[ow[k]];  // sigma[w] / sigma[v] * (1 + delta[v] + omega[v])
        any = true;
      }
    }
    if (!__any_sync(BC_FULL, any)) return;
    unsigned hi = 0u;
    unsigned long long lo = 0ull;
#pragma unroll
    for (int k = 0; k < U; k++) {
      if (k > 0 && ow[k] != ow[k - 1]) {
        acc_add(p, W.v[ow[k - 1]], hi, lo);
        hi = 0u;
        lo = 0ull;
      }
      unsigned long long h, l;
      fx_from(val[k], h, l);
      lo += l;
      hi += (unsigned)h + (lo < l ? 1u : 0u);
    }
    const int o = ow[U - 1];
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const unsigned long long yl = __shfl_down_sync(BC_FULL, lo, s);
      const unsigned yh = __shfl_down_sync(BC_FULL, hi, s);
      const int oo = __shfl_down_sync(BC_FULL, o, s);
      if (lane + s < 32 && oo == o) {
        lo += yl;
        hi += yh + (lo < yl ? 1u : 0u);
      }
    }
    const int prev = __shfl_up_sync(BC_FULL, o, 1);
    if (lane == 0 || prev != o) acc_add(p, W.v[o], hi, lo);
  });
}

// The same sums over the arcs (v, w) of the next level's entries v (push): taken where that level
// has far fewer arcs, as the last levels of a low-diameter graph do (R-MAT scale 20: the level
// before the last walked 15 M arcs for the few thousand that lead on, 242 us).  The terms are
// the same products, so the integer sums are too.
template <bool EXT>
__device__ void push_level(const PK &p, WarpWin &W, int dd, int q0, int q1, int E0, int E1, int gwarp, int nwarps) {
  const int lane = lane_id();
  edge_windows<2, EXT>(p, W, q0, q1, E0, E1, gwarp, nwarps, [&](int e0, int ee) {
    int w[U], ow[U];
#pragma unroll
    for (int k = 0; k < U; k++) {
      const int e = e0 + lane + 32 * k;
      ow[k] = win_owner(W, e);
      w[k] = e < ee ? p.ci[e + W.bias[ow[k]]] : -1;
    }
    int dv[U];
#pragma unroll
    for (int k = 0; k < U; k++) dv[k] = w[k] >= 0 ? p.depth[w[k]] : -1;
#pragma unroll
    for (int k = 0; k < U; k++) {
      if (w[k] < 0 || dv[k] != dd) continue;
      double val = W.sg[ow[k]];
      if (EXT) {
        const XS x = get_xs(p, w[k]);
        val = ldexp(val, x.e - W.ex[ow[k]]) * x.m;
      } else {
        val *= (double)p.sig[w[k]];
      }
      unsigned long long h, l;
      fx_from(val, h, l);
      acc_add(p, w[k], (unsigned)h, l);
    }
  });
}

// delta, BC and r of a level from its sums; sigma is not needed after it and is cleared for the
// next source.
template <bool EXT>
__device__ void finalize_level(const PK &p, int q0, int q1, double ws, int gtid, int nthr) {
  for (int i = q0 + gtid; i < q1; i += nthr) {
    int w = p.Q[i];
    unsigned long long *a = p.acc + 2 * (size_t)w;
    const unsigned long long lo = a[0], hi = a[1];
    if (lo | hi) {
      a[0] = 0ull;
      a[1] = 0ull;
    }
    const double delta = (double)hi + (double)lo * 0x1p-64;
    double om = p.omega ? (double)p.omega[w] : 0.0;
    double sg;
    if (EXT) {
      XS x = get_xs(p, w);
      sg = x.m;
      p.xe[w] = x.e;
    } else {
      sg = (double)p.sig[w];
    }
    if (lo | hi) p.bc[w] += ws * delta;
    p.r[w] = (1.0 + delta + om) / sg;
    p.sig[w] = 0ull;
  }
}

// Exclusive prefix of x over the CTA's threads in thread order; *total = the CTA's sum.
// Contains barriers: every thread of the CTA calls it.
__device__ __forceinline__ int cta_excl_scan(int x, int *total, int *s_warp) {
  const int lane = lane_id(), wid = threadIdx.x >> 5;
  int wt;
  const int pre = warp_excl_scan(x, &wt);
  if (lane == 0) s_warp[wid] = wt;
  __syncthreads();
  if (wid == 0) {
    const int v = lane < kWarps ? s_warp[lane] : 0;
    int t;
    const int vp = warp_excl_scan(v, &t);
    if (lane < kWarps) s_warp[lane] = vp;
    if (lane == 0) s_warp[kWarps] = t;
  }
  __syncthreads();
  const int r = s_warp[wid] + pre;
  *total = s_warp[kWarps];
  __syncthreads();  // s_warp is reused by the next call
  return r;
}

// Sec. 3.1 without its reuse (the ablation BC_NO_CD_REUSE): before the backward sweep first reads
// the degree prefix CD of level d's entries Q[q0, q1), it is scanned again instead of taken
// from the forward appends.  CTAs sum the degrees of equal chunks of the level, then each
// scans its chunk starting from E0 plus the sums of the CTAs before it.  The values equal
// the stored ones (the appends lay entries and their edge offsets out in queue order), so
// only the time differs.  Two grid barriers.
__device__ bool rescan_level(const PK &p, GridSync *gs, int d, int q0, int q1, int E0) {
  __shared__ int s_warp[kWarps + 1];
  __shared__ int s_base;
  const int nb = gridDim.x, b = blockIdx.x;
  const long long len = (long long)q1 - q0;
  const int c0 = q0 + (int)(len * b / nb), c1 = q0 + (int)(len * (b + 1) / nb);
  int part = 0;
  for (int i = c0 + (int)threadIdx.x; i < c1; i += kThreads) {
    const int v = p.Q[i];
    part += p.rp[v + 1] - p.rp[v];
  }
  int tot;
  (void)cta_excl_scan(part, &tot, s_warp);
  if (threadIdx.x == 0) p.ctl->scan_blk[b] = tot;
  if (!phase_sync(p, gs, 8, d)) return false;
  if (threadIdx.x < 32) {
    int acc = 0;
    for (int j = (int)threadIdx.x; j < b; j += 32) acc += ld_volatile_i32(&p.ctl->scan_blk[j]);
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) acc += __shfl_xor_sync(BC_FULL, acc, m);
    if (threadIdx.x == 0) s_base = E0 + acc;
  }
  __syncthreads();
  int base = s_base;
  for (int i0 = c0; i0 < c1; i0 += kThreads) {  // c0, c1 are uniform over the CTA
    const int i = i0 + (int)threadIdx.x;
    int dg = 0;
    if (i < c1) {
      const int v = p.Q[i];
      dg = p.rp[v + 1] - p.rp[v];
    }
    int t;
    const int pre = cta_excl_scan(dg, &t, s_warp);
    if (i < c1) p.CD[i] = base + pre;
    base += t;
  }
  return phase_sync(p, gs, 9, d);
}

// Start of a source: empty bitmaps but for the source's bit, its state, the control words.
__device__ __forceinline__ void start_source(const PK &p, int s, int base, int gtid, int nthr) {
  const int nw = (p.n + 31) / 32;
  for (int i = gtid; i < nw; i += nthr) {
    p.vis[i] = 0u;
    p.ovf[i] = 0u;
    p.lvb[0][i] = i == (s >> 5) ? 1u << (s & 31) : 0u;
    p.lvb[1][i] = 0u;
    p.lvb[2][i] = 0u;
  }
  if (gtid == 0) {
    PlainCtl *ctl = p.ctl;
    const int ds = p.rp[s + 1] - p.rp[s];
    p.depth[s] = base;
    p.sig[s] = 1ull;
    p.Q[0] = s;
    p.CD[0] = 0;
    p.lvl_off[0] = 0;
    p.lvl_off[1] = 1;
    p.lvl_eoff[0] = 0;
    p.lvl_eoff[1] = ds;
    ctl->ns = 0ull;
    ctl->src_ovf = 0;
    for (int k = 0; k < 3; k++) {
      ctl->qpack[k] = 0ull;
      ctl->level_ovf[k] = 0;
      ctl->sigmax[k] = 0ull;
    }
  }
}

// One grid barrier per level of the forward sweep (a second one only where a level passed 2^64 or
// its largest sigma has to be known), two per level of the backward sweep.
// SOLO: the CTA runs every team-th source of the list on a workspace of its own.
template <bool SOLO>
__device__ __forceinline__ void plain_body(const PK &p, unsigned char *smem) {
  __shared__ unsigned long long s_red;
  WarpWin &W = ((WarpWin *)smem)[threadIdx.x >> 5];
  const int gtid = SOLO ? threadIdx.x : blockIdx.x * blockDim.x + threadIdx.x;
  const int nthr = SOLO ? blockDim.x : gridDim.x * blockDim.x;
  const int gwarp = gtid >> 5;
  const int nwarps = nthr >> 5;
  const int nw = (p.n + 31) / 32;
  PlainCtl *ctl = p.ctl;
  GridSync *gs = &ctl->bar;
  const bool sssp = p.out_depth != nullptr;
  int base = p.base;

  for (int si = SOLO ? blockIdx.x : 0; si < p.nsrc; si += SOLO ? gridDim.x : 1) {
    const int s = p.src[si];
    if (SOLO && (s < 0 || s >= p.n)) {
      *p.bad = 1;
      continue;
    }
    if (base > kBaseMax - p.n) {  // depth values near their end: forget all sources before
      for (int v = gtid; v < p.n; v += nthr) p.depth[v] = -1;
      base = 0;
      if (!phase_sync<SOLO>(p, gs, 0, 0)) return;
    }
    start_source(p, s, base, gtid, nthr);
    if (!phase_sync<SOLO>(p, gs, 0, 0)) return;

    // ---------------------------------------------------------------- forward
    int level = 1;
    bool bu = false;
    int q0 = 0, q1 = 1, E0 = 0, E1 = p.rp[s + 1] - p.rp[s];
    double smax = 1.0;  // no sigma of the level before is larger (while none passed 2^64)
    while (true) {
      const int nf = q1 - q0;
      if (nf == 0) break;
      const double mf = (double)(E1 - E0);
      const double mu = (double)(p.nnz - E1);
      if (!bu) {
        if (mf > (double)p.alpha * mu) bu = true;
      } else {
        if ((double)nf * (double)p.beta < (double)p.n && mf < (double)p.alpha * mu) bu = false;
      }
      Lvl L;
      L.level = level;
      L.dv = base + level;
      L.q1 = q1;
      L.E1 = E1;
      L.ctr = &ctl->qpack[level % 3];
      L.ovf = &ctl->level_ovf[level % 3];
      L.povf = *(volatile int *)&ctl->src_ovf != 0;
      L.cur = p.lvb[level % 3];
      L.front = p.lvb[(level + 2) % 3];
      uint32_t *old = p.lvb[(level + 1) % 3];  // level - 2: already in vis, the next level's
      for (int i = gtid; i < nw; i += nthr) {
        const uint32_t f = L.front[i];
        if (f) p.vis[i] |= f;  // readers test vis and front, so either value serves them
        if (old[i]) old[i] = 0u;
      }
      if (gtid == 0) {
        ctl->qpack[(level + 1) % 3] = 0ull;
        ctl->level_ovf[(level + 1) % 3] = 0;
        ctl->sigmax[(level + 1) % 3] = 0ull;
      }
      if (bu) {
        sweep_bottomup(p, L, gwarp, nwarps);
      } else {
        // no 64-bit carry is possible this level if max sigma * max degree < 2^64
        const bool fast = !L.povf && smax * (double)p.max_degree < 1.8e19;
        expand_topdown(p, W, L, q0, E0, gwarp, nwarps, fast);
      }
      if (!phase_sync<SOLO>(p, gs, bu ? 2 : 1, level)) return;

      const unsigned long long pk = *(volatile unsigned long long *)L.ctr;
      const int q2 = q1 + (int)(pk >> 32);
      const bool lvl_ovf = *(volatile int *)L.ovf != 0;
      // the level's largest sigma: bounded by the parents', read only where the bound would
      // keep the next level from the carry-free additions
      smax *= (double)p.max_degree;
      const bool scan = smax * (double)p.max_degree >= 1.8e19 && *(volatile int *)&ctl->src_ovf == 0;
      if ((lvl_ovf || scan) && q2 > q1) {
        if (threadIdx.x == 0) s_red = 0ull;
        __syncthreads();
        unsigned long long mx = 0;
        for (int i = q1 + gtid; i < q2; i += nthr) {
          const int w = p.Q[i];
          const unsigned long long sw = p.sig[w];
          mx = sw > mx ? sw : mx;
          if (lvl_ovf && test_bit(p.ovf, w)) ext_sigma(p, w, base + level - 1);
        }
        if (mx) atomicMax(&s_red, mx);
        __syncthreads();
        if (threadIdx.x == 0 && s_red) atomicMax(&ctl->sigmax[level % 3], s_red);
        if (!phase_sync<SOLO>(p, gs, 3, level)) return;
        smax = (double)*(volatile unsigned long long *)&ctl->sigmax[level % 3];
      }
      q0 = q1;
      q1 = q2;
      E0 = E1;
      E1 += (int)(pk & 0xffffffffull);
      if (gtid == 0) {
        p.lvl_off[level + 1] = q1;
        p.lvl_eoff[level + 1] = E1;
      }
      level++;
    }
    const int D = level - 2;   // deepest non-empty level
    const int qtot = q1;       // reached vertices

    if (sssp) {
      for (int v = gtid; v < p.n; v += nthr) {
        const int d = p.depth[v];
        p.out_depth[v] = d >= base ? d - base : -1;
        p.out_sigma[v] = p.sig[v];
        p.out_ovf[v] = test_bit(p.ovf, v) ? 1 : 0;
        p.sig[v] = 0ull;
      }
    } else {
      // -------------------------------------------------------------- backward
      const bool ext = *(volatile int *)&ctl->src_ovf != 0;
      const double ws = p.omega ? (double)p.omega[s] + 1.0 : 1.0;
      const bool leaf = p.leaf_term && p.omega && p.omega[s] > 0;
      if (leaf && D >= 1) {  // n_s of Eq. 3
        if (threadIdx.x == 0) s_red = 0ull;
        __syncthreads();
        unsigned long long part = 0;
        for (int i = gtid; i < qtot; i += nthr) part += 1ull + (unsigned long long)p.omega[p.Q[i]];
        if (part) atomicAdd(&s_red, part);
        __syncthreads();
        if (threadIdx.x == 0 && s_red) atomicAdd(&ctl->ns, s_red);
      }
      if (D >= 1) {
        // level offsets: written by one thread before a barrier each, or held in registers
        int a0 = p.lvl_off[D], a1 = qtot, f0 = p.lvl_eoff[D], f1 = E1;
        if (ext)
          finalize_level<true>(p, a0, a1, ws, gtid, nthr);
        else
          finalize_level<false>(p, a0, a1, ws, gtid, nthr);
        if (!phase_sync<SOLO>(p, gs, 4, D)) return;
        bool pulled = false;
        for (int d = D - 1; d >= 1; --d) {
          const int b0 = p.lvl_off[d], b1 = a0, g0 = p.lvl_eoff[d], g1 = f0;
          // a pushed arc that leads back costs its own atomics, so push only from far fewer arcs
          const bool push = (long long)(f1 - f0) * kPushFactor <= (long long)(g1 - g0);
          // the prefix that this step reads: the next level's when it pushes, unless the step before
          // pulled and so had it scanned
          if (!SOLO && p.no_cd_reuse && !(push && pulled) &&
              !rescan_level(p, gs, push ? d + 1 : d, push ? a0 : b0, push ? a1 : b1, push ? f0 : g0))
            return;
          pulled = !push;
          if (push) {
            if (ext)
              push_level<true>(p, W, base + d, a0, a1, f0, f1, gwarp, nwarps);
            else
              push_level<false>(p, W, base + d, a0, a1, f0, f1, gwarp, nwarps);
          } else {
            if (ext)
              accumulate_level<true>(p, W, base + d + 1, b0, b1, g0, g1, gwarp, nwarps);
            else
              accumulate_level<false>(p, W, base + d + 1, b0, b1, g0, g1, gwarp, nwarps);
          }
          if (!phase_sync<SOLO>(p, gs, 5, d)) return;
          if (ext)
            finalize_level<true>(p, b0, b1, ws, gtid, nthr);
          else
            finalize_level<false>(p, b0, b1, ws, gtid, nthr);
          if (!phase_sync<SOLO>(p, gs, 6, d)) return;
          a0 = b0;
          a1 = b1;
          f0 = g0;
          f1 = g1;
        }
      }
      if (gtid == 0) {
        if (leaf) {
          double om = (double)p.omega[s];
          double ns = D >= 1 ? (double)*(volatile unsigned long long *)&ctl->ns : 1.0 + om;
          p.bc[s] += om * (2.0 * ns - om - 3.0);
        }
        p.sig[s] = 0ull;
      }
    }
    if (gtid == 0) {
      if (*(volatile int *)&ctl->src_ovf) ctl->ovf_sources++;
      ctl->levels += level - 1;
      ctl->reached += qtot;
      ctl->reached_arcs += E1;
      if (D > ctl->max_depth) ctl->max_depth = D;
    }
    base += D + 2;
    // the next source's start overwrites what the phase after the last barrier may still read
    if ((sssp || D == 0) && !phase_sync<SOLO>(p, gs, 7, 0)) return;
  }
  if (gtid == 0) ctl->base = base;
}

__global__ void __launch_bounds__(kThreads, 1) plain_kernel(PK p) {
  extern __shared__ __align__(16) unsigned char smem[];
  plain_body<false>(p, smem);
}

// Team t's workspace lies t * stride bytes behind team 0's (p); it is cleared here.
__global__ void __launch_bounds__(kThreads, 1) plain_solo(PK p, size_t stride) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ PK q;
  if (threadIdx.x == 0) {
    q = p;
    const size_t o = stride * blockIdx.x;
    auto move = [&](auto *&x) { x = (std::remove_reference_t<decltype(x)>)((char *)x + o); };
    move(q.depth);
    move(q.Q);
    move(q.CD);
    move(q.lvl_off);
    move(q.lvl_eoff);
    move(q.sig);
    move(q.ovf);
    move(q.vis);
    for (int k = 0; k < 3; k++) move(q.lvb[k]);
    move(q.acc);
    move(q.r);
    move(q.xm);
    move(q.xe);
    move(q.ctl);
    move(q.bc);
  }
  __syncthreads();
  for (int v = threadIdx.x; v < p.n; v += blockDim.x) {
    q.depth[v] = -1;
    q.sig[v] = 0ull;
    q.acc[2 * v] = 0ull;
    q.acc[2 * v + 1] = 0ull;
    q.xe[v] = 0;
    q.bc[v] = 0.0;
  }
  for (int i = threadIdx.x; i < (int)(sizeof(PlainCtl) / 4); i += blockDim.x) ((uint32_t *)q.ctl)[i] = 0u;
  __syncthreads();
  plain_body<true>(q, smem);
}

// The dynamic shared-memory size of plain_kernel is an attribute of the function on one
// device: it is set on each device before that device's first launch.
std::mutex g_setup_mu;
bool g_setup_done[128];

bc_status plain_setup(int *blocks_per_sm) {
  int dev = 0;
  BC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 128) return fail(BC_EINVAL, "per-source kernel: device index out of range");
  std::lock_guard<std::mutex> lk(g_setup_mu);
  if (!g_setup_done[dev]) {
    BC_CUDA_TRY(cudaFuncSetAttribute(plain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemBytes));
    BC_CUDA_TRY(cudaFuncSetAttribute(plain_solo, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemBytes));
    int b = 0;
    BC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, plain_kernel, kThreads, kSmemBytes));
    if (b < 1) return fail(BC_ECUDA, "per-source kernel does not fit on an SM");
    g_setup_done[dev] = true;
  }
  *blocks_per_sm = 1;  // one CTA of 1024 threads per SM
  return BC_OK;
}

}  // namespace

int64_t plain_bytes(int32_t n) {
  int64_t N = n + 2, nw = (n + 31) / 32 + 1;
  return N * (4 * 5 + 8 * 6) + nw * 4 * 3 + (int64_t)sizeof(PlainCtl) + 4032;
}

void plain_free(Ctx *ctx, PlainWS *ws) {
  if (!ws->ctl) return;
  void *ptrs[] = {ws->depth, ws->Q, ws->CD, ws->lvl_off, ws->lvl_eoff, ws->sig, ws->ovf,
                  ws->vis, ws->front, ws->acc, ws->r, ws->xm, ws->xe, ws->ctl};
  for (void *q : ptrs) cudaFree(q);
  ctx->mem.release(nullptr, ws->bytes);
  *ws = PlainWS();
}

static bc_status plain_reset(PlainWS *ws, cudaStream_t st) {
  size_t N = (size_t)ws->n + 2, nw = (size_t)(ws->n + 31) / 32 + 1;
  BC_CUDA_TRY(cudaMemsetAsync(ws->depth, 0xff, N * 4, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->sig, 0, N * 8, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->ovf, 0, nw * 4, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->vis, 0, nw * 4, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->front, 0, nw * 4, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->acc, 0, N * 16, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->xe, 0, N * 4, st));
  BC_CUDA_TRY(cudaMemsetAsync(ws->ctl, 0, sizeof(PlainCtl), st));
  ws->base = 0;
  return BC_OK;
}

bc_status plain_ensure(Ctx *ctx, PlainWS *ws, int32_t n) {
  if (ws->ctl && ws->n == n) return BC_OK;
  plain_free(ctx, ws);
  size_t N = (size_t)n + 2, nw = (size_t)(n + 31) / 32 + 1;
  size_t total = (size_t)plain_bytes(n);
  bc_status s = ctx->mem.alloc(nullptr, total);
  if (s) return s;
  cudaError_t e = cudaSuccess;
#define PA(ptr, bytes) \
  if (e == cudaSuccess) e = cudaMalloc((void **)&ws->ptr, (bytes));
  PA(depth, N * 4) PA(Q, N * 4) PA(CD, N * 4) PA(lvl_off, N * 4) PA(lvl_eoff, N * 4)
  PA(sig, N * 8) PA(ovf, nw * 4) PA(vis, nw * 4) PA(front, nw * 4) PA(acc, N * 16)
  PA(r, N * 8) PA(xm, N * 8) PA(xe, N * 4) PA(ctl, sizeof(PlainCtl))
#undef PA
  ws->n = n;
  ws->bytes = total;
  if (e != cudaSuccess) {
    cudaGetLastError();
    plain_free(ctx, ws);
    return fail(BC_ENOMEM, std::string("device allocation for the per-source workspace failed: ") +
                               cudaGetErrorString(e));
  }
  s = plain_reset(ws, 0);
  if (s) return s;
  BC_CUDA_TRY(cudaStreamSynchronize(0));
  return BC_OK;
}

static PK view_params(const PlainWS &ws, const PlainArgs &a, uint64_t limit_ns) {
  PK p;
  memset(&p, 0, sizeof(p));
  p.n = a.g->n;
  p.nnz = a.g->nnz;
  p.max_degree = a.max_degree;
  p.rp = a.g->rp;
  p.ci = a.g->ci;
  p.omega = a.omega;
  p.src = a.src;
  p.nsrc = a.nsrc;
  p.bc = a.bc;
  p.leaf_term = a.leaf_term ? 1 : 0;
  p.depth = ws.depth;
  p.Q = ws.Q;
  p.CD = ws.CD;
  p.lvl_off = ws.lvl_off;
  p.lvl_eoff = ws.lvl_eoff;
  p.sig = ws.sig;
  p.ovf = ws.ovf;
  p.vis = ws.vis;
  p.lvb[0] = ws.front;
  p.lvb[1] = (uint32_t *)ws.r;
  p.lvb[2] = p.lvb[1] + (a.g->n + 31) / 32;
  p.base = ws.base;
  p.acc = ws.acc;
  p.r = ws.r;
  p.xm = ws.xm;
  p.xe = ws.xe;
  p.ctl = ws.ctl;
  p.out_depth = a.out_depth;
  p.out_sigma = a.out_sigma;
  p.out_ovf = a.out_ovf;
  p.alpha = a.alpha;
  p.beta = a.beta;
  p.limit_ns = limit_ns;
  p.no_cd_reuse = a.no_cd_reuse ? 1 : 0;
  return p;
}

// Launch the per-source kernel on a workspace whose arrays the caller has already laid
// out (and cleared: depth -1; sigma, acc, exponents and the control block 0).
// Allocates nothing and creates no events; waits for the kernel and reads its error word
// into *dev_err.
bc_status plain_run_view(const PlainWS &ws, const PlainArgs &a, int ctas, uint64_t limit_ns,
                         cudaStream_t st, int *dev_err) {
  *dev_err = 0;
  if (a.nsrc <= 0) return BC_OK;
  int bps = 0;
  bc_status s = plain_setup(&bps);
  if (s) return s;
  PK p = view_params(ws, a, limit_ns);
  void *args[] = {&p};
  cudaError_t le = cudaLaunchCooperativeKernel((void *)plain_kernel, dim3(ctas * bps),
                                               dim3(kThreads), args, kSmemBytes, st);
  if (le != cudaSuccess) return cuda_fail(le, "cudaLaunchCooperativeKernel(plain_kernel)");
  int err = 0;
  BC_CUDA_TRY(cudaMemcpyAsync(&err, &ws.ctl->bar.err, sizeof(int), cudaMemcpyDeviceToHost, st));
  BC_CUDA_TRY(cudaStreamSynchronize(st));
  *dev_err = err;
  return BC_OK;
}

// The same for `teams` CTAs that run different sources, each on a workspace of its own: team t's
// lies t * stride bytes behind ws, with its BC partial (a.bc: team 0's).  Clears the workspaces;
// sets *bad (device) for source ids outside [0, n), which are skipped.  Does not wait.
bc_status plain_launch_solo(const PlainWS &ws, const PlainArgs &a, int teams, size_t stride, int *bad,
                            cudaStream_t st) {
  int bps = 0;
  bc_status s = plain_setup(&bps);
  if (s) return s;
  PK p = view_params(ws, a, 0);
  p.bad = bad;
  plain_solo<<<teams, kThreads, kSmemBytes, st>>>(p, stride);
  BC_CUDA_TRY(cudaGetLastError());
  return BC_OK;
}

bc_status plain_run(Ctx *ctx, PlainWS *ws, const PlainArgs &a, cudaStream_t st, bc_stats *acc) {
  if (a.nsrc <= 0) return BC_OK;
  int bps = 0;
  {
    const bc_status s = plain_setup(&bps);
    if (s) return s;
  }
  PK p = view_params(*ws, a, ctx->wait_limit_ns);
  if (a.no_cd_reuse && ctx->num_sms * bps > kPlainScanBlocks)
    return fail(BC_EINVAL, "BC_NO_CD_REUSE: more CTAs than the rescan supports");
  static const char *trace_file = getenv("BC_TRACE_FILE");
  if (trace_file) {
    p.trace_cap = 1 << 20;
    if (cudaMalloc(&p.trace, (size_t)p.trace_cap * 16) != cudaSuccess) {
      cudaGetLastError();
      p.trace = nullptr;
      p.trace_cap = 0;
    }
  }
  dim3 grid(ctx->num_sms * bps), block(kThreads);
  void *args[] = {&p};
  BC_CUDA_TRY(cudaMemsetAsync(ws->ctl, 0, sizeof(PlainCtl), st));
  cudaEvent_t e0, e1;
  BC_CUDA_TRY(cudaEventCreate(&e0));
  BC_CUDA_TRY(cudaEventCreate(&e1));
  BC_CUDA_TRY(cudaEventRecord(e0, st));
  cudaError_t le =
      cudaLaunchCooperativeKernel((void *)plain_kernel, grid, block, args, kSmemBytes, st);
  if (le != cudaSuccess) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return cuda_fail(le, "cudaLaunchCooperativeKernel(plain_kernel)");
  }
  BC_CUDA_TRY(cudaEventRecord(e1, st));
  PlainCtl h;
  BC_CUDA_TRY(cudaMemcpyAsync(&h, ws->ctl, sizeof(PlainCtl), cudaMemcpyDeviceToHost, st));
  BC_CUDA_TRY(cudaStreamSynchronize(st));
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (p.trace) {
    int cnt = h.trace_n < p.trace_cap ? h.trace_n : p.trace_cap;
    std::vector<unsigned long long> t((size_t)cnt * 2);
    cudaMemcpy(t.data(), p.trace, (size_t)cnt * 16, cudaMemcpyDeviceToHost);
    cudaFree(p.trace);
    if (FILE *f = fopen(trace_file, "a")) {
      for (int i = 0; i < cnt; i++)
        fprintf(f, "%d,%d,%llu\n", (int)(t[2 * i] >> 56), (int)((t[2 * i] >> 24) & 0xffffffffull),
                t[2 * i + 1]);
      fclose(f);
    }
  }
  if (h.bar.err != 0) {
    bc_status r = plain_reset(ws, st);
    cudaStreamSynchronize(st);
    if (r) return r;
    if (h.bar.err == BCD_TIMEOUT)
      return fail(BC_ETIMEDOUT, "per-source kernel: a grid barrier wait passed its limit");
    return fail(BC_ECUDA, "per-source kernel reported device error " + std::to_string(h.bar.err));
  }
  ws->base = h.base;
  if (acc) {
    acc->seconds += ms * 1e-3;
    acc->sources += a.nsrc;
    acc->sigma_overflow_sources += h.ovf_sources;
    acc->levels += h.levels;
    acc->kernel_launches += 1;
    acc->reached_vertices += h.reached;
    acc->reached_arcs += h.reached_arcs;
    if (h.max_depth > acc->max_depth) acc->max_depth = h.max_depth;
    if (acc->tile_width == 0) acc->tile_width = 1;
  }
  return BC_OK;
}

}  // namespace bcl

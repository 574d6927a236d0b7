// Per-source path, one source per CTA: every CTA runs whole sources on its own.
//
// The method is Brandes' (Alg. 1) with the level-synchronous forward sweep of Alg. 2 /
// Alg. 3 and the successor-checking backward sweep of Alg. 4 / Alg. 5, one source at a
// time.  On a graph of a few thousand vertices a level holds far too little work for the
// whole GPU, and on a road network a level is a ring of a few hundred vertices; grid-wide
// barriers would dominate both.  Here the loop over sources of Alg. 1 is spread over the CTAs
// (the coarse-grained parallelism of Sec. 3.3, applied to the SMs of one GPU): a CTA takes
// sources blockIdx.x, blockIdx.x + gridDim.x, ... and runs each with CTA barriers only, one
// barrier per level and sweep.
//
// What bounds it: dependent memory round trips of a level (a queue entry, its row, the states
// of its neighbours) and L2 transactions.  So a vertex's state is one 16-byte record, read
// with one load: its value (forward: sigma; backward: r, which replaces it), its level, its
// exponent.  Small graphs keep value, level and queue in shared memory instead.
//
// Forward pass l handles the entries w of level l, once per arc: neighbours of level l - 1 are
// parents, their sigma is summed (a pull in arc order: no sigma atomics, and the extended
// range needs no pass of its own); neighbours not reached yet are claimed for level l + 1 by
// an atomic maximum on their level and queued.  The levels carry the source's base, which
// grows by the levels used, so records of earlier sources read as "not reached" and nothing is
// reset between sources.  With state in global memory a queue entry notes which of the first eight
// arcs of a row handled by a lane lead to successors, so the backward sweep leaves the others' records alone.
// Backward level d: a vertex sums its successors' r in float-float arithmetic, delta = sigma *
// sum, r = (1 + omega) / sigma + sum, and the CTA's BC partial grows by (omega[s] + 1) * delta.
// When a sigma of the source passed 2^64 sigma is taken as m 2^e (m in [0.5, 1)) and r is kept
// scaled by 2^e; other sources need no exponents.  A second kernel sums the partials in CTA
// order.  Every sum has a fixed order (how a vertex is handled depends on its degree only), so
// the result repeats bit for bit from run to run.
#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>
#include <vector>

#include "bc_ff.cuh"
#include "bc_internal.h"

namespace bcl {

namespace {

constexpr int kRing = 2048;     // entries of a level kept in shared memory (state in global memory)
constexpr int kThin = 4;        // degree up to which a row record holds the neighbours themselves
constexpr int kGroupDeg = 32;   // above a lane's degree: eight lanes up to here, a warp beyond
constexpr int kNarrowDeg = 8;   // graphs of at most this degree: lanes alone (no code for larger rows)
constexpr uint32_t kBase0 = 2;  // first base: level base - 1 is never in use, nor 0
constexpr uint32_t kBaseMax = 0x3f000000u;
// Queue entries: vertex id (n <= 2^24), above it a bit for each of the row's first eight arcs that leads
// to a successor.  No entry may equal -1, the mark of a missing one, whatever its id: in narrow
// graphs one of a row's arcs, at most eight, leads to a parent; else the eighth arc's bit stays clear
// and its record is always read.
constexpr int kIdMask = 0xffffff;
template <int LD>
constexpr bool kSeven = LD > kNarrowDeg;
constexpr size_t kCtaSmemMax = 224 * 1024;  // state kept in shared memory up to this

struct CtaK {
  int n;
  const int32_t *__restrict__ rp;
  const int32_t *__restrict__ ci;
  const int4 *__restrict__ row4;  // row records (k_cta_rows), or null: read rp and ci
  const int32_t *__restrict__ omega;
  const int32_t *__restrict__ src;
  int nsrc;
  int leaf_term;
  int spread;         // a level's consecutive entries go to different warps (see cta_slot)
  double *bcp;        // [gridDim.x][n] per-CTA BC partials
  char *gws;          // per-CTA global slices
  size_t slice;       // bytes per slice
  int clean;          // slices hold a valid base and records (left so by the last call)
  unsigned long long *stats;  // reached pairs, their arcs, levels, deepest level (max),
                              // sources whose sigma passed 2^64
  const int32_t *tri;         // 2-degree triples (a, b, c), 3 ints each
  int ntri;
  int32_t *out_depth;         // forward-only export of src[0] (sssp), or null
  unsigned long long *out_sigma;
  uint8_t *out_ovf;
  // several requests in one launch (nreq > 0): request q owns the sources
  // [req[q], req[q + 1]) and the CTAs [req[R + q], req[R + q + 1]), R = nreq + 1
  int nreq;
  const int32_t *req;
};

// One vertex of one source, state in global memory.  tag: (base + level) << 1, low bit set once
// sigma passed 2^64; below base << 1: not reached by this source.  val: sigma modulo 2^64, or
// the extended range's mantissa (with exponent e); after the vertex's backward step r (float2).
struct __align__(16) Rec {
  unsigned long long val;
  uint32_t tag;
  int32_t e;
};

__host__ __device__ inline size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }
// Global slice of a CTA: bases | records | queue | level offsets (state in shared memory:
// exponents | level offsets | queue); with triples a second state and c's records.
__host__ __device__ inline size_t cta_state_bytes(int n, bool sm) {
  return (sm ? al16((size_t)n * 4) + al16((size_t)n * 2) : (size_t)n * 16 + al16((size_t)n * 4)) +
         al16(((size_t)n + 2) * 4);
}
// Shared-memory state, n < 32768 (levels and ids in 16 bits): val u64 | tag u16 (level << 1, low
// bit: sigma passed 2^64, 0xffff: not reached) | reached bits | queue u16 (in the slice when it
// does not fit).  Cleared per source.
__host__ __device__ inline size_t cta_smem_bytes(int n, bool with_q) {
  return al16((size_t)n * 8) + (with_q ? 2 : 1) * al16((size_t)n * 2) + al16(((size_t)n + 31) / 32 * 4);
}
__host__ __device__ inline bool cta_smem_q(int n) { return cta_smem_bytes(n, true) <= kCtaSmemMax; }
constexpr uint32_t kSmFree = 0xffffu;

template <bool SM>
struct CtaState {  // state in global memory
  Rec *rec;
  int32_t *Q;
  int32_t *loff;  // level offsets into Q
  uint32_t base;
};
template <>
struct CtaState<true> {  // state in shared memory
  unsigned long long *val;
  uint16_t *tag, *Q;
  uint32_t *vis;
  int32_t *e;     // global memory, valid for sources with overflow
  int32_t *loff;  // global memory
};

template <bool SM>
__device__ __forceinline__ CtaState<SM> cta_carve(char *smem, char *g, int n) {
  CtaState<SM> S;
  if constexpr (SM) {
    S.val = (unsigned long long *)smem;
    smem += al16((size_t)n * 8);
    S.tag = (uint16_t *)smem;
    smem += al16((size_t)n * 2);
    S.vis = (uint32_t *)smem;
    smem += al16(((size_t)n + 31) / 32 * 4);
    S.e = (int32_t *)g;
    S.loff = (int32_t *)(g + al16((size_t)n * 4));
    S.Q = cta_smem_q(n) ? (uint16_t *)smem : (uint16_t *)(g + al16((size_t)n * 4) + al16(((size_t)n + 2) * 4));
  } else {
    S.rec = (Rec *)g;
    S.Q = (int32_t *)(g + (size_t)n * 16);
    S.loff = (int32_t *)(g + (size_t)n * 16 + al16((size_t)n * 4));
    S.base = kBase0;
  }
  return S;
}

// Nothing reached: every tag free (shared memory), or below the first base.
__device__ __forceinline__ void cta_clear(CtaState<true> &S, int n) {
  for (int i = threadIdx.x; i < (int)(al16((size_t)n * 2) / 16); i += blockDim.x)
    ((uint4 *)S.tag)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  for (int i = threadIdx.x; i < (n + 31) / 32; i += blockDim.x) S.vis[i] = 0u;
}
__device__ __forceinline__ void cta_clear(CtaState<false> &S, int n) {
  for (int v = threadIdx.x; v < n; v += blockDim.x) S.rec[v].tag = 0u;
  S.base = kBase0;
}

struct CtaShared {
  int cnt[3];  // entries appended to level l (slot l % 3)
  int ovf;
  unsigned long long ns;
  // statistics of the CTA's sources
  unsigned long long arcs, reached, levels, deepest, ovf_sources;
};

// row4[v] = the neighbours of v (-1 past the last) or, above kThin arcs, {-2, first arc, degree, 0}:
// one 16-byte load instead of the row offsets and then the arcs.
__global__ void k_cta_rows(int n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci, int4 *row4) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const int a = rp[v], d = rp[v + 1] - a;
    int4 q = make_int4(-2, a, d, 0);
    if (d <= kThin)
      q = make_int4(d > 0 ? ci[a] : -1, d > 1 ? ci[a + 1] : -1, d > 2 ? ci[a + 2] : -1, d > 3 ? ci[a + 3] : -1);
    row4[v] = q;
  }
}

// A vertex's row: its degree, where its arcs start, and up to kThin neighbours (then e0 is unused).
struct Row {
  int deg, e0;
  int4 nb;
};
template <bool SM>
__device__ __forceinline__ Row cta_row(const CtaK &p, int v) {
  Row r;
  if (!SM && p.row4) {
    r.nb = p.row4[v];
    r.e0 = r.nb.y;
    r.deg = r.nb.x == -2 ? r.nb.z : (r.nb.x >= 0) + (r.nb.y >= 0) + (r.nb.z >= 0) + (r.nb.w >= 0);
  } else {
    r.e0 = p.rp[v];
    r.deg = p.rp[v + 1] - r.e0;
    r.nb = make_int4(-1, -1, -1, -1);
    if (!SM && r.deg <= kThin) {
      if (r.deg > 0) r.nb.x = p.ci[r.e0];
      if (r.deg > 1) r.nb.y = p.ci[r.e0 + 1];
      if (r.deg > 2) r.nb.z = p.ci[r.e0 + 2];
      if (r.deg > 3) r.nb.w = p.ci[r.e0 + 3];
    }
  }
  return r;
}
__device__ __forceinline__ Row no_row() {
  Row r;
  r.deg = r.e0 = 0;
  r.nb = make_int4(-1, -1, -1, -1);
  return r;
}
// Arcs u .. u + 3 of a row (-1 past lim).
template <bool SM>
__device__ __forceinline__ void row_arcs(const CtaK &p, const Row &r, int u, int lim, int (&x)[4]) {
  if (!SM && r.deg <= kThin) {
    x[0] = r.nb.x;
    x[1] = r.nb.y;
    x[2] = r.nb.z;
    x[3] = r.nb.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; j++) x[j] = u + j < lim ? p.ci[r.e0 + u + j] : -1;
  }
}

// A record of the CTA's own slice, read while other threads of the CTA may raise its tag.
__device__ __forceinline__ Rec ld_rec(const Rec *a) {
  unsigned long long x, y;
  asm volatile("ld.relaxed.cta.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(a) : "memory");
  Rec r;
  r.val = x;
  r.tag = (uint32_t)y;
  r.e = (int32_t)(y >> 32);
  return r;
}
__device__ __forceinline__ void st_rec(Rec *a, const Rec &r) {
  *(ulonglong2 *)a = make_ulonglong2(r.val, (unsigned long long)r.tag | ((unsigned long long)(uint32_t)r.e << 32));
}

// The record of x; from shared memory the value is read only where the tag is one of the
// wanted level's (tag & ~1 == want), and the exponent only with ext.
__device__ __forceinline__ Rec cta_rec(const CtaState<true> &S, int x, uint32_t want, bool ext) {
  Rec r;
  r.tag = *(volatile uint16_t *)&S.tag[x];
  r.val = 0ull;
  r.e = 0;
  if ((r.tag & ~1u) == want) {
    r.val = S.val[x];
    if (ext) r.e = S.e[x];
  }
  return r;
}
__device__ __forceinline__ Rec cta_rec(const CtaState<false> &S, int x, uint32_t, bool) { return ld_rec(S.rec + x); }

// sigma of a record as m 2^e with m in [0.5, 1)
__device__ __forceinline__ XS rec_sigma(const Rec &r) {
  if (r.tag & 1u) {
    XS x;
    x.m = __longlong_as_double((long long)r.val);
    x.e = r.e;
    return x;
  }
  return xs_u64(r.val);
}
__device__ __forceinline__ float2 rec_r(const Rec &r) {
  return make_float2(__uint_as_float((unsigned)r.val), __uint_as_float((unsigned)(r.val >> 32)));
}
__device__ __forceinline__ unsigned long long r_bits(float2 r) {
  return (unsigned long long)__float_as_uint(r.x) | ((unsigned long long)__float_as_uint(r.y) << 32);
}

// Which entry of a window of blockDim.x a thread takes: its own index, or (spread) consecutive
// entries in different warps.  Graphs with rows beyond kThin spread, so that a few large rows
// next to each other in the queue do not fall to one warp; others fill whole warps.
__device__ __forceinline__ int cta_slot(const CtaK &p) {
  const int tid = threadIdx.x;
  return p.spread ? (tid & 31) * (int)(blockDim.x >> 5) + (tid >> 5) : tid;
}

// Rows beyond LD, one per lane of mask m, are taken 32 / W at a time by W lanes each.
// group_take: the lane whose row this lane's group takes next (-1: none left); group_give: the
// owners' copies of their group's value (rank: the owner's number among this batch's).
template <int W>
__device__ __forceinline__ int group_take(unsigned m) {
  if constexpr (W == 32) {
    return __ffs(m) - 1;
  } else {
    int mine = -1;
#pragma unroll
    for (int k = 0; k < 32 / W; k++) {
      if (m && (int)lane_id() / W == k) mine = __ffs(m) - 1;
      m &= m - 1;
    }
    return mine;
  }
}
template <int W>
__device__ __forceinline__ unsigned group_drop(unsigned m) {
#pragma unroll
  for (int k = 0; k < 32 / W; k++) m &= m - 1;
  return m;
}

// ------------------------------------------------------------------ forward
// What a forward pass needs besides the graph and the state.
struct FwdLevel {
  uint32_t t0, tl;  // tags of level 0 and of this level (low bit clear)
  int q1;           // queue position of the next level's first entry
  int *cnt;         // its entries so far
  int32_t *ring;    // state in global memory: its first kRing entries
};
template <bool SM>
__device__ __forceinline__ bool unreached(const FwdLevel &f, uint32_t tag) {
  return SM ? tag == kSmFree : tag < f.t0;
}

// Append the flagged lanes' vertices to the next level (one shared atomic per warp).
__device__ __forceinline__ void fwd_put(const CtaState<true> &S, const FwdLevel &f, int pos, int x) {
  S.Q[f.q1 + pos] = (uint16_t)x;
}
__device__ __forceinline__ void fwd_put(const CtaState<false> &S, const FwdLevel &f, int pos, int x) {
  if (pos < kRing)
    f.ring[pos] = x;
  else
    S.Q[f.q1 + pos] = x;
}
template <bool SM, int K>
__device__ __forceinline__ void fwd_append(const CtaState<SM> &S, const FwdLevel &f, const bool (&nw)[K],
                                           const int (&x)[K]) {
  unsigned m[K];
  int tot = 0;
#pragma unroll
  for (int k = 0; k < K; k++) {
    m[k] = __ballot_sync(BC_FULL, nw[k]);
    tot += __popc(m[k]);
  }
  if (!tot) return;
  int base = 0;
  if (lane_id() == 0) base = atomicAdd(f.cnt, tot);
  base = __shfl_sync(BC_FULL, base, 0);
#pragma unroll
  for (int k = 0; k < K; k++) {
    if (nw[k]) fwd_put(S, f, base + __popc(m[k] & lanemask_lt()), x[k]);
    base += __popc(m[k]);
  }
}

// Claim the K vertices flagged in un for the next level: nw[k] for the one thread that does.  The
// claims are all on their way before the first answer is looked at (an answer from L2 takes as
// long as the records' loads).
template <int K>
__device__ __forceinline__ void fwd_claim(const CtaState<true> &S, const FwdLevel &f, const bool (&un)[K],
                                          const int (&x)[K], bool (&nw)[K]) {
#pragma unroll
  for (int k = 0; k < K; k++) {
    const uint32_t bit = 1u << (x[k] & 31);
    nw[k] = un[k] && !(atomicOr(&S.vis[x[k] >> 5], bit) & bit);
    if (nw[k]) *(volatile uint16_t *)&S.tag[x[k]] = (uint16_t)(f.tl + 2u);
  }
}
template <int K>
__device__ __forceinline__ void fwd_claim(const CtaState<false> &S, const FwdLevel &f, const bool (&un)[K],
                                          const int (&x)[K], bool (&nw)[K]) {
  uint32_t old[K];
#pragma unroll
  for (int k = 0; k < K; k++) {
    old[k] = ~0u;
    if (un[k]) old[k] = atomicMax(&S.rec[x[k]].tag, f.tl + 2u);
  }
#pragma unroll
  for (int k = 0; k < K; k++) nw[k] = old[k] < f.t0;
}

// Store w's sigma: s modulo 2^64, or (ov: it passed 2^64) its extended range a.
__device__ __forceinline__ void fwd_commit(const CtaState<true> &S, const FwdLevel &f, int w, unsigned long long s,
                                           bool ov, bool xp, const XS &a) {
  if (ov) {
    S.tag[w] = (uint16_t)(f.tl | 1u);
    if (!xp) {
      s = (unsigned long long)__double_as_longlong(a.m);
      S.e[w] = a.e;
    }
  }
  S.val[w] = s;
}
__device__ __forceinline__ void fwd_commit(const CtaState<false> &S, const FwdLevel &f, int w, unsigned long long s,
                                           bool ov, bool xp, const XS &a) {
  if (!ov) {
    S.rec[w].val = s;
    return;
  }
  Rec r;
  r.tag = f.tl | 1u;
  r.val = xp ? s : (unsigned long long)__double_as_longlong(a.m);
  r.e = a.e;
  st_rec(S.rec + w, r);
}

__device__ __forceinline__ void sum_carry(unsigned long long &s, bool &ov, unsigned long long v, bool o) {
  const unsigned long long t = s + v;
  ov = ov || t < s || o;
  s = t;
}

template <bool SM, int W>
__device__ __forceinline__ void fwd_groups(const CtaK &p, const CtaState<SM> &S, const FwdLevel &f, unsigned m,
                                           const Row &row, unsigned long long &sum, bool &ovf) {
  constexpr int UN = SM ? 2 : 4;  // arcs of a lane in flight
  const int lane = lane_id(), sub = lane & (W - 1);
  const uint32_t tp = f.tl - 2u;
  while (m) {
    const int src = group_take<W>(m);
    const int ee = __shfl_sync(BC_FULL, row.e0, src < 0 ? 0 : src);
    int dg = __shfl_sync(BC_FULL, row.deg, src < 0 ? 0 : src);
    if (src < 0) dg = 0;
    const int steps = W == 32 ? dg : (int)__reduce_max_sync(BC_FULL, (unsigned)dg);
    unsigned long long s = 0ull;
    bool ov = false;
    for (int u = 0; u < steps; u += W * UN) {
      int x[UN];
      bool nw[UN], un[UN];
#pragma unroll
      for (int k = 0; k < UN; k++) x[k] = u + k * W + sub < dg ? p.ci[ee + u + k * W + sub] : -1;
      Rec r[UN];
#pragma unroll
      for (int k = 0; k < UN; k++) {
        r[k].tag = f.tl;  // neither a parent nor unreached
        if (x[k] >= 0) r[k] = cta_rec(S, x[k], tp, false);
      }
#pragma unroll
      for (int k = 0; k < UN; k++) un[k] = unreached<SM>(f, r[k].tag);
      fwd_claim(S, f, un, x, nw);
#pragma unroll
      for (int k = 0; k < UN; k++)
        if ((r[k].tag & ~1u) == tp) sum_carry(s, ov, r[k].val, r[k].tag & 1u);
      fwd_append<SM, UN>(S, f, nw, x);
    }
#pragma unroll
    for (int o = W / 2; o >= 1; o >>= 1) sum_carry(s, ov, __shfl_xor_sync(BC_FULL, s, o), false);
    const unsigned om = __ballot_sync(BC_FULL, ov);
    // to the owners: the k-th set bit of m took group k's sum
    const int k = __popc(m & lanemask_lt());
    const unsigned long long sk = __shfl_sync(BC_FULL, s, (k * W) & 31);
    if (((m >> lane) & 1u) && k < 32 / W) {
      sum = sk;
      ovf = W == 32 ? om != 0u : ((om >> (k * W)) & ((1u << (W & 31)) - 1u)) != 0u;
    }
    m = group_drop<W>(m);
  }
}

// Extended-range sigma of the lanes' vertices with ov (rows beyond kThin, or not in registers any
// more): the sum over the parents in arc order; rows beyond LD by whole warps, lanes in arc
// order and a fixed-order reduction.
template <bool SM, int LD>
__device__ __noinline__ XS fwd_extended(const CtaK &p, CtaState<SM> S, Row row, uint32_t tp, bool ext, bool ov) {
  XS a;
  a.m = 0.0;
  a.e = 0;
  const int lane = lane_id();
  if (ov && row.deg <= LD) {
    for (int u = 0; u < row.deg; u += 4) {
      int x[4];
      row_arcs<SM>(p, row, u, row.deg, x);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        if (x[j] < 0) continue;
        const Rec r = cta_rec(S, x[j], tp, ext);
        if ((r.tag & ~1u) == tp) xs_add(a, rec_sigma(r));
      }
    }
  }
  unsigned m = LD > kNarrowDeg ? __ballot_sync(BC_FULL, ov && row.deg > LD) : 0u;
  while (m) {
    const int src = __ffs(m) - 1;
    m &= m - 1;
    const int ee = __shfl_sync(BC_FULL, row.e0, src), dg = __shfl_sync(BC_FULL, row.deg, src);
    XS b;
    b.m = 0.0;
    b.e = 0;
    for (int u = lane; u < dg; u += 32) {
      const Rec r = cta_rec(S, p.ci[ee + u], tp, ext);
      if ((r.tag & ~1u) == tp) xs_add(b, rec_sigma(r));
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      XS c;
      c.m = __shfl_xor_sync(BC_FULL, b.m, o);
      c.e = __shfl_xor_sync(BC_FULL, b.e, o);
      xs_add(b, c);
    }
    if (lane == src) a = b;
  }
  return xs_norm(a);
}

// Forward sweep from s (Alg. 2 / Alg. 3, one CTA barrier per level).  Returns the deepest
// non-empty level; *qtot = reached vertices.
template <bool SM, int LD>
__device__ __forceinline__ int cta_forward(const CtaK &p, const CtaState<SM> &S, int s, CtaShared &sh,
                                           int32_t (*ring)[kRing], int *qtot) {
  const int tid = threadIdx.x, slot = cta_slot(p);
  const bool xp = p.out_depth != nullptr;
  FwdLevel f;
  if constexpr (SM)
    f.t0 = 0u;
  else
    f.t0 = S.base << 1;
  f.tl = f.t0;
  bool ext = false;  // some sigma of this source passed 2^64
  __syncthreads();   // the previous source is done with the state and the counters
  if (tid == 0) {
    if constexpr (SM) {
      S.val[s] = 1ull;
      S.tag[s] = 0;
      S.vis[s >> 5] |= 1u << (s & 31);
      S.Q[0] = (uint16_t)s;
    } else {
      Rec r;
      r.val = 1ull;
      r.tag = f.t0;
      r.e = 0;
      st_rec(S.rec + s, r);
      ring[0][0] = s;
    }
    S.loff[0] = 0;
    S.loff[1] = 1;
    sh.cnt[1] = 0;
    sh.ovf = 0;
  }
  __syncthreads();
  int q0 = 0, q1 = 1, l = 0;
  unsigned arcs = 0;  // of the vertices this thread took (nnz < 2^31)
  int c1 = 1, c2 = 2, c0 = 0;  // counter slots of levels l + 1, l + 2, l
  for (;;) {
    const uint32_t tp = f.tl - 2u, tn = f.tl + 2u;
    f.ring = SM ? nullptr : ring[(l + 1) & 1];
    f.q1 = q1;
    f.cnt = &sh.cnt[c1];
    if (tid == 0) sh.cnt[c2] = 0;
    for (int b = q0; b < q1; b += blockDim.x) {
      const int i = b + slot;
      const bool in = i < q1;
      if (!__any_sync(BC_FULL, in)) continue;
      int w = 0;
      if (in) w = SM ? (int)S.Q[i] : (i - q0 < kRing ? ring[l & 1][i - q0] : (int)S.Q[i]);
      const Row row = in ? cta_row<SM>(p, w) : no_row();
      arcs += (unsigned)row.deg;
      unsigned long long sum = 0ull;
      bool ov = false;
      XS a;
      a.m = 0.0;
      a.e = 0;
      int succ = 0;
      const int dl = row.deg <= LD ? row.deg : 0;
      for (int u = 0; __any_sync(BC_FULL, u < dl); u += 4) {
        int x[4];
        row_arcs<SM>(p, row, u, dl, x);
        Rec r[4];
        bool nw[4], un[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
          r[j].tag = f.tl;  // neither a parent nor a successor
          if (u < dl && x[j] >= 0) r[j] = cta_rec(S, x[j], tp, ext);
        }
#pragma unroll
        for (int j = 0; j < 4; j++) un[j] = unreached<SM>(f, r[j].tag);
        fwd_claim(S, f, un, x, nw);
        // the parents' sums while the claims are on their way
        bool allx = true;  // every parent is in the extended range
#pragma unroll
        for (int j = 0; j < 4; j++) {
          if (!SM && (un[j] || r[j].tag == tn) && u < 8) succ |= 1 << (u + j);
          if ((r[j].tag & ~1u) == tp) {
            sum_carry(sum, ov, r[j].val, r[j].tag & 1u);
            allx = allx && (r[j].tag & 1u);
          }
        }
        // u == 0: the one step of such a row.  The loop goes on for longer rows of the warp, and a step
        // without parents would leave the sum with the exponent of none.
        if (!SM && u == 0 && ov && !xp && row.deg <= kThin) {
          if (allx) {  // mantissas brought to the largest exponent (exact) and added in arc order
            a.e = INT_MIN;
#pragma unroll
            for (int j = 0; j < 4; j++)
              if ((r[j].tag & ~1u) == tp) a.e = max(a.e, r[j].e);
#pragma unroll
            for (int j = 0; j < 4; j++)
              if ((r[j].tag & ~1u) == tp) a.m += scale2(__longlong_as_double((long long)r[j].val), r[j].e - a.e);
          } else {
#pragma unroll
            for (int j = 0; j < 4; j++)
              if ((r[j].tag & ~1u) == tp) xs_add(a, rec_sigma(r[j]));
          }
          a = xs_norm(a);
        }
        fwd_append<SM, 4>(S, f, nw, x);
      }
      if constexpr (LD > kNarrowDeg) {
        constexpr int GD = LD > kGroupDeg ? LD : kGroupDeg;
        const unsigned mg = __ballot_sync(BC_FULL, row.deg > LD && row.deg <= GD),
                       mw = __ballot_sync(BC_FULL, row.deg > GD);
        if (mg) fwd_groups<SM, 8>(p, S, f, mg, row, sum, ov);
        if (mw) fwd_groups<SM, 32>(p, S, f, mw, row, sum, ov);
      }
      const bool xs = ov && !xp && (SM || row.deg > kThin);
      if (__any_sync(BC_FULL, xs)) {
        const XS y = fwd_extended<SM, LD>(p, S, row, tp, ext, xs);
        if (xs) a = y;
      }
      if (in) {
        if (!SM) S.Q[i] = w | (kSeven<LD> ? succ & 0x7f : succ) << 24;
        if (l > 0) fwd_commit(S, f, w, sum, ov, xp, a);  // the source keeps sigma = 1
        if (ov) sh.ovf = 1;
      }
    }
    __syncthreads();
    const int q2 = q1 + sh.cnt[c1];
    ext = sh.ovf != 0;
    if (tid == 0) S.loff[l + 2] = q2;
    q0 = q1;
    q1 = q2;
    if (q1 == q0) break;
    l++;
    f.tl = tn;
    const int t = c0;
    c0 = c1;
    c1 = c2;
    c2 = t;
  }
  arcs = __reduce_add_sync(BC_FULL, arcs);
  if (lane_id() == 0 && arcs) atomicAdd(&sh.arcs, (unsigned long long)arcs);
  if (tid == 0) {
    sh.reached += (unsigned long long)q1;
    sh.levels += (unsigned long long)(l + 1);
    if ((unsigned long long)l > sh.deepest) sh.deepest = (unsigned long long)l;
    if (ext) sh.ovf_sources++;
  }
  __syncthreads();  // loff, and everyone has read the counters
  *qtot = q1;
  return l;
}

// ------------------------------------------------------------------ backward
// Rows beyond LD: the sum of the successors' r (rescaled to the owner's exponent ew).
template <bool SM, bool EXT, int W>
__device__ __forceinline__ void bwd_groups(const CtaK &p, const CtaState<SM> &S, unsigned m, const Row &row, int ew,
                                           uint32_t tn, float2 &sum) {
  constexpr int UN = 2;
  const int lane = lane_id(), sub = lane & (W - 1);
  while (m) {
    const int src = group_take<W>(m);
    const int ee = __shfl_sync(BC_FULL, row.e0, src < 0 ? 0 : src);
    int dg = __shfl_sync(BC_FULL, row.deg, src < 0 ? 0 : src);
    const int eo = EXT ? __shfl_sync(BC_FULL, ew, src < 0 ? 0 : src) : 0;
    if (src < 0) dg = 0;
    float2 acc = make_float2(0.0f, 0.0f);
    for (int u = sub; u < dg; u += W * UN) {
      int x[UN];
#pragma unroll
      for (int k = 0; k < UN; k++) x[k] = u + k * W < dg ? p.ci[ee + u + k * W] : -1;
      Rec r[UN];
#pragma unroll
      for (int k = 0; k < UN; k++) {
        r[k].tag = 0u;
        if (x[k] >= 0) r[k] = cta_rec(S, x[k], tn, EXT);
      }
#pragma unroll
      for (int k = 0; k < UN; k++)
        if ((r[k].tag & ~1u) == tn) ff_add(acc, EXT ? ff_scale(rec_r(r[k]), eo - r[k].e) : rec_r(r[k]));
    }
    __syncwarp();
#pragma unroll
    for (int o = W / 2; o >= 1; o >>= 1) ff_add(acc, ff_shfl_xor(acc, o));
    const int k = __popc(m & lanemask_lt());
    const float2 ak = ff_shfl(acc, (k * W) & 31);
    if (((m >> lane) & 1u) && k < 32 / W) sum = ak;
    m = group_drop<W>(m);
  }
}

// Backward sweep of s (Alg. 4 / Alg. 5).  Queue entries, rows and a vertex's own record do not
// depend on the level in progress, so the first window of the next level is loaded before
// the barrier; only the successors' records wait for it.  The BC partial takes a reduction
// without a result: one update per vertex and source, ordered by the barriers between levels.
template <bool SM, int LD, bool EXT>
__device__ __forceinline__ void cta_backward(const CtaK &p, const CtaState<SM> &S, int s, int lmax, double *bcp,
                                             CtaShared &sh) {
  const int tid = threadIdx.x, slot = cta_slot(p);
  const float2 wsrc = ff_u64_bits(1ull + (p.omega ? (unsigned long long)p.omega[s] : 0ull));
  int hi = S.loff[lmax + 1], lo = S.loff[lmax];
  int qe = -1;
  Row row = no_row();
  Rec own;
  own.val = 1ull;
  own.tag = 0u;
  own.e = 0;
  uint32_t tl;
  if constexpr (SM)
    tl = (uint32_t)lmax << 1;
  else
    tl = (S.base + (uint32_t)lmax) << 1;
  auto fetch = [&](int q, uint32_t t) {
    if (q != -1) {
      row = cta_row<SM>(p, q & kIdMask);
      own = cta_rec(S, q & kIdMask, t, EXT);
    } else {
      row.deg = 0;
    }
  };
  if (lmax >= 1 && lo + slot < hi) qe = (int)S.Q[lo + slot];
  fetch(qe, tl);
  int nlo = lmax >= 1 ? S.loff[lmax - 1] : 0;
  for (int dd = lmax; dd >= 1; --dd, tl -= 2u) {
    const uint32_t tn = tl + 2u;
    const int nnlo = dd >= 2 ? S.loff[dd - 2] : 0;
    const int nqe = (dd > 1 && nlo + slot < lo) ? (int)S.Q[nlo + slot] : -1;
    for (int b = lo; b < hi; b += blockDim.x) {
      if (b != lo) {
        qe = b + slot < hi ? (int)S.Q[b + slot] : -1;
        fetch(qe, tl);
      }
      if (!__any_sync(BC_FULL, qe != -1)) continue;
      const int w = qe & kIdMask;
      float2 mw, acc = make_float2(0.0f, 0.0f);
      int ew = 0;
      if (EXT) {
        const XS x = rec_sigma(own);
        mw = ff_mant_bits(x.m);
        ew = x.e;
      } else {
        mw = ff_u64_bits(own.val);
      }
      if (dd < lmax) {
        const int dl = row.deg <= LD ? row.deg : 0;
        const unsigned succ = SM ? 0u : (unsigned)qe >> 24 | (kSeven<LD> ? 0x80u : 0u);
        for (int u = 0; u < dl; u += 4) {
          int x[4];
          row_arcs<SM>(p, row, u, dl, x);
          Rec r[4];
#pragma unroll
          for (int j = 0; j < 4; j++) {
            r[j].tag = 0u;  // not a successor
            if (x[j] >= 0 && (SM || u >= 8 || ((succ >> (u + j)) & 1u))) r[j] = cta_rec(S, x[j], tn, EXT);
          }
#pragma unroll
          for (int j = 0; j < 4; j++)
            if ((r[j].tag & ~1u) == tn) ff_add(acc, EXT ? ff_scale(rec_r(r[j]), ew - r[j].e) : rec_r(r[j]));
        }
        __syncwarp();
        if constexpr (LD > kNarrowDeg) {
          constexpr int GD = LD > kGroupDeg ? LD : kGroupDeg;
          const unsigned mg = __ballot_sync(BC_FULL, row.deg > LD && row.deg <= GD),
                         mb = __ballot_sync(BC_FULL, row.deg > GD);
          if (mg) bwd_groups<SM, EXT, 8>(p, S, mg, row, ew, tn, acc);
          if (mb) bwd_groups<SM, EXT, 32>(p, S, mb, row, ew, tn, acc);
        }
      }
      if (qe != -1) {
        const float2 om1 = ff_u64_bits(1ull + (p.omega ? (unsigned long long)p.omega[w] : 0ull));
        float2 rw = ff_mul(om1, ff_rcp(mw));
        ff_add(rw, acc);
        if constexpr (SM) {
          S.val[w] = r_bits(rw);
          if (EXT) S.e[w] = ew;
        } else if (EXT) {
          own.val = r_bits(rw);
          own.e = ew;
          st_rec(S.rec + w, own);
        } else {
          S.rec[w].val = r_bits(rw);
        }
        const float2 dl = ff_mul(wsrc, ff_mul(mw, acc));
        if (!ff_zero(dl)) atomicAdd(bcp + w, ff_to(dl));
      }
    }
    qe = nqe;
    fetch(qe, tl - 2u);
    __syncthreads();
    hi = lo;
    lo = nlo;
    nlo = nnlo;
  }
  if (tid == 0 && p.leaf_term && p.omega && p.omega[s] > 0) {
    const double om = (double)p.omega[s];
    atomicAdd(bcp + s, om * (2.0 * (double)sh.ns - om - 3.0));
  }
}

// n_s of Eq. 3: the reached vertices Q[0, qtot) weighted by 1 + omega (a source with
// omega(s) > 0 only; the sum is an integer, so its order does not matter).  Ends with a barrier.
template <typename QT>
__device__ __forceinline__ void cta_weighted_size(const CtaK &p, const QT *Q, int qtot, CtaShared &sh) {
  if (threadIdx.x == 0) sh.ns = 0ull;
  __syncthreads();
  unsigned long long part = 0ull;
  for (int i = threadIdx.x; i < qtot; i += blockDim.x) part += 1ull + (unsigned long long)p.omega[(int)Q[i] & kIdMask];
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) part += __shfl_xor_sync(BC_FULL, part, m);
  if ((threadIdx.x & 31) == 0 && part) atomicAdd(&sh.ns, part);
  __syncthreads();
}

// ---- 2-degree vertex c with neighbours a, b (Sec. 3.4.2): its shortest-path DAG follows
// from those of a and b.  For v != c: level_c(v) = 1 + min(level_a(v), level_b(v)) and
// sigma_c(v) = sigma_a(v), sigma_b(v) or their sum as the smaller level comes from a, from b
// or from both (Eq. in Sec. 3.4.2, by the Bellman criterion); level_c(c) = 0, sigma_c(c) = 1.
__device__ __forceinline__ int rec_level(const CtaState<false> &S, const Rec &r) {
  return r.tag < (S.base << 1) ? -1 : (int)((r.tag >> 1) - S.base);
}

// Backward sweep of the 2-degree vertex c on its derived DAG, level by level (the dynamic
// merging of frontiers, Alg. 8 / Alg. 9): c's level D holds the vertices of a's level D - 1
// whose level from b is not smaller, and those of b's level D - 1 whose level from a is
// larger.  C holds c's records as far as the sweep has come: a neighbour is a successor when
// its record carries the level after, so the states of a and b are read for a vertex's own
// sigma only.  EXT (sigma of a or b passed 2^64): r scaled by 2^e of sigma_c.  Runs before the
// backward sweeps of a and b, which replace their sigma.  On a residual graph (1-degree
// reduction) the leaf weights enter as in cta_backward; c, a and b share a component, so the
// weighted component size in sh.ns (set for the triple) is also c's.
template <int LD, bool EXT>
__device__ __forceinline__ void cta_backward_deg2(const CtaK &p, const CtaState<false> &A, const CtaState<false> &B,
                                                  const CtaState<false> &C, int lmaxA, int lmaxB, int c, double *bcp,
                                                  CtaShared &sh) {
  const int lane = lane_id(), slot = cta_slot(p);
  const int lmax = 1 + (lmaxA > lmaxB ? lmaxA : lmaxB);
  const float2 wsrc = ff_u64_bits(1ull + (p.omega ? (unsigned long long)p.omega[c] : 0ull));
  for (int D = lmax; D >= 1; --D) {
    const uint32_t tc = (C.base + (uint32_t)D) << 1, tn = tc + 2u;
#pragma unroll 1
    for (int side = 0; side < 2; side++) {
      if (D - 1 > (side ? lmaxB : lmaxA)) continue;
      const int32_t *Q = side ? B.Q : A.Q, *loff = side ? B.loff : A.loff;
      const int i1 = loff[D];
      for (int b = loff[D - 1]; b < i1; b += blockDim.x) {
        const int i = b + slot;
        const int w = i < i1 ? Q[i] & kIdMask : c;
        bool mine = w != c;
        Row row = no_row();
        float2 mw = make_float2(1.0f, 0.0f);
        int ew = 0;
        if (mine) {
          row = cta_row<false>(p, w);
          const Rec ra = ld_rec(A.rec + w), rb = ld_rec(B.rec + w);
          const int da = rec_level(A, ra), db = rec_level(B, rb);
          // w belongs to c's level D through this side (ties go to a)
          mine = side == 0 ? (db < 0 || da <= db) : (da < 0 || db < da);
          if (EXT) {
            XS x = rec_sigma(side ? rb : ra);
            if (da == db) {
              xs_add(x, rec_sigma(rb));
              x = xs_norm(x);
            }
            mw = ff_mant_bits(x.m);
            ew = x.e;
          } else {
            mw = ff_sum_u64(side ? rb.val : ra.val, da == db ? rb.val : 0ull);
          }
        }
        float2 acc = make_float2(0.0f, 0.0f);
        if (D < lmax) {
          const int dl = mine && row.deg <= LD ? row.deg : 0;
          for (int u = 0; u < dl; u += 4) {
            int x[4];
            row_arcs<false>(p, row, u, dl, x);
            Rec r[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
              r[j].tag = 0u;
              if (x[j] >= 0) r[j] = ld_rec(C.rec + x[j]);
            }
#pragma unroll
            for (int j = 0; j < 4; j++)
              if (r[j].tag == tn) ff_add(acc, EXT ? ff_scale(rec_r(r[j]), ew - r[j].e) : rec_r(r[j]));
          }
          __syncwarp();
          unsigned m = LD > kNarrowDeg ? __ballot_sync(BC_FULL, mine && row.deg > LD) : 0u;
          while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const int ee = __shfl_sync(BC_FULL, row.e0, src), dg = __shfl_sync(BC_FULL, row.deg, src),
                      eo = __shfl_sync(BC_FULL, ew, src);
            float2 t = make_float2(0.0f, 0.0f);
            for (int u = lane; u < dg; u += 32) {
              const Rec r = ld_rec(C.rec + p.ci[ee + u]);
              if (r.tag == tn) ff_add(t, EXT ? ff_scale(rec_r(r), eo - r.e) : rec_r(r));
            }
            __syncwarp();
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) ff_add(t, ff_shfl_xor(t, o));
            if (lane == src) acc = t;
          }
        }
        if (mine) {
          const float2 om1 = ff_u64_bits(1ull + (p.omega ? (unsigned long long)p.omega[w] : 0ull));
          float2 rw = ff_mul(om1, ff_rcp(mw));
          ff_add(rw, acc);
          Rec r;
          r.val = r_bits(rw);
          r.tag = tc;
          r.e = ew;
          st_rec(C.rec + w, r);
          const float2 dl = ff_mul(wsrc, ff_mul(mw, acc));
          if (!ff_zero(dl)) atomicAdd(bcp + w, ff_to(dl));
        }
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && p.leaf_term && p.omega && p.omega[c] > 0) {
    const double om = (double)p.omega[c];
    atomicAdd(bcp + c, om * (2.0 * (double)sh.ns - om - 3.0));
  }
}

// SM: state in shared memory; TRI: 2-degree triples (a second state, both in global memory).
template <bool SM, bool TRI, int MAXT, int LD>
__global__ void __launch_bounds__(MAXT, 1) k_cta_sources(CtaK p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = p.n;
  const int tid = threadIdx.x;
  uint32_t *hdr = (uint32_t *)(p.gws + (size_t)blockIdx.x * p.slice);  // the states' bases
  char *g = (char *)hdr + 16;
  // shared memory: the state, or the ring of the last two levels' entries
  int32_t(*ring)[kRing] = SM ? nullptr : (int32_t(*)[kRing])smem;
  CtaState<SM> A = cta_carve<SM>((char *)smem, g, n);
  CtaState<SM> B = A;  // TRI only
  CtaState<SM> C = A;  // TRI only: c's records
  if constexpr (TRI) {
    B = cta_carve<SM>(nullptr, g + cta_state_bytes(n, false), n);
    C.rec = (Rec *)(g + 2 * cta_state_bytes(n, false));
  }
  double *bcp = p.bcp + (size_t)blockIdx.x * n;
  __shared__ CtaShared sh;

  for (int v = tid; v < n; v += blockDim.x) bcp[v] = 0.0;
  // records of earlier sources and calls read as not reached below the base
  if constexpr (SM) {
    cta_clear(A, n);
  } else {
    if (!p.clean) {
      cta_clear(A, n);
      if (TRI) cta_clear(B, n);
      if (TRI) cta_clear(C, n);
    } else {
      A.base = hdr[0];
      if (TRI) B.base = hdr[1];
      if (TRI) C.base = hdr[2];
    }
  }
  if (tid == 0) sh.arcs = sh.reached = sh.levels = sh.deepest = sh.ovf_sources = 0ull;
  __syncthreads();

  auto done_with = [&](CtaState<SM> &S, int lmax) {
    if constexpr (SM) {
      __syncthreads();
      cta_clear(S, n);
    } else {  // the levels just used are behind the next base
      S.base += (uint32_t)lmax + 2u;
      if (S.base > kBaseMax) {
        __syncthreads();
        cta_clear(S, n);
      }
    }
  };
  int s0 = (int)blockIdx.x, s1 = p.nsrc, sstep = (int)gridDim.x;
  if (!TRI && p.nreq > 0) {  // the sources of this CTA's request, strided over the request's CTAs
    const int32_t *rcta = p.req + p.nreq + 1;
    int q = 0;
    while (q + 1 < p.nreq && (int)blockIdx.x >= rcta[q + 1]) q++;
    s0 = p.req[q] + ((int)blockIdx.x - rcta[q]);
    s1 = p.req[q + 1];
    sstep = rcta[q + 1] - rcta[q];
  }
  if constexpr (!TRI) {
    for (int si = s0; si < s1; si += sstep) {
      const int s = p.src[si];
      int qtot = 0;
      const int lmax = cta_forward<SM, LD>(p, A, s, sh, ring, &qtot);
      if (p.leaf_term && p.omega && p.omega[s] > 0) cta_weighted_size(p, A.Q, qtot, sh);
      if (p.out_depth) {  // forward-only export (sssp of src[0])
        for (int v = tid; v < n; v += blockDim.x) {
          int d = -1;
          unsigned long long x = 0ull;
          uint32_t t;
          if constexpr (SM) {
            t = A.tag[v];
            if (t != kSmFree) {
              d = (int)(t >> 1);
              x = A.val[v];
            }
          } else {
            const Rec r = ld_rec(A.rec + v);
            t = r.tag;
            if (t >= (A.base << 1)) {
              d = (int)((t >> 1) - A.base);
              x = r.val;
            }
          }
          p.out_depth[v] = d;
          p.out_sigma[v] = x;
          p.out_ovf[v] = d >= 0 ? (uint8_t)(t & 1u) : (uint8_t)0;
        }
      } else if (sh.ovf) {
        cta_backward<SM, LD, true>(p, A, s, lmax, bcp, sh);
      } else {
        cta_backward<SM, LD, false>(p, A, s, lmax, bcp, sh);
      }
      done_with(A, lmax);
    }
  } else {
    // single sources, then the 2-degree triples (a, b, c): a and b as usual, c from their two
    // DAGs before their backward sweeps replace sigma by r
    for (int u = blockIdx.x; u < p.nsrc + p.ntri; u += gridDim.x) {
      const bool tri = u >= p.nsrc;
      const int ti = 3 * (u - p.nsrc);
      const int va = tri ? p.tri[ti] : p.src[u], vb = tri ? p.tri[ti + 1] : 0, vc = tri ? p.tri[ti + 2] : 0;
      int la = 0, lb = 0, qtot = 0, xa = 0, xb = 0;
#pragma unroll 1
      for (int k = 0; k <= (int)tri; k++) {
        const int l = cta_forward<SM, LD>(p, k ? B : A, k ? vb : va, sh, ring, &qtot);
        if (k) {
          lb = l;
          xb = sh.ovf;
        } else {
          la = l;
          xa = sh.ovf;
        }
      }
      // a, b and c share a component: one weighted size (of the state run last) serves all three
      if (p.leaf_term && p.omega && (p.omega[va] > 0 || (tri && (p.omega[vb] > 0 || p.omega[vc] > 0))))
        cta_weighted_size(p, tri ? B.Q : A.Q, qtot, sh);
      if (tri) {
        if (xa | xb)
          cta_backward_deg2<LD, true>(p, A, B, C, la, lb, vc, bcp, sh);
        else
          cta_backward_deg2<LD, false>(p, A, B, C, la, lb, vc, bcp, sh);
        done_with(C, 1 + max(la, lb));
      }
#pragma unroll 1
      for (int k = 0; k <= (int)tri; k++) {
        if (k ? xb : xa)
          cta_backward<SM, LD, true>(p, k ? B : A, k ? vb : va, k ? lb : la, bcp, sh);
        else
          cta_backward<SM, LD, false>(p, k ? B : A, k ? vb : va, k ? lb : la, bcp, sh);
      }
      done_with(A, la);
      if (tri) done_with(B, lb);
    }
  }
  __syncthreads();
  if (tid == 0) {
    if constexpr (!SM) {
      hdr[0] = A.base;
      if (TRI) hdr[1] = B.base;
      if (TRI) hdr[2] = C.base;
    }
    atomicAdd(&p.stats[0], sh.reached);
    atomicAdd(&p.stats[1], sh.arcs);
    atomicAdd(&p.stats[2], sh.levels);
    atomicMax(&p.stats[3], sh.deepest);
    if (sh.ovf_sources) atomicAdd(&p.stats[4], sh.ovf_sources);
  }
}

// bc[v] += sum over CTAs c (in order) of bcp[c][v]; sixteen partials in flight at a time
__device__ __forceinline__ double cta_partials(const double *bcp, int c0, int c1, int n, int v) {
  double sum = 0.0;
  int c = c0;
  for (; c + 16 <= c1; c += 16) {
    double x[16];
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = bcp[(size_t)(c + k) * n + v];
#pragma unroll
    for (int k = 0; k < 16; k++) sum += x[k];
  }
  for (; c < c1; c++) sum += bcp[(size_t)c * n + v];
  return sum;
}
__global__ void k_cta_reduce(const double *bcp, int ncta, int n, double *bc) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const double sum = cta_partials(bcp, 0, ncta, n, v);
    if (sum != 0.0) bc[v] += sum;
  }
}

// Several requests: req_bc[q][v] += sum over request q's CTAs c (in order) of bcp[c][v]
// (rc: the requests' CTA ranges, nreq + 1 offsets).
__global__ void k_cta_reduce_req(const double *bcp, int nreq, const int32_t *rc, double *const *req_bc, int n) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    for (int q = 0; q < nreq; q++) {
      const double sum = cta_partials(bcp, rc[q], rc[q + 1], n, v);
      if (sum != 0.0) req_bc[q][v] += sum;
    }
  }
}

}  // namespace

struct CtaWS {
  int n = 0, rows = 0;  // BC partials (CTAs) that bcp holds
  int kind = -1;        // slice layout of the last completed launch: 0 global, 1 shared, 2 triples
  int clean = 0;        // slices (CTAs from 0 on) whose bases and records are valid for that layout
  size_t b_gws = 0;     // bytes of gws, cut into slices of the layout of each launch
  double *bcp = nullptr;
  char *gws = nullptr;
  int4 *row4 = nullptr;  // row records (null: they did not fit the HBM budget)
  unsigned long long *stats = nullptr;
  int32_t *req = nullptr;  // request offsets of a launch with several requests
  size_t bytes = 0;
};

void cta_free(Ctx *ctx, CtaWS *ws) {
  if (!ws) return;
  cudaFree(ws->bcp);
  cudaFree(ws->gws);
  cudaFree(ws->row4);
  cudaFree(ws->stats);
  cudaFree(ws->req);
  ctx->mem.release(nullptr, ws->bytes);
  delete ws;
}

// How a call runs: state in shared memory or not, threads per CTA, CTAs of the whole GPU.
struct CtaPlan {
  int kind = 0, threads = 512, ncta = 0;
  size_t smem = 0;
  const void *kernel = nullptr;
};

// The rule, and both sides of its lines (ms per call, this GPU, a pair on the same code; the grids
// went from 5.5 and 59 to 4.9 and 53 when a level's claims were sent together):
// * State in shared memory where it fits (n <= 22,654): G(n, 4n) n = 16,384, 500 sources 1.15
//   against 1.79 from global memory, social graph n = 20,001, 3000 sources 9.9 against 16.3.
//   Narrow graphs (largest degree <= 8, road-like: levels of about sqrt(n) vertices) only while
//   three CTAs' states fit an SM: their levels leave a large CTA idle, so many small CTAs win
//   (roads with chains, all sources: n = 9,600 7.2 from global memory with eight CTAs per SM,
//   18 with one state per SM; n = 4,900 2.6 from shared, 2.7 from global memory).
// * 64 registers and 1024 threads per SM where rows beyond 64 arcs keep whole warps busy (R-MAT
//   scale 12 all sources 3.3 against 4.1 with 128 registers and 512 threads; social graph above
//   10.0 against 10.7), else 128 registers and 512 threads (G(9000, 36,000) all sources 9.0
//   against 10.0), a lane then taking rows of up to 32 arcs instead of 12 (G(9000, 72,000): 12.9,
//   with 16 16.4, with 12 20.5; the social graph 9.6 with 12, 9.9 with 16, 11.1 with 32).  From
//   global memory 128 registers (64 spill in the sweeps: grid 1024^2, 500 sources, 99 against 69);
//   narrow graphs need no code for larger rows and run with 80 (53).
// * Threads: an SM's threads over the states that fit it and have a source (one source on
//   n = 1000: 85 us with 512, 95 with 128); from global memory 512 (social graph
//   n = 60,001, 500 sources: 11.9, 13.3 with 256), narrow graphs 96 / 192 / 384 by size.  Grids, 500
//   sources, with 192 and 384: n = 499,849 25.8 and 25.7, 722,500 41 and 37, 1,048,576 66 and 54.
//   With 96 and 192: every vertex a source 8,100 6.5 and 9.4, 16,129 23.0 and 28.7, 32,400 81 and
//   98; 500 sources 0.92 and 0.91, 1.59 and 1.36, 2.75 and 2.12.  So below 500,000 it is the number of
//   sources per SM that decides; the line at 16,384 takes calls below it as exact ones, above it as
//   a few hundred sources.  With triples 96 and 128 are alike (n = 10,944 15.2 and 14.6, 17,176 31.2
//   and 33.6, 28,997 83 and 84).
static bc_status cta_plan(Ctx *ctx, int n, int max_degree, int units, bool tri, CtaPlan *pl) {
  const bool narrow = max_degree > 0 && max_degree <= kNarrowDeg;
  const bool fits = !tri && n < (1 << 15) && cta_smem_bytes(n, false) <= kCtaSmemMax;
  // CTAs whose state fits an SM's shared memory (1 KB per CTA is the system's, the rest static)
  const int per_sm = fits ? (int)((size_t)227 * 1024 / (cta_smem_bytes(n, cta_smem_q(n)) + 1280)) : 0;
  const bool sm = fits && (!narrow || per_sm >= 3);
  const int lb = sm && max_degree > 64 ? 1024 : 512;
  pl->kind = tri ? 2 : sm ? 1 : 0;
  if (tri)
    pl->kernel = narrow ? (const void *)k_cta_sources<false, true, 512, kNarrowDeg>
                        : (const void *)k_cta_sources<false, true, 512, 16>;
  else if (!sm)
    pl->kernel = narrow ? (const void *)k_cta_sources<false, false, 768, kNarrowDeg>
                        : (const void *)k_cta_sources<false, false, 512, 16>;
  else if (narrow)
    pl->kernel = (const void *)k_cta_sources<true, false, 640, kNarrowDeg>;
  else
    pl->kernel = lb == 512 ? (const void *)k_cta_sources<true, false, 512, 32>
                           : (const void *)k_cta_sources<true, false, 1024, 12>;
  pl->smem = sm ? cta_smem_bytes(n, cta_smem_q(n)) : sizeof(int32_t) * 2 * kRing;
  const int busy = std::min(per_sm, (units + ctx->num_sms - 1) / ctx->num_sms);  // CTAs per SM in use
  if (sm)
    pl->threads = narrow ? std::max(64, 640 / std::min(per_sm, 8) & ~31) : std::max(128, lb / std::min(busy, 8) & ~31);
  else
    pl->threads = !narrow ? 512 : n < 16384 ? 96 : n < 500000 ? (tri ? 128 : 192) : 384;
  {
    // the attribute is per function and device: set it once, to the largest size used, so
    // that concurrent callers (serving workers on graphs of different sizes) never lower it
    // under another's launch
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    BC_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= 64 || !done[dev]) {
      for (const void *k : {(const void *)k_cta_sources<true, false, 640, kNarrowDeg>,
                            (const void *)k_cta_sources<true, false, 512, 32>,
                            (const void *)k_cta_sources<true, false, 1024, 12>})
        BC_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCtaSmemMax));
      if (dev >= 0 && dev < 64) done[dev] = true;
    }
  }
  int bps = 0;
  BC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, pl->kernel, pl->threads, pl->smem));
  if (bps < 1) return fail(BC_ECUDA, "CTA per-source kernel does not fit on an SM");
  pl->ncta = ctx->num_sms * bps;
  return BC_OK;
}

static bc_status cta_alloc(Ctx *ctx, CtaWS **wsp, int n, int rows, size_t b_gws) {
  CtaWS *ws = new (std::nothrow) CtaWS();
  if (!ws) return fail(BC_ENOMEM, "host allocation failed");
  ws->n = n;
  ws->rows = rows;
  ws->b_gws = b_gws;
  const size_t b_bcp = (size_t)rows * n * 8;
  ws->bytes = b_bcp + b_gws + 64 + 2 * (kCtaMaxReq + 1) * sizeof(int32_t);
  bc_status s = ctx->mem.alloc(nullptr, ws->bytes);
  if (s) {
    delete ws;
    return s;
  }
  cudaError_t e = cudaMalloc((void **)&ws->bcp, b_bcp);
  if (e == cudaSuccess) e = cudaMalloc((void **)&ws->gws, b_gws);
  if (e == cudaSuccess) e = cudaMalloc((void **)&ws->stats, 64);
  if (e == cudaSuccess) e = cudaMalloc((void **)&ws->req, 2 * (kCtaMaxReq + 1) * sizeof(int32_t));
  if (e != cudaSuccess) {
    cudaGetLastError();
    cta_free(ctx, ws);
    return fail(BC_ENOMEM, "CTA per-source workspace allocation failed");
  }
  *wsp = ws;
  return BC_OK;
}

// Row records where the budget leaves room (the kernel reads rp and ci without them), at the first call
// whose state lies in global memory.
static void cta_row_records(Ctx *ctx, CtaWS *ws, const CtaPlan &pl) {
  const size_t b_row = (size_t)ws->n * 16;
  if (pl.kind == 1 || ws->row4 || (ctx->mem.budget && ctx->mem.used.load() + 4 * b_row >= ctx->mem.budget) ||
      ctx->mem.alloc(nullptr, b_row) != BC_OK)
    return;
  if (cudaMalloc((void **)&ws->row4, b_row) == cudaSuccess) {
    ws->bytes += b_row;
  } else {
    cudaGetLastError();
    ws->row4 = nullptr;
    ctx->mem.release(nullptr, b_row);
  }
}

// Bytes of a CTA's slice in a plan's layout (a second state and c's records only with triples).
static size_t cta_slice(const CtaPlan &pl, int n) {
  size_t slice = 16 + cta_state_bytes(n, pl.kind == 1);
  if (pl.kind == 2) slice += cta_state_bytes(n, false) + (size_t)n * 16;
  return (slice + 255) & ~(size_t)255;
}

// A workspace for min(plan's CTAs, CTAs the call can use) in the plan's layout, *max_cta = how many it
// holds.  It grows to at least twice the CTAs (calls whose number of sources grows one by one would
// free and allocate it each time: k = 33 to 150 on n = 60,000 took 118 allocations, now at most 4) and keeps
// what other layouts needed (one- and two-state calls taking turns), as far as half of the
// context's free budget, else the device's memory, allows.
static bc_status cta_ensure(Ctx *ctx, CtaWS **wsp, int n, int64_t units, const CtaPlan &pl, int *max_cta) {
  CtaWS *ws = *wsp;
  const size_t slice = cta_slice(pl, n), per_cta = (size_t)n * 8 + slice;
  const bool same = ws && ws->n == n;
  const int have = same ? (int)std::min<size_t>({(size_t)ws->rows, ws->b_gws / slice, (size_t)pl.ncta}) : 0;
  int ncta = (int)std::min<int64_t>(pl.ncta, std::max<int64_t>(units, 32));
  size_t room = SIZE_MAX;
  if (ctx->mem.budget) {  // fewer CTAs when the context's HBM budget is tight: at most half
    // of what is free, so that requests arriving meanwhile still find room (serving)
    const size_t used = ctx->mem.used.load() - (ws ? ws->bytes : 0);
    const size_t avail = ctx->mem.budget > used + 64 ? ctx->mem.budget - used - 64 : 0;
    room = avail / 2;
    ncta = (int)std::min<size_t>((size_t)ncta, std::max<size_t>(room / per_cta, avail >= per_cta ? 1 : 0));
    if (ncta < 1) return fail(BC_ENOMEM, "CTA per-source workspace exceeds the context HBM budget");
  }
  *max_cta = have;
  if (have >= ncta) {
    cta_row_records(ctx, ws, pl);
    return BC_OK;
  }
  int rows = ncta;
  size_t b_gws = slice * ncta;
  if (same) {
    const int grown = std::max(ncta, (int)std::min<size_t>({(size_t)pl.ncta, (size_t)2 * have, room / per_cta}));
    const int r2 = std::max(grown, ws->rows);
    const size_t g2 = std::max(slice * grown, ws->b_gws);
    if ((size_t)r2 * n * 8 + g2 <= room) {
      rows = r2;
      b_gws = g2;
    }
  }
  cta_free(ctx, ws);
  *wsp = nullptr;
  bc_status s = cta_alloc(ctx, wsp, n, rows, b_gws);
  if (s && (rows != ncta || b_gws != slice * ncta)) s = cta_alloc(ctx, wsp, n, ncta, slice * ncta);
  if (s) return s;
  *max_cta = (int)std::min<size_t>({(size_t)(*wsp)->rows, (*wsp)->b_gws / slice, (size_t)pl.ncta});
  cta_row_records(ctx, *wsp, pl);
  return BC_OK;
}

bool cta_fits(int32_t n) { return n > 0 && n <= kCtaMaxN; }

bc_status cta_run(Ctx *ctx, Graph *g, CtaWS **wsp, const PlainArgs &a, cudaStream_t st, bc_stats *acc) {
  const DeviceGraph *dg = a.g;
  const int n = dg->n;
  const bool sssp = a.out_depth != nullptr;
  if (a.nsrc <= 0 && a.ntri <= 0) return BC_OK;
  CtaPlan pl;
  const int units = sssp ? 1 : std::max(a.nsrc, a.ntri);
  bc_status s = cta_plan(ctx, n, a.max_degree, units, !sssp && a.ntri > 0, &pl);
  int max_cta = 0;
  if (!s) s = cta_ensure(ctx, wsp, n, units, pl, &max_cta);
  if (s) return s;
  CtaWS *ws = *wsp;
  CtaK p;
  memset(&p, 0, sizeof(p));
  p.n = n;
  p.rp = dg->rp;
  p.ci = dg->ci;
  p.omega = a.omega;
  p.src = a.src;
  p.nsrc = sssp ? 1 : a.nsrc;
  p.leaf_term = a.leaf_term ? 1 : 0;
  p.bcp = ws->bcp;
  p.gws = ws->gws;
  p.slice = cta_slice(pl, n);
  p.row4 = pl.kind == 1 ? nullptr : ws->row4;
  p.spread = a.max_degree <= 0 || a.max_degree > kThin;
  p.stats = ws->stats;
  p.out_depth = a.out_depth;
  p.out_sigma = a.out_sigma;
  p.out_ovf = a.out_ovf;
  p.tri = a.tri;
  p.ntri = sssp ? 0 : a.ntri;
  if (a.nreq > 0 && (sssp || p.ntri || a.nreq > kCtaMaxReq || !a.h_req_k || !a.req_bc))
    return fail(BC_EINVAL, "CTA per-source kernel: bad request list");
  // requests per launch: groups of consecutive requests, each request with CTAs of its own
  // (at most max_cta requests per launch)
  std::vector<std::vector<int32_t>> hreq;
  int nlaunch = 0, launched_max = 0;
  BC_CUDA_TRY(cudaMemsetAsync(ws->stats, 0, 64, st));
  cudaEvent_t e0, e1;
  BC_CUDA_TRY(cudaEventCreate(&e0));
  BC_CUDA_TRY(cudaEventCreate(&e1));
  cudaEventRecord(e0, st);
  const int was_clean = ws->kind == pl.kind ? ws->clean : 0;
  ws->clean = 0;  // until the launches are known to have completed
  if (p.row4) k_cta_rows<<<ctx->num_sms * 4, 256, 0, st>>>(n, dg->rp, dg->ci, ws->row4);
  cudaError_t le = cudaSuccess;
  auto launch = [&](const CtaK &kp, int ncta, const int32_t *rc, double *const *rbc) {
    CtaK q = kp;
    q.clean = std::max(was_clean, launched_max) >= ncta ? 1 : 0;
    void *args[] = {&q};
    le = cudaLaunchKernel(pl.kernel, dim3(ncta), dim3(pl.threads), args, pl.smem, st);
    launched_max = std::max(launched_max, ncta);
    nlaunch++;
    if (le == cudaSuccess && !sssp && q.nreq > 0) {
      k_cta_reduce_req<<<ctx->num_sms * 4, 256, 0, st>>>(ws->bcp, q.nreq, rc, rbc, n);
      le = cudaGetLastError();
    } else if (le == cudaSuccess && !sssp && a.bc) {
      k_cta_reduce<<<ctx->num_sms * 4, 256, 0, st>>>(ws->bcp, ncta, n, a.bc);
      le = cudaGetLastError();
    }
  };
  if (a.nreq <= 0) {
    launch(p, std::max(1, std::min(max_cta, std::max(p.nsrc, p.ntri))), nullptr, nullptr);
  } else {
    int q0 = 0, soff = 0;
    while (q0 < a.nreq && le == cudaSuccess) {
      const int q1 = std::min(a.nreq, q0 + max_cta);
      const int R = q1 - q0;
      long long K = 0;
      for (int q = q0; q < q1; q++) K += a.h_req_k[q];
      const int C = (int)std::max<long long>(R, std::min<long long>(max_cta, K));
      // CTAs in proportion to the sources (at least one each, at most one per source), then
      // the rest, one at a time, to the request with the most rounds of sources per CTA
      std::vector<int> c(R);
      int used = 0;
      for (int j = 0; j < R; j++) {
        const long long k = a.h_req_k[q0 + j];
        c[j] = (int)std::max<long long>(1, std::min<long long>(k, K > 0 ? C * k / K : 1));
        used += c[j];
      }
      while (used > C) {
        int jm = -1;
        for (int j = 0; j < R; j++)
          if (c[j] > 1 && (jm < 0 || c[j] > c[jm])) jm = j;
        if (jm < 0) break;
        c[jm]--;
        used--;
      }
      while (used < C) {
        int jm = -1;
        long long best = 0;
        for (int j = 0; j < R; j++) {
          const long long k = a.h_req_k[q0 + j];
          const long long rounds = (k + c[j] - 1) / c[j];
          if (c[j] < k && rounds > best) {
            best = rounds;
            jm = j;
          }
        }
        if (jm < 0) break;
        c[jm]++;
        used++;
      }
      std::vector<int32_t> &h = hreq.emplace_back(2 * (R + 1));
      h[0] = 0;
      h[R + 1] = 0;
      for (int j = 0; j < R; j++) {
        h[j + 1] = h[j] + a.h_req_k[q0 + j];
        h[R + 2 + j] = h[R + 1 + j] + c[j];
      }
      le = cudaMemcpyAsync(ws->req, h.data(), h.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st);
      if (le != cudaSuccess) break;
      CtaK kp = p;
      kp.src = a.src + soff;
      kp.nsrc = h[R];
      kp.nreq = R;
      kp.req = ws->req;
      launch(kp, used, ws->req + R + 1, a.req_bc + q0);
      soff += h[R];
      q0 = q1;
    }
  }
  cudaEventRecord(e1, st);
  if (le != cudaSuccess) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return cuda_fail(le, "CTA per-source kernel launch");
  }
  unsigned long long hs[5];
  cudaMemcpyAsync(hs, ws->stats, sizeof(hs), cudaMemcpyDeviceToHost, st);
  const cudaError_t se = cudaEventSynchronize(e1);
  float ms = 0.f;
  if (se == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (se != cudaSuccess) return cuda_fail(se, "CTA per-source kernel");
  BC_CUDA_TRY(cudaStreamSynchronize(st));
  // the launched CTAs left their state cleared; CTAs not launched kept theirs
  ws->clean = std::max(was_clean, launched_max);
  ws->kind = pl.kind;
  if (acc) {
    acc->seconds += ms * 1e-3;
    acc->sources += p.nsrc + 3ll * p.ntri;
    acc->sigma_overflow_sources += (int64_t)hs[4];
    acc->reached_vertices += (int64_t)hs[0];
    acc->reached_arcs += (int64_t)hs[1];
    acc->levels += (int64_t)hs[2];
    if ((int32_t)hs[3] > acc->max_depth) acc->max_depth = (int32_t)hs[3];
    acc->kernel_launches += (sssp ? nlaunch : 2 * nlaunch) + (p.row4 ? 1 : 0);
    if (acc->tile_width == 0) acc->tile_width = 1;
  }
  return BC_OK;
}

}  // namespace bcl

// Device 1-degree preprocessing (Alg. 6 on one GPU; Eq. 3's omega).
//
// A vertex u with deg(u) = 1 whose only neighbour v has deg(v) >= 2 is removed and
// omega[v] counts it; both arcs (u,v) and (v,u) leave the graph (Sec. 3.4.1).  A K2
// component keeps both ends (removing both would lose the pair).  One removal round
// only (Sec. 3.4.1 footnote 1).  The residual CSR keeps the original vertex ids, so
// depths, sigma and BC of residual vertices are indexed as in the input graph.
#include <algorithm>

#include "bc_internal.h"
#include "bc_scan.cuh"

namespace bcl {

namespace {

__global__ void k_mark_leaves(int32_t n, const int32_t *rp, const int32_t *ci, int32_t *omega,
                              uint8_t *removed) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
       u += (int64_t)gridDim.x * blockDim.x) {
    int32_t a = rp[u];
    uint8_t rem = 0;
    if (rp[u + 1] - a == 1) {
      int32_t v = ci[a];
      if (rp[v + 1] - rp[v] >= 2) {
        rem = 1;
        atomicAdd(omega + v, 1);
      }
    }
    removed[u] = rem;
  }
}

// Kept arcs as a bit mask over col_idx (bit e = arc e stays), 32 arcs per warp and word: the
// target of a kept arc is not removed.  The arcs of removed vertices, one each, are cleared by
// k_drop_leaf_arcs.  Residual rows are then a compaction of col_idx by this mask, so no thread
// walks a row: a thread per row took 26 ms on R-MAT scale 20 (its largest row has 64 k arcs).
__global__ void k_kept_arcs(int64_t nnz, const int32_t *__restrict__ ci, const uint8_t *__restrict__ removed,
                            uint32_t *kept) {
  const int lane = lane_id();
  const int64_t nw = (nnz + 31) / 32, step = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < nw; i += step) {
    const int64_t e = i * 32 + lane;
    const unsigned m = __ballot_sync(BC_FULL, e < nnz && !removed[ci[e]]);
    if (lane == 0) kept[i] = m;
  }
}

__global__ void k_drop_leaf_arcs(int32_t n, const int32_t *rp, const uint8_t *removed, uint32_t *kept) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
    if (removed[u]) atomicAnd(kept + (rp[u] >> 5), ~(1u << (rp[u] & 31)));
}

// cnt[i] = kept arcs of word i (i < nw), cnt[nw] = 0: its exclusive scan ends in the total
__global__ void k_kept_counts(int64_t nw, const uint32_t *kept, int32_t *cnt) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= nw; i += (int64_t)gridDim.x * blockDim.x)
    cnt[i] = i < nw ? __popc(kept[i]) : 0;
}

// Residual row offsets (kept arcs before a row's first arc) from the mask and the scan of its
// word counts, and the flags of the pruned run's sources: every non-removed vertex that has a
// residual edge or removed leaves (the latter still owes its deferred leaf term).
__device__ __forceinline__ int32_t kept_before(int64_t e, int64_t nw, const uint32_t *kept, const int32_t *pre) {
  const int64_t i = e >> 5;
  return pre[i] + (i < nw ? __popc(kept[i] & ((1u << (e & 31)) - 1u)) : 0);
}
__global__ void k_residual_rows(int32_t n, const int32_t *rp, int64_t nw, const uint32_t *kept, const int32_t *pre,
                                const uint8_t *removed, const int32_t *omega, int32_t *rrp, int32_t *flag) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u <= n; u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = kept_before(rp[u], nw, kept, pre);
    rrp[u] = a;
    flag[u] = (u < n && !removed[u] && (kept_before(rp[u + 1], nw, kept, pre) > a || omega[u] > 0)) ? 1 : 0;
  }
}

__global__ void k_residual_fill(int64_t nnz, const int32_t *__restrict__ ci, const uint32_t *__restrict__ kept,
                                const int32_t *__restrict__ pre, int32_t *rci) {
  const int lane = lane_id();
  const int64_t nw = (nnz + 31) / 32, step = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < nw; i += step) {
    const uint32_t m = kept[i];
    if ((m >> lane) & 1u) rci[pre[i] + __popc(m & lanemask_lt())] = ci[i * 32 + lane];
  }
}

// out[pos[u]] = u for the flagged vertices: the sources in increasing vertex order, so every
// call gives the same sources to the same tiles and CTAs
__global__ void k_pruned_sources(int32_t n, const int32_t *flag, const int32_t *pos, int32_t *out) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
    if (flag[u]) out[pos[u]] = (int32_t)u;
}

int blocks_for(int64_t work, Ctx *c) {
  int64_t b = (work + 255) / 256, cap = (int64_t)c->num_sms * 16;
  return (int)(b < 1 ? 1 : b > cap ? cap : b);
}

}  // namespace

void prune_free(Ctx *ctx, PruneCache *p) {
  if (!p->omega) return;
  const size_t n = (size_t)p->res.n;
  ctx->mem.release(p->omega, n * 4);
  ctx->mem.release(p->removed, n);
  ctx->mem.release(p->src, n * 4 + 4);
  ctx->mem.release(p->res.rp, (n + 1) * 4);
  if (p->res.ci) ctx->mem.release(p->res.ci, (size_t)p->res.nnz * 4 + 4);
  *p = PruneCache();
}

bc_status prune_build(Ctx *ctx, Graph *g, cudaStream_t st) {
  if (g->prune.ready) return BC_OK;
  prune_free(ctx, &g->prune);
  PruneCache &p = g->prune;
  const int32_t n = g->g.n;
  const size_t N = (size_t)n;
  p.res.n = n;
  bc_status s = ctx->mem.alloc((void **)&p.omega, N * 4);
  if (!s) s = ctx->mem.alloc((void **)&p.removed, N);
  if (!s) s = ctx->mem.alloc((void **)&p.src, N * 4 + 4);
  if (!s) s = ctx->mem.alloc((void **)&p.res.rp, (N + 1) * 4);
  if (s) {
    if (p.omega) ctx->mem.release(p.omega, N * 4);
    if (p.removed) ctx->mem.release(p.removed, N);
    if (p.src) ctx->mem.release(p.src, N * 4 + 4);
    p = PruneCache();
    return s;
  }
  // temporary arrays, carved from one allocation: mask, word counts and their scan, source
  // flags and their scan, scan scratch
  const int64_t nnz = g->g.nnz, nw = (nnz + 31) / 32;
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t o_cnt = up((size_t)nw * 4), o_pre = o_cnt + up((size_t)(nw + 1) * 4),
               o_flag = o_pre + up((size_t)(nw + 1) * 4), o_pos = o_flag + up((N + 1) * 4),
               o_scr = o_pos + up((N + 1) * 4),
               total_tmp = o_scr + std::max(scan_scratch_bytes(nw + 1), scan_scratch_bytes(n + 1));
  char *tmp = nullptr;
  cudaError_t e = cudaMalloc(&tmp, total_tmp);
  uint32_t *kept = (uint32_t *)tmp;
  int32_t *cnt = (int32_t *)(tmp + o_cnt), *pre = (int32_t *)(tmp + o_pre), *flag = (int32_t *)(tmp + o_flag),
          *pos = (int32_t *)(tmp + o_pos);
  if (e == cudaSuccess) e = cudaMemsetAsync(p.omega, 0, N * 4, st);
  const int nb = blocks_for(n, ctx), ab = blocks_for(nnz, ctx), wb = blocks_for(nw + 1, ctx);
  if (e == cudaSuccess) {
    k_mark_leaves<<<nb, 256, 0, st>>>(n, g->g.rp, g->g.ci, p.omega, p.removed);
    k_kept_arcs<<<ab, 256, 0, st>>>(nnz, g->g.ci, p.removed, kept);
    k_drop_leaf_arcs<<<nb, 256, 0, st>>>(n, g->g.rp, p.removed, kept);
    k_kept_counts<<<wb, 256, 0, st>>>(nw, kept, cnt);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = scan_exclusive_i32(cnt, pre, nw + 1, tmp + o_scr, st);
  if (e == cudaSuccess) {
    k_residual_rows<<<nb, 256, 0, st>>>(n, g->g.rp, nw, kept, pre, p.removed, p.omega, p.res.rp, flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = scan_exclusive_i32(flag, pos, n + 1, tmp + o_scr, st);
  if (e == cudaSuccess) {
    k_pruned_sources<<<nb, 256, 0, st>>>(n, flag, pos, p.src);
    e = cudaGetLastError();
  }
  int32_t total = 0, h = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&total, p.res.rp + n, 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, pos + n, 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) {
    p.res.nnz = total;
    s = ctx->mem.alloc((void **)&p.res.ci, (size_t)total * 4 + 4);
    if (s) {
      cudaFree(tmp);
      prune_free(ctx, &p);
      return s;
    }
    k_residual_fill<<<ab, 256, 0, st>>>(nnz, g->g.ci, kept, pre, p.res.ci);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (tmp) cudaFree(tmp);
  if (e != cudaSuccess) {
    prune_free(ctx, &p);
    return cuda_fail(e, "1-degree preprocessing");
  }
  p.nsrc = h;
  p.n_removed = (nnz - total) / 2;  // each removed vertex takes its two arcs out
  p.ready = true;
  return BC_OK;
}

}  // namespace bcl

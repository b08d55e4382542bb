// Plain form of RandomSP (Section III-B): for every sampled pair one
// cooperative launch runs a level-synchronous sigma-counting BFS from s over
// the whole GPU (frontier queues; a warp takes eight rows, all of it a long one,
// and 32 warps a hub's; block 0 alone the small levels), truncated once
// t's level is discovered, then one single-warp launch backtracks a uniform
// shortest path.  This is the baseline the batched form is measured against.
// It also serves VertexDiamUB and the single-source BFS inspection call.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace percis {

namespace {

// Launch shape: one 1,024-thread block per SM (a grid barrier costs with the
// number of blocks).  A warp takes kPerWarp frontier vertices at a time, kGroup lanes
// on each row up to kGroupRow edges, then all lanes on longer ones; rows above kHeavyRow
// edges are split over kHeavyParts warps.  (A hub's row on one warp set the time: R-MAT
// 2^20 one full BFS 4.33 ms with it, 0.62 ms split.)  While the frontier is small --
// at most kSoloVerts vertices whose rows cannot hold more than kSoloEdges edges, or 32
// vertices, and no split row -- block 0 runs the levels alone between block barriers, up
// to kSoloLevels at a time, and the others wait at a grid barrier: the levels of a
// high-diameter graph are far too small for the grid (300 x 300 grid, ~600 levels:
// 6.9 ms with two grid barriers a level, 2.0 ms).
constexpr int kPlainBlock = 1024;
constexpr int kPlainWarps = kPlainBlock / 32;
#ifndef PERCIS_PLAIN_GROUP
#define PERCIS_PLAIN_GROUP 4
#endif
constexpr int kGroup = PERCIS_PLAIN_GROUP;  // lanes per row
constexpr int kPerWarp = 32 / kGroup;       // rows a warp takes together
constexpr int kGroupRow = 64;
constexpr int64_t kHeavyRow = 1024;
constexpr int kHeavyParts = 32;
static_assert(kHeavyParts == kPlainWarps, "block 0 alone gives a part to each warp");
constexpr int kSoloVerts = 1024;
constexpr unsigned long long kSoloEdges = 16384;
constexpr int kSoloLevels = 64;
constexpr int kClaimBuf = 256;

using u64 = unsigned long long;

struct PlainArgs {
    int64_t n;
    const int64_t *rp;
    const int32_t *col;
    const int64_t *irp;
    const int32_t *icol;
    u64 *stamp;  // epoch << 32 | level of the vertices the current BFS has reached (older epochs: not reached)
    double *sigma;
    int32_t *qa;  // frontier queues (even and odd levels): from the back, rows above kHeavyRow
    int32_t *qb;
    int32_t *hub;   // new vertices of in-degree > kHeavyRow
    double *part;   // their partial sums, kHeavyParts each
    const u64 *max_degree;
    PlainCtl *ctl;
    const int32_t *s_dev;
    const int32_t *t_dev;
    const int32_t *kind;
    int64_t idx;
    int32_t s_host, t_host;
    int32_t epoch;
    int32_t levels_only;  // levels (eccentricity) only: no path counts
    uint64_t budget_ns;
};

__global__ void __launch_bounds__(kPlainBlock, 1) k_plain_bfs(PlainArgs a) {
    const int32_t s = a.s_dev ? a.s_dev[a.idx] : a.s_host;
    const int32_t t = a.t_dev ? a.t_dev[a.idx] : a.t_host;
    if (a.kind && a.kind[a.idx] != 0) return;  // zero-weight pair: no path needed (uniform over the grid)
    __shared__ int s_cnt[3];  // block 0 alone: next frontier, its heavy rows, in-degree hubs
    __shared__ int s_found;
    __shared__ int4 s_res;
    __shared__ double s_red[kPlainWarps];
    __shared__ int32_t s_buf[kPlainWarps][kClaimBuf];  // claimed vertices on their way to the frontier
    PlainCtl *ctl = a.ctl;
    GridBarrier *bar = &ctl->bar;
    uint32_t *status = &ctl->status;
    const u64 ep = (u64)(uint32_t)a.epoch << 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane / kGroup, gl = lane % kGroup;
    const unsigned lt = (1u << lane) - 1u;
    const u64 maxdeg = __ldg(a.max_degree);
    const bool hubs = maxdeg > (u64)kHeavyRow;  // some row may be split
    // the frontier, the same in every block: rows of ordinary length, long rows, level
    const bool s_long = a.rp[s + 1] - a.rp[s] > kHeavyRow;
    int nq = s_long ? 0 : 1, nh = s_long ? 1 : 0, L = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.stamp[s] = ep;
        a.sigma[s] = 1.0;
        a.qa[s_long ? a.n - 1 : 0] = s;
        for (int k = 0; k < 3; ++k) ctl->qsize[k] = ctl->hsize[k] = ctl->nhub[k] = 0;
        ctl->level = 0;
        ctl->found = 0;
    }
    if (!grid_sync(bar, status, a.budget_ns)) return;

    // Each warp gathers the vertices it claims in shared memory and appends them to the
    // next frontier kClaimBuf / 2 or more at a time (an append per step queues at the
    // frontier's counter: R-MAT 2^20 1.01 ms, gathered 0.98 ms, before the hubs were split further).
    int held = 0;  // (the same in every lane)
    auto flush = [&](int32_t *nxt, int *qn) {
        if (held == 0) return;
        __syncwarp();
        int pos = 0;
        if (lane == 0) pos = atomicAdd(qn, held);
        pos = __shfl_sync(0xffffffffu, pos, 0);
        for (int q = lane; q < held; q += 32) nxt[pos + q] = s_buf[warp][q];
        __syncwarp();
        held = 0;
    };
    // claim the undiscovered of four edges' targets (v < 0: none) for the next
    // frontier; every lane of the warp calls it
    auto claim4 = [&](const int32_t (&v)[4], int level, int32_t *nxt, int *qn, int *qh, int *nhub) {
        u64 st[4];
        bool mine[4], heavy[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) st[q] = v[q] >= 0 ? __ldcg(&a.stamp[v[q]]) : ep;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            mine[q] = (st[q] >> 32) != (ep >> 32) && atomicMax(&a.stamp[v[q]], ep | (u64)(level + 1)) < ep;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            heavy[q] = false;
            if (hubs && mine[q]) {
                heavy[q] = a.rp[v[q] + 1] - a.rp[v[q]] > kHeavyRow;
                if (heavy[q]) nxt[a.n - 1 - atomicAdd(qh, 1)] = v[q];
                if (!a.levels_only && a.irp[v[q] + 1] - a.irp[v[q]] > kHeavyRow) a.hub[atomicAdd(nhub, 1)] = v[q];
            }
            const unsigned m = __ballot_sync(0xffffffffu, mine[q] && !heavy[q]);
            if (mine[q] && !heavy[q]) s_buf[warp][held + __popc(m & lt)] = v[q];
            held += __popc(m);
        }
        if (held > kClaimBuf - 128) flush(nxt, qn);  // (a step adds at most 128)
    };
    // expand the light rows of the frontier (warps w0, w0 + nw, ...)
    auto expand = [&](int64_t w0, int64_t nw, int nq, int level, const int32_t *cur, int32_t *nxt, int *qn, int *qh,
                      int *nhub) {
        for (int64_t k0 = w0 * kPerWarp; k0 < nq; k0 += nw * kPerWarp) {
            const int64_t k = k0 + g;
            int64_t e0 = 0, e1 = 0;
            if (k < nq) {
                const int32_t u = __ldcg(&cur[k]);
                e0 = a.rp[u];
                e1 = a.rp[u + 1];
            }
            const bool big = e1 - e0 > kGroupRow;
            const unsigned bm = __ballot_sync(0xffffffffu, big && gl == 0);
            const int steps = __reduce_max_sync(0xffffffffu, big ? 0 : ((int)(e1 - e0) + 4 * kGroup - 1) / (4 * kGroup));
            for (int r = 0; r < steps; ++r) {
                int32_t v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int64_t e = e0 + kGroup * (4 * r + q) + gl;
                    v[q] = !big && e < e1 ? a.col[e] : -1;
                }
                claim4(v, level, nxt, qn, qh, nhub);
            }
            for (unsigned b = bm; b; b &= b - 1) {
                const int src = __ffs(b) - 1;
                const int64_t f0 = __shfl_sync(0xffffffffu, e0, src), f1 = __shfl_sync(0xffffffffu, e1, src);
                for (int64_t base = f0; base < f1; base += 128) {
                    int32_t v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int64_t e = base + 32 * q + lane;
                        v[q] = e < f1 ? a.col[e] : -1;
                    }
                    claim4(v, level, nxt, qn, qh, nhub);
                }
            }
        }
        flush(nxt, qn);
    };
    // sum of the counts of in-edges [e, e1), `step` apart, whose tail is at `level`
    auto tails = [&](int64_t e, int64_t e1, int64_t step, int level) -> double {
        double acc = 0.0;
        const u64 want = ep | (u64)level;
        for (; e < e1; e += 4 * step) {
            int32_t u[4];
            double c[4];
            bool at[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) u[q] = e + q * step < e1 ? a.icol[e + q * step] : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                at[q] = u[q] >= 0 && __ldcg(&a.stamp[u[q]]) == want;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                c[q] = at[q] ? __ldcg(&a.sigma[u[q]]) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (at[q]) acc += c[q];
        }
        return acc;
    };
    auto settle = [&](int32_t v, double acc, int *found) {
        a.sigma[v] = acc;
        if (acc >= kTwo53) atomicOr(status, DEV_SIGMA_OVERFLOW);
        if (v == t) *(volatile int *)found = 1;
    };
    // counts of the new vertices of in-degree <= kHeavyRow (fixed summation order)
    auto pull = [&](int64_t w0, int64_t nw, int nl, int nh, int level, const int32_t *nxt, int *found) {
        const int nn = nl + nh;
        for (int64_t k0 = w0 * kPerWarp; k0 < nn; k0 += nw * kPerWarp) {
            const int64_t k = k0 + g;
            int64_t e0 = 0, e1 = 0;
            int32_t v = -1;
            if (k < nn) {
                v = __ldcg(&nxt[k < nl ? k : a.n - 1 - (k - nl)]);
                e0 = a.irp[v];
                e1 = a.irp[v + 1];
            }
            const bool hub = e1 - e0 > kHeavyRow, big = e1 - e0 > kGroupRow && !hub;
            const unsigned bm = __ballot_sync(0xffffffffu, big && gl == 0);
            double acc = big || hub ? 0.0 : tails(e0 + gl, e1, kGroup, level);
            __syncwarp();
#pragma unroll
            for (int o = kGroup / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (gl == 0 && v >= 0 && !big && !hub) settle(v, acc, found);
            for (unsigned b = bm; b; b &= b - 1) {
                const int src = __ffs(b) - 1;
                const int64_t f0 = __shfl_sync(0xffffffffu, e0, src), f1 = __shfl_sync(0xffffffffu, e1, src);
                const int32_t fv = __shfl_sync(0xffffffffu, v, src);
                acc = tails(f0 + lane, f1, 32, level);
                __syncwarp();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) settle(fv, acc, found);
            }
        }
    };
    // one part of a hub's in-row by the warp: the sum, in every lane
    auto hub_part = [&](int64_t r, int p, int level) -> double {
        const int32_t v = __ldcg(&a.hub[r]);
        const int64_t e0 = a.irp[v], len = a.irp[v + 1] - e0, per = (len + kHeavyParts - 1) / kHeavyParts;
        const int64_t b = e0 + p * per, e = min(e0 + len, b + per);
        double acc = tails(b + lane, e, 32, level);
        __syncwarp();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        return acc;
    };

    const int64_t gw = (int64_t)blockIdx.x * kPlainWarps + warp, nwarps = (int64_t)gridDim.x * kPlainWarps;
    auto solo_ok = [&](int cnt, int heavy) {
        return heavy == 0 && cnt <= kSoloVerts && (cnt <= 32 || (u64)cnt * maxdeg <= kSoloEdges);
    };
    // Sizes reach the other blocks through slots that are written again only after
    // every block has passed a later barrier: three in turn for the grid's levels
    // (step), two in turn for block 0's stints.
    int step = 0, stint = 0;
    // a target equal to the source is settled at level 0: nothing to expand
    for (; t < 0 || t != s;) {
        int found = 0;
        if (solo_ok(nq, nh)) {
            if (blockIdx.x == 0) {
                if (threadIdx.x == 0) s_found = 0;
                for (int r = 0; r < kSoloLevels && nq > 0 && solo_ok(nq, nh) && !found; ++r, ++L) {
                    if (threadIdx.x < 3) s_cnt[threadIdx.x] = 0;
                    __syncthreads();
                    int32_t *nxt = (L & 1) ? a.qa : a.qb;
                    expand(warp, kPlainWarps, nq, L, (L & 1) ? a.qb : a.qa, nxt, &s_cnt[0], &s_cnt[1], &s_cnt[2]);
                    __syncthreads();
                    nq = s_cnt[0];
                    nh = s_cnt[1];
                    if (!a.levels_only) {
                        const int nhub = s_cnt[2];
                        pull(warp, kPlainWarps, nq, nh, L, nxt, &s_found);
                        for (int h = 0; h < nhub; ++h) {
                            const double part = hub_part(h, warp, L);
                            if (lane == 0) s_red[warp] = part;
                            __syncthreads();
                            if (threadIdx.x == 0) {
                                double acc = 0.0;
                                for (int p = 0; p < kHeavyParts; ++p) acc += s_red[p];
                                settle(__ldcg(&a.hub[h]), acc, &s_found);
                            }
                            __syncthreads();
                        }
                        __syncthreads();
                        found = *(volatile int *)&s_found;
                    }
                    __syncthreads();  // the counters are cleared for the next level
                }
                if (threadIdx.x == 0) ctl->solo[stint & 1] = make_int4(nq, nh, L, found);
            }
            if (!grid_sync(bar, status, a.budget_ns)) return;
            if (threadIdx.x == 0) s_res = __ldcg(&ctl->solo[stint & 1]);  // (one request a block)
            __syncthreads();
            const int4 res = s_res;
            nq = res.x;
            nh = res.y;
            L = res.z;
            found = res.w;
            ++stint;
        } else {
            const int nx = (step + 1) % 3, n2 = (step + 2) % 3;
            if (blockIdx.x == 0 && threadIdx.x == 0) ctl->qsize[n2] = ctl->hsize[n2] = ctl->nhub[n2] = 0;
            const int32_t *cur = (L & 1) ? a.qb : a.qa;
            int32_t *nxt = (L & 1) ? a.qa : a.qb;
            for (int64_t it = gw; it < (int64_t)nh * kHeavyParts; it += nwarps) {
                const int32_t u = __ldcg(&cur[a.n - 1 - it / kHeavyParts]);
                const int64_t e0 = a.rp[u], len = a.rp[u + 1] - e0, per = (len + kHeavyParts - 1) / kHeavyParts;
                const int64_t b = e0 + (it % kHeavyParts) * per, e1 = min(e0 + len, b + per);
                for (int64_t base = b; base < e1; base += 128) {
                    int32_t v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int64_t e = base + 32 * q + lane;
                        v[q] = e < e1 ? a.col[e] : -1;
                    }
                    claim4(v, L, nxt, &ctl->qsize[nx], &ctl->hsize[nx], &ctl->nhub[nx]);
                }
            }
            expand(gw, nwarps, nq, L, cur, nxt, &ctl->qsize[nx], &ctl->hsize[nx], &ctl->nhub[nx]);
            if (!grid_sync(bar, status, a.budget_ns)) return;
            if (threadIdx.x == 0)
                s_res = make_int4((int)ld_relaxed_u32((const uint32_t *)&ctl->qsize[nx]),
                                  (int)ld_relaxed_u32((const uint32_t *)&ctl->hsize[nx]),
                                  (int)ld_relaxed_u32((const uint32_t *)&ctl->nhub[nx]), 0);
            __syncthreads();
            nq = s_res.x;
            nh = s_res.y;
            if (!a.levels_only) {
                const int nhub = s_res.z;
                for (int64_t it = gw; it < (int64_t)nhub * kHeavyParts; it += nwarps) {
                    const double acc = hub_part(it / kHeavyParts, (int)(it % kHeavyParts), L);
                    if (lane == 0) a.part[it] = acc;
                }
                pull(gw, nwarps, nq, nh, L, nxt, &ctl->found);
                if (!grid_sync(bar, status, a.budget_ns)) return;
                if (nhub > 0) {
                    for (int64_t h = (int64_t)blockIdx.x * kPlainBlock + threadIdx.x; h < nhub;
                         h += (int64_t)gridDim.x * kPlainBlock) {
                        double acc = 0.0;
                        for (int p = 0; p < kHeavyParts; ++p) acc += __ldcg(&a.part[h * kHeavyParts + p]);
                        settle(__ldcg(&a.hub[h]), acc, &ctl->found);
                    }
                    if (!grid_sync(bar, status, a.budget_ns)) return;
                }
                if (t >= 0) {  // (written between barriers of a grid level only)
                    if (threadIdx.x == 0) s_found = (int)ld_relaxed_u32((const uint32_t *)&ctl->found);
                    __syncthreads();
                    found = s_found;
                }
            }
            ++L;
            ++step;
        }
        if (nq + nh == 0) {
            --L;  // the deepest level was the one before
            break;
        }
        if (found) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->level = L;
}

// Backtrack of one sample with one warp: from w = t, draw u in (0,1] and
// move to the first predecessor (in-adjacency order) whose running sigma sum
// reaches u * sigma_w.  The running sums are exact (integers below 2^53), so a
// warp-parallel scan picks the same predecessor as a sequential scan.
__global__ void k_plain_backtrack(const int64_t *irp, const int32_t *icol, const u64 *stamp,
                                  const double *sigma, int32_t epoch, const int32_t *s_arr, const int32_t *t_arr,
                                  int32_t *kind, int64_t idx, uint64_t seed, uint32_t tag, int32_t *ilen,
                                  long long *path_off, int32_t *arena, unsigned long long *arena_top,
                                  int64_t arena_cap, unsigned long long *cnt, uint32_t *status) {
    const int lane = threadIdx.x & 31;
    const int32_t s = s_arr[idx], t = t_arr[idx];
    if (kind[idx] != 0 || (int32_t)(stamp[t] >> 32) != epoch) {
        if (lane == 0) {
            if (kind[idx] == 0) kind[idx] = 2;
            ilen[idx] = 0;
            path_off[idx] = 0;
        }
        return;
    }
    const int32_t d = (int32_t)(uint32_t)stamp[t];
    const int32_t len = d - 1;
    unsigned long long off = 0;
    if (lane == 0) {
        off = atomicAdd(arena_top, (unsigned long long)len);
        ilen[idx] = len;
        path_off[idx] = (long long)off;
        if ((int64_t)(off + len) > arena_cap) atomicOr(status, DEV_ARENA_OVERFLOW);
    }
    off = __shfl_sync(0xffffffffu, off, 0);
    const bool store = (int64_t)(off + len) <= arena_cap;
    int32_t w = t;
    int32_t lw = d;
    uint32_t step = 0;
    int32_t k = 0;
    while (w != s) {
        const double target = __dmul_rn(uniform_at(seed, (uint64_t)idx, tag, step), sigma[w]);
        const int64_t e0 = irp[w], e1 = irp[w + 1];
        double carry = 0.0;
        int32_t pick = -1;
        for (int64_t base = e0; base < e1 && pick < 0; base += 32) {
            const int64_t e = base + lane;
            int32_t p = -1;
            double val = 0.0;
            if (e < e1) {
                p = icol[e];
                if (stamp[p] == ((u64)(uint32_t)epoch << 32 | (uint32_t)(lw - 1))) val = sigma[p];
            }
            const double cum = __dadd_rn(carry, warp_inclusive_scan(val));
            const unsigned hit = __ballot_sync(0xffffffffu, val > 0.0 && cum >= target);
            if (hit) pick = __shfl_sync(0xffffffffu, p, __ffs(hit) - 1);
            carry = __shfl_sync(0xffffffffu, cum, 31);
        }
        if (pick < 0) {
            if (lane == 0) atomicOr(status, DEV_BAD_PATH);
            return;
        }
        if (pick != s) {
            if (lane == 0) {
                if (store) arena[off + k] = pick;
                atomicAdd(&cnt[pick], 1ULL);
            }
            ++k;
        }
        w = pick;
        --lw;
        ++step;
    }
}

__global__ void k_dist_sigma(const u64 *stamp, const double *sigma, int32_t epoch, int64_t n,
                             int32_t *dist, double *sig) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const u64 st = stamp[v];
        const bool in = (int32_t)(st >> 32) == epoch;
        if (dist) dist[v] = in ? (int32_t)(uint32_t)st : -1;
        if (sig) sig[v] = in ? sigma[v] : 0.0;
    }
}

__global__ void k_argmax_degree(const int64_t *rp, const u64 *stamp, const int32_t *seen_epoch_lo, int64_t n,
                                unsigned long long *best) {
    // key = (degree << 32) | (~v): max degree, ties to the smallest id
    unsigned long long m = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int64_t dg = rp[v + 1] - rp[v];
        if (dg > 0 && (int32_t)(stamp[v] >> 32) < *seen_epoch_lo) {
            const unsigned long long key = ((unsigned long long)dg << 32) | (0xffffffffu - (uint32_t)v);
            m = m > key ? m : key;
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, off);
        m = m > o ? m : o;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(best, m);
}

}  // namespace

static percis_status ensure_plain(percis_ctx *ctx) {
    const int64_t n = ctx->n;
    const bool fresh = ctx->stamp.bytes < sizeof(u64) * (size_t)n;
    PERCIS_TRY(ensure(ctx, ctx->stamp, sizeof(u64) * n, "level stamps"));
    const int64_t hubs = ctx->nnz / kHeavyRow + 1;  // vertices of in-degree > kHeavyRow, at most
    PERCIS_TRY(ensure(ctx, ctx->plain_hub, (sizeof(double) * kHeavyParts + sizeof(int32_t)) * hubs, "hub sums"));
    PERCIS_TRY(ensure(ctx, ctx->sigma1, sizeof(double) * n, "sigma"));
    PERCIS_TRY(ensure(ctx, ctx->qa, sizeof(int32_t) * n, "queue"));
    PERCIS_TRY(ensure(ctx, ctx->qb, sizeof(int32_t) * n, "queue"));
    PERCIS_TRY(ensure(ctx, ctx->plain_ctl, 256, "plain ctl"));
    if (fresh || ctx->epoch <= 0 || ctx->epoch > (1 << 30)) {
        // (all of the buffer: a larger graph that still fits it is not fresh)
        PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->stamp.p, 0, ctx->stamp.bytes, ctx->stream));
        PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->plain_ctl.p, 0, 256, ctx->stream));
        ctx->epoch = 0;
    }
    if (ctx->plain_grid == 0) {  // co-resident blocks on this context's device
        int per_sm = 0;
        PERCIS_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_plain_bfs, kPlainBlock, 0));
        ctx->plain_grid = std::max(1, per_sm) * ctx->num_sms;
    }
    return PERCIS_OK;
}

percis_status plain_bfs(percis_ctx *ctx, const int32_t *s_dev, const int32_t *t_dev, int64_t idx, int32_t s_host,
                        int32_t t_host, bool levels_only) {
    PERCIS_TRY(ensure_plain(ctx));
    ctx->epoch++;
    PlainArgs a;
    a.n = ctx->n;
    a.rp = ctx->rp.as<int64_t>();
    a.col = ctx->col.as<int32_t>();
    a.irp = ctx->directed ? ctx->irp.as<int64_t>() : ctx->rp.as<int64_t>();
    a.icol = ctx->directed ? ctx->icol.as<int32_t>() : ctx->col.as<int32_t>();
    a.stamp = ctx->stamp.as<u64>();
    a.part = ctx->plain_hub.as<double>();
    a.hub = reinterpret_cast<int32_t *>(a.part + kHeavyParts * (ctx->nnz / kHeavyRow + 1));
    a.max_degree = ctx->graph_info.as<u64>();
    a.sigma = ctx->sigma1.as<double>();
    a.qa = ctx->qa.as<int32_t>();
    a.qb = ctx->qb.as<int32_t>();
    a.ctl = ctx->plain_ctl.as<PlainCtl>();
    a.s_dev = s_dev;
    a.t_dev = t_dev;
    a.kind = s_dev ? ctx->kind.as<int32_t>() : nullptr;
    a.idx = idx;
    a.s_host = s_host;
    a.t_host = t_host;
    a.epoch = ctx->epoch;
    a.levels_only = levels_only ? 1 : 0;
    a.budget_ns = (uint64_t)(ctx->opt.timeout_s * 1e9);
    void *args[] = {&a};
    PERCIS_CUDA(ctx, cudaLaunchCooperativeKernel((const void *)k_plain_bfs, dim3(ctx->plain_grid), dim3(kPlainBlock),
                                                 args, 0, ctx->stream));
    ctx->launches++;
    return PERCIS_OK;
}

percis_status plain_backtrack(percis_ctx *ctx, uint64_t seed, uint32_t tag, int64_t idx) {
    k_plain_backtrack<<<1, 32, 0, ctx->stream>>>(
        ctx->directed ? ctx->irp.as<int64_t>() : ctx->rp.as<int64_t>(),
        ctx->directed ? ctx->icol.as<int32_t>() : ctx->col.as<int32_t>(), ctx->stamp.as<u64>(), ctx->sigma1.as<double>(), ctx->epoch, ctx->pair_s.as<int32_t>(),
        ctx->pair_t.as<int32_t>(), ctx->kind.as<int32_t>(), idx, seed, tag, ctx->ilen.as<int32_t>(),
        ctx->path_off.as<long long>(), ctx->arena.as<int32_t>(), ctx->arena_top.as<unsigned long long>(),
        ctx->arena_cap, ctx->cnt.as<unsigned long long>(), &ctx->plain_ctl.as<PlainCtl>()->status);
    PERCIS_CHECK_LAUNCH(ctx, "plain backtrack");
    return PERCIS_OK;
}

percis_status plain_phase(percis_ctx *ctx, uint64_t seed, uint32_t tag_path, int64_t count) {
    for (int64_t i = 0; i < count; ++i) {
        PERCIS_TRY(plain_bfs(ctx, ctx->pair_s.as<int32_t>(), ctx->pair_t.as<int32_t>(), i, 0, 0));
        PERCIS_TRY(plain_backtrack(ctx, seed, tag_path, i));
    }
    return PERCIS_OK;
}

percis_status plain_dist_sigma(percis_ctx *ctx, int32_t *dist, double *sigma) {
    k_dist_sigma<<<grid_for(ctx, ctx->n, 256), 256, 0, ctx->stream>>>(
        ctx->stamp.as<u64>(), ctx->sigma1.as<double>(), ctx->epoch, ctx->n, dist, sigma);
    PERCIS_CHECK_LAUNCH(ctx, "dist sigma");
    return PERCIS_OK;
}

// VertexDiamUB: for undirected graphs, one full BFS from the largest-degree
// vertex of every component (ties to the smallest id); D = max(2 ecc - 1, 0).
// Directed graphs: D = n - 2.
percis_status vertex_diam_ub(percis_ctx *ctx, int64_t *D) {
    const int64_t n = ctx->n;
    if (ctx->directed) {
        *D = n >= 2 ? n - 2 : 0;
        return PERCIS_OK;
    }
    PERCIS_TRY(ensure_plain(ctx));
    PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->plain_ctl.p, 0, sizeof(PlainCtl), ctx->stream));
    // vertices of earlier components carry epochs >= first_epoch
    const int32_t first_epoch = ctx->epoch + 1;
    PERCIS_TRY(ensure(ctx, ctx->red, 64, "argmax"));
    int32_t *lo_dev = (int32_t *)(ctx->red.as<unsigned long long>() + 1);
    PERCIS_CUDA(ctx, cudaMemcpyAsync(lo_dev, &first_epoch, sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream));
    int64_t best_D = 0;
    for (int64_t comp = 0; comp < n; ++comp) {
        unsigned long long key = 0;
        PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->red.p, 0, sizeof(unsigned long long), ctx->stream));
        k_argmax_degree<<<grid_for(ctx, n, 256), 256, 0, ctx->stream>>>(
            ctx->rp.as<int64_t>(), ctx->stamp.as<u64>(), lo_dev, n, ctx->red.as<unsigned long long>());
        PERCIS_CHECK_LAUNCH(ctx, "argmax degree");
        PERCIS_CUDA(ctx, cudaMemcpyAsync(&key, ctx->red.p, sizeof(key), cudaMemcpyDeviceToHost, ctx->stream));
        PERCIS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        if (key == 0) break;
        const int32_t v = (int32_t)(0xffffffffu - (uint32_t)(key & 0xffffffffu));
        PERCIS_TRY(plain_bfs(ctx, nullptr, nullptr, 0, v, -1, true));
        PlainCtl hc;
        PERCIS_CUDA(ctx, cudaMemcpyAsync(&hc, ctx->plain_ctl.p, sizeof(hc), cudaMemcpyDeviceToHost, ctx->stream));
        PERCIS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        if (hc.status & DEV_TIMEOUT) return set_err(ctx, PERCIS_E_TIMEOUT, "VertexDiamUB BFS timed out");
        const int64_t b = 2 * (int64_t)hc.level - 1;
        best_D = std::max(best_D, b);
    }
    *D = best_D;
    return PERCIS_OK;
}

}  // namespace percis

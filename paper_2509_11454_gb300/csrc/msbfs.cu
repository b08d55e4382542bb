// Batched form of RandomSP: up to W = 64*K distinct sources ("lanes") share
// one persistent cooperative launch.  Per vertex the launch keeps K 64-bit
// words of visited bits and, for every level L, K words of frontier bits
// F_L(v) (bit j set iff v is at distance L from lane j's source).  A level finds
// its vertices by a pull over all that some lane has not visited, or by a push
// over the frontier's out-edges, whichever is estimated to be less work:
//     c = active & ~visited(v),  F_{L+1}(v) = OR_{u in in(v)} F_L(u) & c,
//     sigma_j(v) = sum over u in in(v) with bit j of F_L(u) & c of sigma_j(u)
// (the sigma recurrence of the oracle, summed in any order: the values are
// integers below 2^53, so every order gives the same exact result).  A lane
// retires once every target of its samples is discovered (its level is then
// complete) or its frontier is empty.  Where only samples are wanted the counts
// come after the levels, for the vertices their paths can pass (ms_batch).  Then the same launch
// backtracks every sample of the batch (one warp per sample) exactly as the
// plain form does, reading the frontier history for the predecessor test.
//
// sigma is kept as exact integers: a dependent FP64 add costs ~64 cycles on
// GB300 while integer adds are cheap, and below 2^53 every conversion to FP64
// is exact, so the backtrack compares exactly the FP64 values a plain FP64
// implementation would.  Counts are stored in 32 bits (half the bytes per
// sector) until one reaches 2^32 (DEV_SIGMA_WIDE: the host reruns the phase
// with 64-bit storage), and in FP64 once one reaches 2^53
// (DEV_SIGMA_OVERFLOW), where counts beyond 2^53 round like FP64 sums.
//
// Layout in HBM (vertex-major so one warp reads a vertex's lanes coalesced):
//   visited  uint64 [n][K]
//   history  uint64 [Lcap+1][n][K]
//   sigma    uint64 or double [n][W]
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace percis {

namespace {

constexpr int kMsBlock = 256;
#ifndef PERCIS_BLOCK_DEG
#define PERCIS_BLOCK_DEG 256
#endif
constexpr int kGroupLanes = 8;      // lanes that share a vertex
constexpr int64_t kMidRow = 64;     // rows above it: a whole warp
constexpr int64_t kBigRow = 256;    // in-rows above it: a whole block (listed once per graph)
constexpr int64_t kLightOut = 64;   // out-rows above it: a whole block
constexpr int kBackChunks = 4;       // of 32 candidates, in flight in a backtrack step
constexpr int kQueueBuf = 96;       // queue entries a warp gathers before it appends them
constexpr int64_t kBlockDeg = PERCIS_BLOCK_DEG;  // in-degree above which a whole block counts one (vertex, word)

struct MsArgs {
    // batches of the persistent launch: a host plan, or W-lane batches over the
    // device-resident lane count *u_dev, or the single batch below
    const LaneBatch *plan;
    int32_t nplan;
    const long long *u_dev;
    // A launch covers the vertex range [vlo, vlo + n) of the loaded graph (the
    // whole graph, or the graphs of a multi-graph batch): rp / irp point at
    // entry vlo, column entries and sample vertices are global ids, and the
    // visited, frontier, count and queue arrays are indexed by id - vlo.
    int64_t n;
    int32_t vlo;
    const int64_t *irp;
    const int32_t *icol;
    uint64_t *vis;
    uint64_t *fh;
    void *sigma;
    MsCtl *ctl;
    uint32_t *status;                 // one word for all groups
    int32_t Lcap;
    int32_t lane_base;
    int32_t nlanes;
    const int32_t *lane_src;
    const long long *lane_off;
    const int32_t *samp_t;
    const int32_t *samp_lane;
    const int32_t *sorted_samples;
    int32_t *found;
    int32_t *remaining;
    uint64_t seed;
    uint32_t tag;
    int32_t *kind;
    int32_t *ilen;
    long long *path_off;
    int32_t *arena;
    unsigned long long *arena_top;
    int64_t arena_cap;
    unsigned long long *cnt;
    int32_t full;
    uint64_t budget_ns;
    // push levels: out-adjacency, frontier queues, level stamps
    const int32_t *col;
    int32_t *fq0;
    int32_t *fq1;
    // long rows, needed vertices (see ms_batch); nlist holds ncap entries, ncnt and
    // cont are per level: {light, heavy} counts twice over, lanes that go on
    const int32_t *big;
    const int32_t *big_count;
    const int32_t *lsafe;
    uint64_t *need;
    int32_t *nlist;
    int64_t ncap;
    int32_t *ncnt;
    uint64_t *cont;
    int32_t policy;                   // 0 = pull every level, 1 = push every level, 2 = by work estimate
    double push_alpha;                // policy 2: push while alpha * push work < pull work
    // instrumentation (INSTR variant only)
    const int64_t *rp;                // out-CSR offsets (out-degrees)
    unsigned long long *counters;     // 8 work counters (see percis_info.work)
    unsigned long long *levdeg;       // [W][Lcap+1] out-degree sums per lane and level
    // all-paths estimator: per-warp scratch (tau counts, claim stamps, two level lists)
    int32_t allpaths;
    int32_t ap_warps;
    int32_t ap_epoch;
    double *acc_ap;                   // per-vertex sum of sigma_sv tau_v / sigma_st
    unsigned long long *ap_tau;       // [ap_warps][n]
    int32_t *ap_stamp;                // [ap_warps][n]
    int32_t *ap_list;                 // [ap_warps][2n]
};

// A launch's blocks form `groups` groups, each with a batch of its own and the state for
// one (the arguments of group g are g[g]).  A batch alternates between passes over its
// vertices and waits for their slowest block: one batch at a time kept the issue slots
// 14% busy, half of every warp's time at a barrier.  The groups' blocks alternate on the
// SMs, so one batch's passes fill another's waits.  Batched estimate on Barabasi-Albert
// 100k: 11.3 ms with one group, 8.5 with two, 7.8 with three, 7.0 to 7.4 with four, 6.7
// with six, 7.2 with eight; all-paths estimate of 20k: 3.3, 2.3, 2.2, 2.2, 2.3, 2.1.
constexpr int kMaxGroups = 4;
struct MsLaunch {
    MsArgs g[kMaxGroups];
    int32_t groups;
};
// a block's place in its group, and the group's blocks
struct Place {
    int32_t block, blocks;
};

template <int K>
__device__ __forceinline__ void load_words(const uint64_t *p, uint64_t (&out)[K]) {
    if constexpr (K == 1) {
        out[0] = __ldcg(p);
    } else {
#pragma unroll
        for (int w = 0; w < K; w += 2) {
            const ulonglong2 q = __ldcg(reinterpret_cast<const ulonglong2 *>(p + w));
            out[w] = q.x;
            out[w + 1] = q.y;
        }
    }
}

template <class S>
__device__ __forceinline__ S warp_incl_scan(S v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const S o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    return v;
}

// Sum the counts of one 32-edge chunk's parents into the 64 lanes of word w:
// lane l's edge has parent u and frontier bits fw (already restricted to the
// lanes being counted).  Parents are taken in edge order, four per round so
// their loads overlap; acc0 / acc1 collect lanes l and l+32 of the word.
template <int SM, class ST, class S>
__device__ __forceinline__ void gather_chunk(const ST *sig, int W, int w, uint64_t fw, int32_t u, S &acc0, S &acc1,
                                             bool &ovf) {
    constexpr bool FPSIG = SM == 2;
    constexpr unsigned long long kLimit = SigmaMode<SM>::limit;
    const int lane = threadIdx.x & 31;
    unsigned nz = __ballot_sync(0xffffffffu, fw != 0ull);
    while (nz) {
        const int j0 = __ffs(nz) - 1;
        nz &= nz - 1;
        const bool h1 = nz != 0u;
        const int j1 = h1 ? __ffs(nz) - 1 : j0;
        if (h1) nz &= nz - 1;
        const bool h2 = nz != 0u;
        const int j2 = h2 ? __ffs(nz) - 1 : j0;
        if (h2) nz &= nz - 1;
        const bool h3 = nz != 0u;
        const int j3 = h3 ? __ffs(nz) - 1 : j0;
        if (h3) nz &= nz - 1;
        const uint64_t f0 = shfl64(fw, j0);
        const uint64_t f1 = h1 ? shfl64(fw, j1) : 0ull;
        const uint64_t f2 = h2 ? shfl64(fw, j2) : 0ull;
        const uint64_t f3 = h3 ? shfl64(fw, j3) : 0ull;
        const ST *r0 = sig + (int64_t)__shfl_sync(0xffffffffu, u, j0) * W + 64 * w;
        const ST *r1 = sig + (int64_t)__shfl_sync(0xffffffffu, u, j1) * W + 64 * w;
        const ST *r2 = sig + (int64_t)__shfl_sync(0xffffffffu, u, j2) * W + 64 * w;
        const ST *r3 = sig + (int64_t)__shfl_sync(0xffffffffu, u, j3) * W + 64 * w;
        S a0 = S(0), a1 = S(0), a2 = S(0), a3 = S(0), b0 = S(0), b1 = S(0), b2 = S(0), b3 = S(0);
        if ((f0 >> lane) & 1ull) a0 = __ldcg(r0 + lane);
        if ((f1 >> lane) & 1ull) a1 = __ldcg(r1 + lane);
        if ((f2 >> lane) & 1ull) a2 = __ldcg(r2 + lane);
        if ((f3 >> lane) & 1ull) a3 = __ldcg(r3 + lane);
        if ((f0 >> (lane + 32)) & 1ull) b0 = __ldcg(r0 + lane + 32);
        if ((f1 >> (lane + 32)) & 1ull) b1 = __ldcg(r1 + lane + 32);
        if ((f2 >> (lane + 32)) & 1ull) b2 = __ldcg(r2 + lane + 32);
        if ((f3 >> (lane + 32)) & 1ull) b3 = __ldcg(r3 + lane + 32);
        if (FPSIG) {
            // keep the in-adjacency order of the additions
            acc0 += a0; acc0 += a1; acc0 += a2; acc0 += a3;
            acc1 += b0; acc1 += b1; acc1 += b2; acc1 += b3;
        } else {
            acc0 += (a0 + a1) + (a2 + a3);
            acc1 += (b0 + b1) + (b2 + b3);
            // flag before four more addends could wrap 2^64
            ovf |= (acc0 >= kLimit) | (acc1 >= kLimit);
        }
    }
}

// Counts of level L for the listed vertices (nl from the front of lq, those of
// in-degree > 32, nh, from the back of hq): of a vertex's level-L lanes, all
// (every), or those of `cont` and need.
template <int K, bool INSTR, int SM>
__device__ __noinline__ void count_level(const MsArgs &a, const Place at, int64_t n, int32_t vlo, const int64_t *irp, int L,
                                         const int32_t *lq, int64_t nl, const int32_t *hq, int64_t nh, bool every,
                                         const uint64_t *cont, bool *ovf_out, unsigned long long *work) {
    constexpr int W = 64 * K;
    constexpr bool FPSIG = SM == 2;
    using S = typename SigmaMode<SM>::S;
    using ST = typename SigmaMode<SM>::ST;
    constexpr unsigned long long kLimit = SigmaMode<SM>::limit;
    __shared__ S s_red[kMsBlock / 32][64];  // per-warp partial sums of a block-wide gather
    ST *sig = static_cast<ST *>(a.sigma);
    const int lane = threadIdx.x & 31, warp_in_block = threadIdx.x >> 5;
    const int64_t gwarp = ((int64_t)at.block * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)at.blocks * blockDim.x) >> 5;
    const int64_t nk = n * K;
    const uint64_t *fl = a.fh + (int64_t)L * nk;
    bool ovf = false;
    unsigned long long n_sload = 0, n_swrite = 0;
    auto bits = [&](int32_t v, int wd) -> uint64_t {
        const int64_t q = (int64_t)v * K + wd;
        const uint64_t f = __ldcg(&fl[q]);
        if (every) return f;
        return f & ((cont ? __ldcg(&cont[wd]) : 0ull) | __ldcg(&a.need[q]));
    };
    const uint64_t *fprev = a.fh + (int64_t)(L - 1) * nk;
    if (!FPSIG) {
        // in-degree > kBlockDeg: one block per (vertex, word), its warps
        // splitting the edges; the partial sums meet in shared memory
        // (integer sums, so the order does not matter)
        for (int64_t hi = at.block; hi < nh * K; hi += at.blocks) {
            const int64_t h = hi / K;
            const int wd = (int)(hi - h * K);
            const int32_t v = __ldcg(&hq[-h]);
            const int64_t e0 = irp[v], e1 = irp[v + 1];
            if (e1 - e0 <= kBlockDeg) continue;  // a warp item below; the same for the whole block
            const uint64_t nbw = bits(v, wd);
            if (nbw == 0ull) continue;
            S acc0 = S(0), acc1 = S(0);
            for (int64_t base = e0 + warp_in_block * 32; base < e1; base += kMsBlock) {
                const int64_t e = base + lane;
                int32_t u = 0;
                uint64_t fw = 0ull;
                if (e < e1) {
                    u = a.icol[e] - vlo;
                    fw = __ldcg(&fprev[(int64_t)u * K + wd]) & nbw;
                }
                if (INSTR) n_sload += (unsigned long long)__popcll(fw);
                gather_chunk<SM, ST, S>(sig, W, wd, fw, u, acc0, acc1, ovf);
            }
            s_red[warp_in_block][lane] = acc0;
            s_red[warp_in_block][lane + 32] = acc1;
            __syncthreads();
            if (warp_in_block == 0) {
                S t0 = S(0), t1 = S(0);
#pragma unroll
                for (int q = 0; q < kMsBlock / 32; ++q) {
                    t0 += s_red[q][lane];
                    t1 += s_red[q][lane + 32];
                }
                ovf |= (t0 >= (S)kLimit) | (t1 >= (S)kLimit);
                ST *drow = sig + (int64_t)v * W + 64 * wd;
                if ((nbw >> lane) & 1ull) drow[lane] = (ST)t0;
                if ((nbw >> (lane + 32)) & 1ull) drow[lane + 32] = (ST)t1;
                if (INSTR) n_swrite += lane == 0 ? (unsigned long long)__popcll(nbw) : 0ull;
            }
            __syncthreads();
        }
    }
    for (int64_t it = gwarp; it < nl + nh * K; it += nwarps) {
        if (it < nl) {
            // in-degree <= 32: one warp per vertex, its parents and all their
            // words loaded once; lane w < K holds the word's lanes to count
            const int32_t v = __ldcg(&lq[it]);
            uint64_t nbl = 0ull;
            if (lane < K) nbl = bits(v, lane);
            const unsigned wm = __ballot_sync(0xffffffffu, nbl != 0ull);
            if (!wm) continue;
            const int64_t e0 = irp[v], e1 = irp[v + 1];
            ST *drow = sig + (int64_t)v * W;
            const int64_t e = e0 + lane;
            int32_t u = 0;
            uint64_t f[K];
            if (e < e1) {
                u = a.icol[e] - vlo;
                load_words<K>(fprev + (int64_t)u * K, f);
            } else {
#pragma unroll
                for (int q = 0; q < K; ++q) f[q] = 0ull;
            }
#pragma unroll
            for (int q = 0; q < K; ++q) {
                if (!((wm >> q) & 1u)) continue;
                const uint64_t nbw = shfl64(nbl, q);
                const uint64_t fw = f[q] & nbw;
                if (INSTR) n_sload += (unsigned long long)__popcll(fw);
                S acc0 = S(0), acc1 = S(0);
                gather_chunk<SM, ST, S>(sig, W, q, fw, u, acc0, acc1, ovf);
                if (FPSIG) ovf |= (acc0 >= (S)kLimit) | (acc1 >= (S)kLimit);
                if ((nbw >> lane) & 1ull) drow[64 * q + lane] = (ST)acc0;
                if ((nbw >> (lane + 32)) & 1ull) drow[64 * q + lane + 32] = (ST)acc1;
                if (INSTR) n_swrite += lane == 0 ? (unsigned long long)__popcll(nbw) : 0ull;
            }
        } else {
            // in-degree in (32, kBlockDeg] (any, for FP64 counts, whose
            // additions keep the in-adjacency order): one warp per
            // (vertex, word) over 32-edge chunks
            const int64_t h = (it - nl) / K;
            const int wd = (int)(it - nl - h * K);
            const int32_t v = __ldcg(&hq[-h]);
            const int64_t e0 = irp[v], e1 = irp[v + 1];
            if (!FPSIG && e1 - e0 > kBlockDeg) continue;
            const uint64_t nbw = bits(v, wd);
            if (nbw == 0ull) continue;
            S acc0 = S(0), acc1 = S(0);
            for (int64_t base = e0; base < e1; base += 32) {
                const int64_t e = base + lane;
                int32_t u = 0;
                uint64_t fw = 0ull;
                if (e < e1) {
                    u = a.icol[e] - vlo;
                    fw = __ldcg(&fprev[(int64_t)u * K + wd]) & nbw;
                }
                if (INSTR) n_sload += (unsigned long long)__popcll(fw);
                gather_chunk<SM, ST, S>(sig, W, wd, fw, u, acc0, acc1, ovf);
            }
            if (FPSIG) ovf |= (acc0 >= (S)kLimit) | (acc1 >= (S)kLimit);
            ST *drow = sig + (int64_t)v * W + 64 * wd;
            if ((nbw >> lane) & 1ull) drow[lane] = (ST)acc0;
            if ((nbw >> (lane + 32)) & 1ull) drow[lane + 32] = (ST)acc1;
            if (INSTR) n_swrite += lane == 0 ? (unsigned long long)__popcll(nbw) : 0ull;
        }
    }
    if (ovf) *ovf_out = true;
    if (INSTR) {
        work[0] += n_sload;
        work[1] += n_swrite;
    }
}

// One batch of lanes: levels, counts and the backtrack of its samples.  The
// batch covers lanes lane_base .. lane_base + nlanes - 1 and the vertex range
// [vlo, vlo + n); rp / irp point at entry vlo.  Returns false when the launch
// must stop (a bounded wait ran out, or the frontier history is too short).
//
// A full traversal counts every vertex.  A sampling batch needs the counts of a
// target's ancestors alone (the backtrack reads predecessors of what it has
// reached), a few hundred of the 100,000 vertices a lane reaches: after the
// levels, one backward pass over the frontier history marks them (one bit per
// lane: need), and a forward pass counts those.  This is only done where no count
// anywhere can reach 2^53 (the number of walks of that length, *a.lsafe), so that
// the overflow flag says the same; otherwise every vertex of a continuing lane is
// counted, as in FP64 reruns.  Barabasi-Albert 100k, 512 lanes: 1.54 ms a batch
// with counts everywhere (the gathers of the two largest levels), 0.70 ms (0.57 with
// the control words below read once a block).
//
// Eight lanes share a vertex, lane w mod K on its word w (8 / K edges side by side
// for K < 8): an edge's K words are one coalesced access and the OR over a row
// stays in registers.
template <int K, bool INSTR, int SM>
__device__ __forceinline__ bool ms_batch(const MsArgs &a, const Place at, const int32_t lane_base, const int32_t nlanes,
                                         const int32_t vlo, const int64_t n, const int64_t *rp, const int64_t *irp,
                                         const int32_t ap_epoch) {
    constexpr int W = 64 * K;
    constexpr int SUB = kGroupLanes / K;     // edges a vertex's eight lanes take side by side
    constexpr int GW = 32 / kGroupLanes;     // vertices a warp takes together
    constexpr int EW = 32 / K;               // edges a whole warp takes side by side
    constexpr int EB = kMsBlock / K;         // edges a whole block takes side by side
    constexpr bool FPSIG = SM == 2;
    using S = typename SigmaMode<SM>::S;
    using ST = typename SigmaMode<SM>::ST;
    ST *sig = static_cast<ST *>(a.sigma);
    bool ovf = false;
    unsigned long long n_s[2] = {0, 0}, n_uv = 0, n_ue = 0;  // sigma reads and writes; frontier vertices, edges
    MsCtl *ctl = a.ctl;
    GridBarrier *bar = &ctl->bar;
    uint32_t *status = a.status;
    const int lane = threadIdx.x & 31;
    const int warp_in_block = threadIdx.x >> 5;
    const int64_t tid = (int64_t)at.block * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)at.blocks * blockDim.x;
    const int64_t gwarp = tid >> 5;
    const int64_t nwarps = nthreads >> 5;
    const int64_t nk = n * K;
    const long long p0 = a.full ? 0 : a.lane_off[lane_base];
    const long long p1 = a.full ? 0 : a.lane_off[lane_base + nlanes];
    const int w = lane % K;  // this lane's word wherever lanes share a vertex
    const int nbig = (int)__ldg(a.big_count);
    const unsigned gmask = ((kGroupLanes == 32 ? 0u : (1u << kGroupLanes)) - 1u) << (lane & ~(kGroupLanes - 1));

    // ---- prologue: clear visited, need, frontiers 0 and 1; reset lane state
    for (int64_t i = tid; i < nk; i += nthreads) {
        a.vis[i] = 0ull;
        if (!a.full) a.need[i] = 0ull;
        a.fh[i] = 0ull;
        a.fh[nk + i] = 0ull;
    }
    for (long long p = p0 + tid; p < p1; p += nthreads) a.found[p] = -1;
    if (!a.full)
        for (int64_t i = tid; i < 4 * (int64_t)(a.Lcap + 2); i += nthreads) a.ncnt[i] = 0;
    if (INSTR)
        for (int64_t i = tid; i < (int64_t)W * (a.Lcap + 1); i += nthreads) a.levdeg[i] = 0ull;
    if (at.block == 0) {
        for (int j = threadIdx.x; j < W; j += blockDim.x) a.remaining[j] = 0;
        if (threadIdx.x < K) {
            const int lo = threadIdx.x * 64;
            const int cntl = max(0, min(64, nlanes - lo));
            ctl->active[threadIdx.x] = cntl == 64 ? ~0ull : ((1ull << cntl) - 1ull);
            ctl->nonempty[0][threadIdx.x] = 0ull;
            ctl->nonempty[1][threadIdx.x] = 0ull;
        }
        if (threadIdx.x == 0) {
            ctl->ticket = 0;
            ctl->level = 0;
            ctl->qn[0] = 0;
            ctl->qn[1] = 0;
            ctl->qh[0] = 0;
            ctl->qh[1] = 0;
            for (int q = 0; q < 2; ++q) ctl->fedges[q] = ctl->uedges[q] = 0ull;  // (a last level leaves its own)
            ctl->push_next = a.policy != 0;
            ctl->t_start = globaltimer_ns();
        }
    }
    if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;
    for (int64_t j = tid; j < nlanes; j += nthreads) {
        const int32_t v = a.lane_src[lane_base + j] - vlo;
        const uint64_t bit = 1ull << (j & 63);
        atomicOr((unsigned long long *)&a.vis[(int64_t)v * K + (j >> 6)], (unsigned long long)bit);
        atomicOr((unsigned long long *)&a.fh[(int64_t)v * K + (j >> 6)], (unsigned long long)bit);
        sig[(int64_t)v * W + j] = ST(1);
        if (rp[v + 1] - rp[v] > kLightOut) a.fq0[n - 1 - atomicAdd(&ctl->qh[0], 1)] = v;
        else a.fq0[atomicAdd(&ctl->qn[0], 1)] = v;
        if (INSTR) a.levdeg[(int64_t)j * (a.Lcap + 1)] = (unsigned long long)(rp[v + 1] - rp[v]);
        if (!a.full) {
            const long long q0 = a.lane_off[lane_base + j], q1 = a.lane_off[lane_base + j + 1];
            a.remaining[j] = (int32_t)(q1 - q0);
        }
    }
    if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;

    __shared__ unsigned long long s_nonempty[K];
    __shared__ unsigned long long s_act[K];
    __shared__ unsigned long long s_or[K];
    __shared__ int32_t s_q[kMsBlock / 32][kQueueBuf];
    __shared__ int s_last, s_ctl[3];

    // append the vertices of lanes with `any` (light from the front, heavy from the
    // back); a warp's light ones go out in runs.  Every lane of the warp calls it.
    int held = 0;  // (the same in every lane)
    auto flush = [&](int32_t *q, int32_t *qn, int64_t cap) {
        if (held == 0) return;
        __syncwarp();
        int pos = 0;
        if (lane == 0) pos = atomicAdd(qn, held);
        pos = __shfl_sync(0xffffffffu, pos, 0);
        for (int k = lane; k < held; k += 32)
            if (pos + k < cap) q[pos + k] = s_q[warp_in_block][k];
        __syncwarp();
        held = 0;
    };
    auto append = [&](bool light, bool heavy, int32_t v, int32_t *q, int32_t *qn, int32_t *qh, int64_t cap,
                      int64_t hoff) {
        const unsigned am = __ballot_sync(0xffffffffu, light);
        if (light) s_q[warp_in_block][held + __popc(am & ((1u << lane) - 1u))] = v;
        held += __popc(am);
        if (held > kQueueBuf - 32) flush(q, qn, cap);
        if (heavy) {
            const int64_t pos = hoff + atomicAdd(qh, 1);
            if (pos < cap) q[cap - 1 - pos] = v;
        }
    };

    int L = 0;
    for (;;) {
        // the level's control words, read by one warp of the block (every warp reading
        // them queued 40,000 requests at one L2 line, 8 to 17 us after each barrier)
        if (threadIdx.x < K) {
            s_nonempty[threadIdx.x] = 0ull;
            s_act[threadIdx.x] = ld_relaxed_u64((const uint64_t *)&ctl->active[threadIdx.x]);
        } else if (threadIdx.x == K) {
            s_ctl[0] = (int)ld_relaxed_u32((const uint32_t *)&ctl->push_next);
            s_ctl[1] = (int)ld_relaxed_u32((const uint32_t *)&ctl->qn[L & 1]);
            s_ctl[2] = (int)ld_relaxed_u32((const uint32_t *)&ctl->qh[L & 1]);
        }
        __syncthreads();
        unsigned long long any_act = 0ull;
#pragma unroll
        for (int q = 0; q < K; ++q) any_act |= s_act[q];
        if (!any_act) break;  // (the same in every block)
        if (L + 1 > a.Lcap) {
            if (tid == 0) atomicOr(status, DEV_NEED_LEVELS);
            return false;
        }
        const uint64_t actw = s_act[w];
        const uint64_t *fcur = a.fh + (int64_t)L * nk;
        uint64_t *fnext = a.fh + (int64_t)(L + 1) * nk;
        const int32_t *qcur = (L & 1) ? a.fq1 : a.fq0;
        int32_t *qnext = (L & 1) ? a.fq0 : a.fq1;
        const bool push = s_ctl[0] != 0;
        const int64_t qn = s_ctl[1], qh = s_ctl[2];

        // ---- discover level L+1 (frontier bits only)
        if (push) {
            auto push_edges = [&](int64_t e, int64_t e1, int64_t stride, uint64_t fu) {
                for (; e < e1; e += 4 * stride) {
                    int32_t v[4];
                    uint64_t m[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] = e + q * stride < e1 ? a.col[e + q * stride] - vlo : -1;
#pragma unroll
                    for (int q = 0; q < 4; ++q) m[q] = v[q] >= 0 ? fu & ~__ldcg(&a.vis[(int64_t)v[q] * K + w]) : 0ull;
#pragma unroll
                    for (int q = 0; q < 4; ++q)  // fire-and-forget: collected after the barrier
                        if (m[q]) atomicOr((unsigned long long *)&fnext[(int64_t)v[q] * K + w], (unsigned long long)m[q]);
                }
            };
            // long rows one block each, then one warp per vertex
            for (int64_t r = at.block; r < qh; r += at.blocks) {
                const int32_t u = __ldcg(&qcur[n - 1 - r]);
                push_edges(rp[u] + threadIdx.x / K, rp[u + 1], EB, __ldcg(&fcur[(int64_t)u * K + w]) & actw);
            }
            for (int64_t k = gwarp; k < qn; k += nwarps) {
                const int32_t u = __ldcg(&qcur[k]);
                push_edges(rp[u] + lane / K, rp[u + 1], EW, __ldcg(&fcur[(int64_t)u * K + w]) & actw);
            }
        } else {
            // every vertex with unvisited active lanes; a row's scan stops once each
            // such lane has found a parent
            for (int b = at.block; b < nbig; b += at.blocks) {  // rows above kBigRow: a block each
                const int64_t v = (int64_t)a.big[b] - vlo;
                if (v < 0 || v >= n) continue;  // (the same for the whole block)
                const uint64_t c = actw & ~__ldcg(&a.vis[v * K + w]);
                if (threadIdx.x < K) s_or[threadIdx.x] = 0ull;
                if (!__syncthreads_or(c != 0ull)) continue;
                uint64_t nb = 0ull;
                const int64_t e1 = irp[v + 1];
                for (int64_t e = irp[v] + threadIdx.x / K; e < e1 && (c & ~nb); e += 4 * EB) {
                    int32_t u[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) u[q] = e + q * EB < e1 ? a.icol[e + q * EB] - vlo : -1;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (u[q] >= 0) nb |= __ldcg(&fcur[(int64_t)u[q] * K + w]);
                }
                nb &= c;
                if (nb) atomicOr(&s_or[w], (unsigned long long)nb);
                __syncthreads();
                if (threadIdx.x < K && s_or[threadIdx.x]) fnext[v * K + threadIdx.x] = s_or[threadIdx.x];
                __syncthreads();
            }
            for (int64_t vb = gwarp * GW; vb < n; vb += nwarps * GW) {
                const int64_t v = vb + lane / kGroupLanes;
                uint64_t c = 0ull;
                if (v < n) c = actw & ~__ldcg(&a.vis[v * K + w]);
                const bool some = (__ballot_sync(0xffffffffu, c != 0ull) & gmask) != 0u;
                int64_t e0 = 0, e1 = 0;
                if (some) {
                    e0 = irp[v];
                    e1 = irp[v + 1];
                    if (e1 - e0 > kBigRow) e1 = e0;  // above
                }
                const bool mid = e1 - e0 > kMidRow;
                uint64_t nb = 0ull;
                for (int64_t e = e0 + (lane % kGroupLanes) / K;; e += 4 * SUB) {
                    const bool go = !mid && e < e1 && (SUB > 1 || (c & ~nb) != 0ull);
                    if (!__any_sync(0xffffffffu, go)) break;
                    int32_t u[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) u[q] = go && e + q * SUB < e1 ? a.icol[e + q * SUB] - vlo : -1;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (u[q] >= 0) nb |= __ldcg(&fcur[(int64_t)u[q] * K + w]);
                }
#pragma unroll
                for (int o = K; o < kGroupLanes; o <<= 1) nb |= __shfl_xor_sync(0xffffffffu, nb, o);
                nb &= c;
                if (nb && lane % kGroupLanes < K) fnext[v * K + w] = nb;
                for (unsigned mm = __ballot_sync(0xffffffffu, mid && lane % kGroupLanes == 0); mm; mm &= mm - 1) {
                    const int src = __ffs(mm) - 1;  // a row of middle length, by the whole warp
                    const int64_t f0 = __shfl_sync(0xffffffffu, e0, src), f1 = __shfl_sync(0xffffffffu, e1, src);
                    const uint64_t cm = shfl64(c, src + w);
                    uint64_t mb = 0ull;
                    for (int64_t e = f0 + lane / K; __any_sync(0xffffffffu, e < f1 && (cm & ~mb)); e += 4 * EW) {
                        int32_t u[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) u[q] = e + q * EW < f1 ? a.icol[e + q * EW] - vlo : -1;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (u[q] >= 0) mb |= __ldcg(&fcur[(int64_t)u[q] * K + w]);
                    }
#pragma unroll
                    for (int o = K; o < 32; o <<= 1) mb |= __shfl_xor_sync(0xffffffffu, mb, o);
                    mb &= cm;
                    if (mb && lane < K) fnext[(vb + src / kGroupLanes) * K + w] = mb;
                }
            }
        }
        // full traversal: the counts of level L, whose frontier is settled, meanwhile
        if (a.full && L > 0)
            count_level<K, INSTR, SM>(a, at, n, vlo, irp, L, qcur, qn, qcur + (n - 1), qh, true, nullptr, &ovf, n_s);
        if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;
        if (tid == 0 && L < 32) ctl->lvl_rec[L][4] = globaltimer_ns() - ctl->t_start;

        // ---- settle the new frontier: visited bits, non-empty lanes, the queue of its
        // vertices, the next level's work estimates; the frontier after it starts empty
        {
            uint64_t ne = 0ull;
            unsigned long long fe = 0ull, ue = 0ull;
            uint64_t *f2 = L + 2 <= a.Lcap ? a.fh + (int64_t)(L + 2) * nk : nullptr;
            int32_t *qn_next = &ctl->qn[(L + 1) & 1], *qh_next = &ctl->qh[(L + 1) & 1];
            for (int64_t ib = gwarp * 32; ib < nk; ib += nwarps * 32) {
                const int64_t it = ib + lane, v = it / K;
                uint64_t fn = 0ull, un = 0ull;
                if (it < nk) {
                    fn = __ldcg(&fnext[it]);
                    const uint64_t vv = __ldcg(&a.vis[it]) | fn;
                    if (fn) a.vis[it] = vv;
                    if (f2) f2[it] = 0ull;
                    un = actw & ~vv;
                    ne |= fn;
                }
                const unsigned fm = __ballot_sync(0xffffffffu, fn != 0ull), um = __ballot_sync(0xffffffffu, un != 0ull);
                const unsigned km = (K == 32 ? 0xffffffffu : ((1u << K) - 1u)) << (lane & ~(K - 1));
                bool light = false, heavy = false;
                if (w == 0 && (((fm | um) & km) != 0u)) {
                    const int64_t din = irp[v + 1] - irp[v];
                    ue += (unsigned long long)din * __popc(um & km);
                    if (fm & km) {
                        const int64_t dout = rp[v + 1] - rp[v];
                        fe += (unsigned long long)dout * __popc(fm & km);
                        heavy = din > 32 || dout > kLightOut;
                        light = !heavy;
                        if (INSTR) {
                            n_uv += 1;
                            n_ue += (unsigned long long)dout;
                        }
                    }
                }
                append(light, heavy, (int32_t)v, qnext, qn_next, qh_next, n, 0);
                if (INSTR && fn) {
                    const unsigned long long dg = (unsigned long long)(rp[v + 1] - rp[v]);
                    uint64_t m2 = fn;
                    while (m2) {
                        const int b = __ffsll((long long)m2) - 1;
                        m2 &= m2 - 1;
                        atomicAdd(&a.levdeg[(int64_t)(64 * w + b) * (a.Lcap + 1) + L + 1], dg);
                    }
                }
            }
            flush(qnext, qn_next, n);
            if (ne) atomicOr(&s_nonempty[w], (unsigned long long)ne);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                fe += __shfl_xor_sync(0xffffffffu, fe, off);
                ue += __shfl_xor_sync(0xffffffffu, ue, off);
            }
            if (lane == 0 && fe) atomicAdd(&ctl->fedges[(L + 1) & 1], fe);
            if (lane == 0 && ue) atomicAdd(&ctl->uedges[(L + 1) & 1], ue);
        }
        // settled targets
        if (!a.full) {
            for (long long p = p0 + tid; p < p1; p += nthreads) {
                if (a.found[p] >= 0) continue;
                const int32_t j = a.samp_lane[p] - lane_base;
                const int32_t t = a.samp_t[p] - vlo;
                const int64_t q = (int64_t)t * K + (j >> 6);
                if (((__ldcg(&a.vis[q]) | __ldcg(&fnext[q])) >> (j & 63)) & 1ull) {
                    a.found[p] = L + 1;
                    atomicOr((unsigned long long *)&a.need[q], 1ull << (j & 63));
                    atomicSub(&a.remaining[j], 1);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < K && s_nonempty[threadIdx.x])
            atomicOr(&ctl->nonempty[L & 1][threadIdx.x], s_nonempty[threadIdx.x]);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(&ctl->ticket, 1u) == (uint32_t)at.blocks - 1u;
        }
        __syncthreads();
        if (s_last) {
            // the last block: lanes that go on (a new frontier, and a target left)
            __threadfence();
            if (threadIdx.x < K) s_or[threadIdx.x] = a.full ? ~0ull : 0ull;
            __syncthreads();
            if (!a.full) {
                for (int j = threadIdx.x; j < W; j += blockDim.x) {
                    const unsigned bm = __ballot_sync(0xffffffffu, __ldcg(&a.remaining[j]) > 0);
                    if (lane == 0 && bm) atomicOr(&s_or[j >> 6], (unsigned long long)bm << (j & 32));
                }
                __syncthreads();
            }
            if (threadIdx.x < K) {
                const uint64_t nact = s_act[threadIdx.x] & s_or[threadIdx.x] &
                                      ld_relaxed_u64((const uint64_t *)&ctl->nonempty[L & 1][threadIdx.x]);
                ctl->active[threadIdx.x] = nact;
                ctl->nonempty[L & 1][threadIdx.x] = 0ull;
                // lanes whose counts of level L+1 every vertex would need (a target is left)
                if (!a.full) a.cont[(int64_t)(L + 1) * K + threadIdx.x] = s_act[threadIdx.x] & s_or[threadIdx.x];
            }
            if (threadIdx.x == 0) {
                ctl->ticket = 0;
                ctl->level = L + 1;
                if (L < 32) {
                    ctl->lvl_rec[L][0] = ctl->lvl_rec[L][5] = globaltimer_ns() - ctl->t_start;
                    ctl->lvl_rec[L][1] = (push ? 1ull : 0ull) | (ctl->uedges[L & 1] << 1);
                    ctl->lvl_rec[L][2] = (unsigned long long)(ctl->qn[L & 1] + ctl->qh[L & 1]);
                    ctl->lvl_rec[L][3] = ctl->fedges[L & 1];
                }
                ctl->qn[L & 1] = 0;  // the queue just consumed is refilled at level L+2
                ctl->qh[L & 1] = 0;
                const unsigned long long fe = ctl->fedges[(L + 1) & 1];
                const unsigned long long ue = ctl->uedges[(L + 1) & 1];
                ctl->fedges[L & 1] = 0ull;
                ctl->uedges[L & 1] = 0ull;
                ctl->push_next = a.policy == 1 || (a.policy == 2 && a.push_alpha * (double)fe < (double)ue);
            }
        }
        if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;
        ++L;
    }

    if (!a.full && L > 0) {
        // ---- the vertices whose counts the samples' paths can need
        const bool cone = !FPSIG && L <= (int)__ldg(a.lsafe);
        const int64_t cap = a.ncap;
        int64_t nl = 0, nh = 0;  // entries listed so far (deepest level first)
        auto counts_at = [&](const int32_t *p) -> int2 {  // {light, heavy}, one request a block
            __syncthreads();
            if (threadIdx.x < 2) s_ctl[threadIdx.x] = __ldcg(&p[threadIdx.x]);
            __syncthreads();
            return make_int2(s_ctl[0], s_ctl[1]);
        };
        for (int l = L; cone && l >= 1; --l) {
            const uint64_t *fl = a.fh + (int64_t)l * nk, *fp = a.fh + (int64_t)(l - 1) * nk;
            auto mark_parents = [&](int64_t e, int64_t e1, int64_t stride, uint64_t b) {
                for (; e < e1; e += 4 * stride) {
                    int32_t u[4];
                    uint64_t m[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) u[q] = e + q * stride < e1 ? a.icol[e + q * stride] - vlo : -1;
#pragma unroll
                    for (int q = 0; q < 4; ++q) m[q] = u[q] >= 0 ? b & __ldcg(&fp[(int64_t)u[q] * K + w]) : 0ull;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (m[q]) atomicOr((unsigned long long *)&a.need[(int64_t)u[q] * K + w], (unsigned long long)m[q]);
                }
            };
            for (int b = at.block; l > 1 && b < nbig; b += at.blocks) {  // rows above kBigRow: a block each
                const int64_t v = (int64_t)a.big[b] - vlo;
                if (v < 0 || v >= n) continue;
                const uint64_t bits = __ldcg(&a.need[v * K + w]) & __ldcg(&fl[v * K + w]);
                mark_parents(irp[v] + threadIdx.x / K, bits ? irp[v + 1] : 0, EB, bits);
            }
            for (int64_t ib = gwarp * GW; ib < n; ib += nwarps * GW) {
                const int64_t v = ib + lane / kGroupLanes;
                uint64_t bits = 0ull;
                if (v < n) {
                    bits = __ldcg(&a.need[v * K + w]);
                    if (bits) bits &= __ldcg(&fl[v * K + w]);
                }
                const unsigned bm = __ballot_sync(0xffffffffu, bits != 0ull);
                if (!bm) continue;
                int64_t e0 = 0, e1 = 0;
                if (bm & gmask) {
                    e0 = irp[v];
                    e1 = irp[v + 1];
                }
                const bool rep = (bm & gmask) && lane % kGroupLanes == 0;
                append(rep && e1 - e0 <= 32, rep && e1 - e0 > 32, (int32_t)v, a.nlist + nl, &a.ncnt[2 * l],
                       &a.ncnt[2 * l + 1], cap - nl, nh);
                if (l == 1) continue;
                if (e1 - e0 > kBigRow) e1 = e0;  // above
                const bool mid = e1 - e0 > kMidRow;
                mark_parents(e0 + (lane % kGroupLanes) / K, mid ? e0 : e1, SUB, bits);
                for (unsigned mm = __ballot_sync(0xffffffffu, mid && lane % kGroupLanes == 0); mm; mm &= mm - 1) {
                    const int src = __ffs(mm) - 1;
                    const int64_t f0 = __shfl_sync(0xffffffffu, e0, src), f1 = __shfl_sync(0xffffffffu, e1, src);
                    mark_parents(f0 + lane / K, f1, EW, shfl64(bits, src + w));
                    __syncwarp();
                }
            }
            flush(a.nlist + nl, &a.ncnt[2 * l], cap - nl);
            if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;
            const int2 c = counts_at(a.ncnt + 2 * l);
            nl += c.x;
            nh += c.y;
        }
        // ---- their counts, level by level
        if (cone && nl + nh <= cap) {
            for (int l = 1; l <= L; ++l) {
                const int2 c = counts_at(a.ncnt + 2 * l);
                nl -= c.x;
                nh -= c.y;
                count_level<K, INSTR, SM>(a, at, n, vlo, irp, l, a.nlist + nl, c.x, a.nlist + (cap - 1 - nh), c.y, false,
                                          nullptr, &ovf, n_s);
                if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;
            }
        } else {
            // every vertex of the lanes that go on, and what is needed of the others: the
            // vertices of a level are listed while the level before is counted
            int32_t *dcnt = a.ncnt + 2 * (a.Lcap + 2);
            for (int l = 0; l <= L; ++l) {
                if (l < L) {
                    const uint64_t *fl = a.fh + (int64_t)(l + 1) * nk;
                    const uint64_t cw = cone ? 0ull : __ldcg(&a.cont[(int64_t)(l + 1) * K + w]);
                    int32_t *q = (l & 1) ? a.fq1 : a.fq0, *qc = dcnt + 2 * (l + 1);
                    for (int64_t ib = gwarp * GW; ib < n; ib += nwarps * GW) {
                        const int64_t v = ib + lane / kGroupLanes;
                        uint64_t bits = 0ull;
                        if (v < n) bits = __ldcg(&fl[v * K + w]) & (cw | __ldcg(&a.need[v * K + w]));
                        const bool rep = (__ballot_sync(0xffffffffu, bits != 0ull) & gmask) && lane % kGroupLanes == 0;
                        const int64_t din = rep ? irp[v + 1] - irp[v] : 0;
                        append(rep && din <= 32, rep && din > 32, (int32_t)v, q, &qc[0], &qc[1], n, 0);
                    }
                    flush(q, &qc[0], n);
                }
                if (l > 0) {
                    const int32_t *q = (l & 1) ? a.fq0 : a.fq1;  // listed one round ago
                    const int2 c = counts_at(dcnt + 2 * l);
                    count_level<K, INSTR, SM>(a, at, n, vlo, irp, l, q, c.x, q + (n - 1), c.y, false,
                                              cone ? nullptr : a.cont + (int64_t)l * K, &ovf, n_s);
                }
                if (!grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return false;
            }
        }
    }
    if (__any_sync(0xffffffffu, ovf) && lane == 0) atomicOr(status, SigmaMode<SM>::flag);
    if (INSTR) {
        for (int off = 16; off > 0; off >>= 1) {
            n_s[0] += __shfl_xor_sync(0xffffffffu, n_s[0], off);
            n_s[1] += __shfl_xor_sync(0xffffffffu, n_s[1], off);
            n_uv += __shfl_xor_sync(0xffffffffu, n_uv, off);
            n_ue += __shfl_xor_sync(0xffffffffu, n_ue, off);
        }
        if (lane == 0) {
            atomicAdd(&a.counters[0], n_s[0]);
            atomicAdd(&a.counters[1], n_s[1]);
            atomicAdd(&a.counters[2], n_uv);
            atomicAdd(&a.counters[3], n_ue);
        }
        if (tid == 0) atomicAdd(&a.counters[5], (unsigned long long)L);
    }
    if (a.full) return true;

    if (a.allpaths) {
        // ---- all-paths form (warp per sample): reverse sweep from t over the
        // shortest-path DAG of lane j; tau_v = number of shortest v-t paths
        // (exact integers), and every internal v receives
        // f(v) = sigma_sv tau_v / sigma_st.  Scratch is per warp; entries are
        // valid only where the claim stamp equals this sample's epoch.
        if (gwarp >= a.ap_warps) return true;
        S *tau = reinterpret_cast<S *>(a.ap_tau) + gwarp * n;  // integers, or FP64 beyond 2^53
        int32_t *stamp = a.ap_stamp + gwarp * n;
        int32_t *la = a.ap_list + gwarp * 2 * n;
        int32_t *lb = la + n;
        const unsigned lt = (1u << lane) - 1u;
        for (long long p = p0 + gwarp; p < p1; p += a.ap_warps) {
            const int32_t i = a.sorted_samples[p];
            const int32_t j = a.samp_lane[p] - lane_base;
            const int32_t t = a.samp_t[p] - vlo;
            const int32_t d = __ldcg(&a.found[p]);
            if (lane == 0) {
                if (d < 0) a.kind[i] = 2;
                a.ilen[i] = d < 0 ? 0 : d - 1;
                a.path_off[i] = 0;
            }
            if (d < 2) continue;
            const int32_t ep = ap_epoch + (int32_t)p + 1;  // sample positions are unique in a phase
            const int wj = j >> 6;
            const uint64_t bj = 1ull << (j & 63);
            const double sst = (double)(S)__ldcg(&sig[(int64_t)t * W + j]);
            if (lane == 0) {
                la[0] = t;
                tau[t] = S(1);
                stamp[t] = ep;
            }
            int na = 1;
            __syncwarp();
            for (int L = d - 1; L >= 1; --L) {
                const uint64_t *fL = a.fh + (int64_t)L * nk;
                int nb = 0;
                // claim the predecessors at level L (first claimer zeroes tau)
                for (int q = 0; q < na; ++q) {
                    const int32_t w = __ldcg(&la[q]);
                    const int64_t e0 = irp[w], e1 = irp[w + 1];
                    for (int64_t base = e0; base < e1; base += 32) {
                        const int64_t ee = base + lane;
                        bool mine = false;
                        int32_t pv = 0;
                        if (ee < e1) {
                            pv = a.icol[ee] - vlo;
                            if (__ldcg(&fL[(int64_t)pv * K + wj]) & bj) {
                                mine = atomicExch(&stamp[pv], ep) != ep;
                                if (mine) tau[pv] = S(0);
                            }
                        }
                        const unsigned m = __ballot_sync(0xffffffffu, mine);
                        if (mine) lb[nb + __popc(m & lt)] = pv;
                        nb += __popc(m);
                    }
                }
                __syncwarp();
                // tau_p += tau_w over the DAG edges into level L+1
                for (int q = 0; q < na; ++q) {
                    const int32_t w = __ldcg(&la[q]);
                    const S tw = __ldcg(&tau[w]);
                    const int64_t e0 = irp[w], e1 = irp[w + 1];
                    for (int64_t ee = e0 + lane; ee < e1; ee += 32) {
                        const int32_t pv = a.icol[ee] - vlo;
                        if (__ldcg(&fL[(int64_t)pv * K + wj]) & bj) atomicAdd(&tau[pv], tw);
                    }
                }
                __syncwarp();
                for (int q = lane; q < nb; q += 32) {
                    const int32_t v = __ldcg(&lb[q]);
                    const double f = (double)(S)__ldcg(&sig[(int64_t)v * W + j]) * (double)__ldcg(&tau[v]) / sst;
                    atomicAdd(&a.acc_ap[v + vlo], f);
                }
                __syncwarp();
                int32_t *tmp = la;
                la = lb;
                lb = tmp;
                na = nb;
            }
        }
        return true;
    }

    // ---- backtrack every sample of the batch (warp per sample)
    for (long long p = p0 + gwarp; p < p1; p += nwarps) {
        const int32_t i = a.sorted_samples[p];
        const int32_t j = a.samp_lane[p] - lane_base;
        const int32_t t = a.samp_t[p] - vlo;
        const int32_t s = a.lane_src[lane_base + j] - vlo;
        const int32_t d = __ldcg(&a.found[p]);
        if (INSTR) {
            // edges a top-down truncated BFS from s scans before settling t
            const int32_t lmax = d < 0 ? a.Lcap : d - 1;
            unsigned long long e = 0;
            for (int32_t Lq = lane; Lq <= lmax; Lq += 32) e += a.levdeg[(int64_t)j * (a.Lcap + 1) + Lq];
            for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
            if (lane == 0) {
                atomicAdd(&a.counters[4], e);
                atomicAdd(&a.counters[6], 1ull);
            }
        }
        if (d < 0) {
            if (lane == 0) {
                a.kind[i] = 2;
                a.ilen[i] = 0;
                a.path_off[i] = 0;
            }
            continue;
        }
        const int32_t len = d - 1;
        unsigned long long off = 0;
        if (lane == 0) {
            off = atomicAdd(a.arena_top, (unsigned long long)len);
            a.ilen[i] = len;
            a.path_off[i] = (long long)off;
            if ((int64_t)(off + len) > a.arena_cap) atomicOr(status, DEV_ARENA_OVERFLOW);
        }
        off = __shfl_sync(0xffffffffu, off, 0);
        const bool store = (int64_t)(off + len) <= a.arena_cap;
        const int wj = j >> 6;
        const uint64_t bj = 1ull << (j & 63);
        int32_t w = t;
        int32_t lw = d;
        uint32_t step = 0;
        int32_t k = 0;
        while (w != s) {
            const double target = __dmul_rn(uniform_at(a.seed, (uint64_t)i, a.tag, step),
                                            (double)(S)__ldcg(&sig[(int64_t)w * W + j]));
            const uint64_t *fprev = a.fh + (int64_t)(lw - 1) * nk;
            const int64_t e0 = irp[w], e1 = irp[w + 1];
            S carry = S(0);
            int32_t pick = -1;
            // kBackChunks chunks of 32 candidates in flight (a hub's row is thousands long)
            for (int64_t base = e0; base < e1 && pick < 0; base += 32 * kBackChunks) {
                int32_t pv[kBackChunks];
                S val[kBackChunks];
#pragma unroll
                for (int q = 0; q < kBackChunks; ++q) {
                    const int64_t e = base + 32 * q + lane;
                    pv[q] = e < e1 ? a.icol[e] - vlo : -1;
                }
                bool in[kBackChunks];
#pragma unroll
                for (int q = 0; q < kBackChunks; ++q) in[q] = pv[q] >= 0 && (__ldcg(&fprev[(int64_t)pv[q] * K + wj]) & bj);
#pragma unroll
                for (int q = 0; q < kBackChunks; ++q) val[q] = in[q] ? (S)__ldcg(&sig[(int64_t)pv[q] * W + j]) : S(0);
#pragma unroll
                for (int q = 0; q < kBackChunks; ++q) {
                    if (pick >= 0 || !__any_sync(0xffffffffu, in[q])) continue;
                    // running sums are exact (integers; FP64 sums of integers below 2^53)
                    const S cum = carry + warp_incl_scan<S>(val[q]);
                    const unsigned hit = __ballot_sync(0xffffffffu, val[q] > S(0) && (double)cum >= target);
                    if (hit) pick = __shfl_sync(0xffffffffu, pv[q], __ffs(hit) - 1);
                    carry = __shfl_sync(0xffffffffu, cum, 31);
                }
            }
            if (pick < 0) {
                if (lane == 0) atomicOr(status, DEV_BAD_PATH);
                break;
            }
            if (pick != s) {
                if (lane == 0) {
                    if (store) a.arena[off + k] = pick + vlo;
                    atomicAdd(&a.cnt[pick + vlo], 1ULL);
                }
                ++k;
            }
            w = pick;
            --lw;
            ++step;
        }
    }
    return true;
}

// The persistent launch: every batch of a phase in turn, separated by grid
// barriers.  Batches come from a host plan (many graphs), from the lane count
// the grouping left in device memory (W lanes each, so a phase needs no host
// round trip), or are the single batch given in the arguments.
template <int K, bool INSTR, int SM>
__global__ void __launch_bounds__(kMsBlock, 4) k_msbfs(const __grid_constant__ MsLaunch l) {
    constexpr int W = 64 * K;
    // (the groups' blocks alternate, so that every SM holds some of each)
    const int32_t grp = (int32_t)blockIdx.x % l.groups;
    const Place at{(int32_t)blockIdx.x / l.groups, (int32_t)gridDim.x / l.groups};
    const MsArgs &a = l.g[grp];
    GridBarrier *bar = &a.ctl->bar;
    uint32_t *status = a.status;
    int64_t B = 1;
    long long U = 0;
    if (a.plan) {
        B = a.nplan;
    } else if (a.u_dev) {
        U = *a.u_dev;
        B = (U + W - 1) / W;
    }
    for (int64_t b = grp; b < B; b += l.groups) {
        int32_t lane_base = a.lane_base, nlanes = a.nlanes, vlo = a.vlo;
        int64_t n = a.n;
        if (a.plan) {
            lane_base = a.plan[b].lane_base;
            nlanes = a.plan[b].nlanes;
            vlo = a.plan[b].vlo;
            n = a.plan[b].nr;
        } else if (a.u_dev) {
            lane_base = (int32_t)(b * W);
            nlanes = (int32_t)min((long long)W, U - b * W);
        }
        // the group's previous batch's backtrack reads what this batch's prologue clears
        if (b > grp && !grid_sync(bar, status, a.budget_ns, (uint32_t)at.blocks)) return;
        if (!ms_batch<K, INSTR, SM>(a, at, lane_base, nlanes, vlo, n, a.rp + vlo, a.irp + vlo, a.ap_epoch)) return;
    }
}

// dist/sigma of every lane after a full traversal, source-major output.
template <int K, int SM>
__global__ void k_ms_extract(const uint64_t *fh, const void *sigma_v, int64_t n, int32_t levels, int32_t nsrc,
                             int32_t *dist, double *sig) {
    constexpr int W = 64 * K;
    using ST = typename SigmaMode<SM>::ST;
    const ST *sigma = static_cast<const ST *>(sigma_v);
    const int64_t total = n * (int64_t)nsrc;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += stride) {
        const int64_t j = q / n, v = q % n;
        int32_t d = -1;
        for (int32_t L = 0; L <= levels; ++L) {
            if ((fh[(int64_t)L * n * K + v * K + (j >> 6)] >> (j & 63)) & 1ull) {
                d = L;
                break;
            }
        }
        if (dist) dist[q] = d;
        if (sig) sig[q] = d >= 0 ? (double)sigma[v * W + j] : 0.0;
    }
}

struct GridCache {
    int grid[2][3][4] = {};
};
GridCache g_ms_grid;

template <int K, bool INSTR, int SM>
int ms_grid(percis_ctx *ctx) {
    const int idx = K == 1 ? 0 : K == 2 ? 1 : K == 4 ? 2 : 3;
    int &slot = g_ms_grid.grid[INSTR ? 1 : 0][SM][idx];
    if (slot == 0) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_msbfs<K, INSTR, SM>, kMsBlock, 0);
        slot = std::max(1, per_sm) * ctx->num_sms;
    }
    return slot;
}

template <int K, bool INSTR, int SM>
percis_status launch_ms(percis_ctx *ctx, MsLaunch &l) {
    void *args[] = {&l};
    const int grid = ms_grid<K, INSTR, SM>(ctx) / l.groups * l.groups;
    PERCIS_CUDA(ctx, cudaLaunchCooperativeKernel((const void *)k_msbfs<K, INSTR, SM>, dim3(grid), dim3(kMsBlock),
                                                 args, 0, ctx->stream));
    ctx->launches++;
    return PERCIS_OK;
}

template <int SM>
percis_status launch_ms_k2(percis_ctx *ctx, int K, MsLaunch &a) {
    const bool instr = a.g[0].counters != nullptr;
    switch (K) {
        case 1: return instr ? launch_ms<1, true, SM>(ctx, a) : launch_ms<1, false, SM>(ctx, a);
        case 2: return instr ? launch_ms<2, true, SM>(ctx, a) : launch_ms<2, false, SM>(ctx, a);
        case 4: return instr ? launch_ms<4, true, SM>(ctx, a) : launch_ms<4, false, SM>(ctx, a);
        default: return instr ? launch_ms<8, true, SM>(ctx, a) : launch_ms<8, false, SM>(ctx, a);
    }
}

int ms_grid_for(percis_ctx *ctx, int K) {
    switch (K) {
        case 1: return ms_grid<1, false, 0>(ctx);
        case 2: return ms_grid<2, false, 0>(ctx);
        case 4: return ms_grid<4, false, 0>(ctx);
        default: return ms_grid<8, false, 0>(ctx);
    }
}

percis_status launch_ms_k(percis_ctx *ctx, int K, MsLaunch &a) {
    switch (ctx->sigma_mode) {
        case 0: return launch_ms_k2<0>(ctx, K, a);
        case 1: return launch_ms_k2<1>(ctx, K, a);
        default: return launch_ms_k2<2>(ctx, K, a);
    }
}

// Number of walks of length k that end at a vertex, one step: next[v] += cur[u] over
// the out-edges u -> v, and the largest entry of cur (k = 1: in-degrees) in *wmax.
__global__ void k_walk_step(const int64_t *rp, const int32_t *col, int64_t n, const double *cur, double *next,
                            unsigned long long *wmax) {
    const int lane = threadIdx.x & 31, g = lane >> 3;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long m = 0ull;
    for (int64_t u0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; u0 < n; u0 += warps * 4) {
        const int64_t u = u0 + g;
        const double c = u < n ? cur[u] : 0.0;
        m = max(m, (unsigned long long)__double_as_longlong(c));
        int64_t e0 = 0, e1 = 0;
        if (next && c != 0.0) {
            e0 = rp[u];
            e1 = rp[u + 1];
        }
        const bool big = e1 - e0 > kMidRow;  // by the whole warp below
        for (int64_t e = e0 + (lane & 7); e < e1 && !big; e += 8) atomicAdd(&next[col[e]], c);
        for (unsigned b = __ballot_sync(0xffffffffu, big && (lane & 7) == 0); b; b &= b - 1) {
            const int src = __ffs(b) - 1;
            const int64_t f0 = __shfl_sync(0xffffffffu, e0, src), f1 = __shfl_sync(0xffffffffu, e1, src);
            const double fc = __shfl_sync(0xffffffffu, c, src);
#pragma unroll 4
            for (int64_t e = f0 + lane; e < f1; e += 32) atomicAdd(&next[col[e]], fc);
            __syncwarp();
        }
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0 && m) atomicMax(wmax, m);
}

// in-degrees (the walks of length 1), or the vertices of in-degree > kBigRow
__global__ void k_in_rows(const int64_t *irp, int64_t n, double *deg, int32_t *big, int32_t *nbig) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int64_t d = irp[v + 1] - irp[v];
        if (deg) deg[v] = (double)d;
        else if (d > kBigRow) big[atomicAdd(nbig, 1)] = (int32_t)v;
    }
}

// The levels up to which no path count can reach 2^53: a count at level 4 q + r is at
// most (walks of length 4)^q (walks of length r), each the largest over the vertices.
__global__ void k_safe_levels(const unsigned long long *wmax, int32_t *lsafe) {
    if (threadIdx.x != 0) return;
    double w[5];
    w[0] = 1.0;
    for (int k = 1; k <= 4; ++k) w[k] = __longlong_as_double((long long)wmax[k]);
    double p = 1.0;
    int L = 0;
    while (L < 4096 && p * w[4] < 0x1p52) {
        if (w[4] < 2.0) {  // 0 or 1: the product stays
            L = 4096;
            break;
        }
        p *= w[4];
        L += 4;
    }
    int r = 0;
    while (r < 3 && p * w[r + 1] < 0x1p52) ++r;
    *lsafe = L + r;
}

// The loaded graph's long in-rows, and for sampling phases the levels no count can
// pass 2^53 in, on first use by a batched launch.
percis_status prep_ms_graph(percis_ctx *ctx, bool full) {
    const int64_t n = ctx->n;
    const int64_t *irp = ctx->directed ? ctx->irp.as<int64_t>() : ctx->rp.as<int64_t>();
    const int g = grid_for(ctx, n, 256);
    PERCIS_TRY(ensure(ctx, ctx->ms_big, 64 + sizeof(int32_t) * (ctx->nnz / kBigRow + 1), "long rows"));
    int32_t *nbig = ctx->ms_big.as<int32_t>(), *lsafe = nbig + 1;
    unsigned long long *wmax = reinterpret_cast<unsigned long long *>(nbig + 2);  // [1..4] of five
    if (!ctx->ms_rows_ready) {
        PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->ms_big.p, 0, 64, ctx->stream));
        k_in_rows<<<g, 256, 0, ctx->stream>>>(irp, n, nullptr, nbig + 16, nbig);
        PERCIS_CHECK_LAUNCH(ctx, "long rows");
        ctx->ms_rows_ready = true;
    }
    if (full || ctx->ms_walks_ready) return PERCIS_OK;
    PERCIS_TRY(ensure(ctx, ctx->ms_walks, sizeof(double) * 2 * n, "walk counts"));
    double *wa = ctx->ms_walks.as<double>(), *wb = wa + n;
    k_in_rows<<<g, 256, 0, ctx->stream>>>(irp, n, wa, nullptr, nullptr);
    PERCIS_CHECK_LAUNCH(ctx, "in-degrees");
    for (int k = 1; k <= 4; ++k) {
        if (k < 4) PERCIS_CUDA(ctx, cudaMemsetAsync(wb, 0, sizeof(double) * n, ctx->stream));
        k_walk_step<<<grid_for(ctx, n * 8, 256), 256, 0, ctx->stream>>>(ctx->rp.as<int64_t>(), ctx->col.as<int32_t>(),
                                                                      n, wa, k < 4 ? wb : nullptr, wmax + k);
        PERCIS_CHECK_LAUNCH(ctx, "walk counts");
        std::swap(wa, wb);
    }
    k_safe_levels<<<1, 32, 0, ctx->stream>>>(wmax, lsafe);
    PERCIS_CHECK_LAUNCH(ctx, "walk bound");
    ctx->ms_walks_ready = true;
    return PERCIS_OK;
}

// one group's share of each buffer, a multiple of 256 bytes
size_t group_share(size_t bytes) { return (bytes + 255) / 256 * 256; }

struct MsSizes {
    size_t queue, vis, hist, sigma, list, levels;
};
MsSizes ms_sizes(int W, int Lcap, int64_t n) {
    const size_t K = (size_t)W / 64;
    MsSizes z;
    z.queue = group_share(sizeof(int32_t) * (size_t)n);
    z.vis = group_share(sizeof(uint64_t) * (size_t)n * K);
    z.hist = group_share(sizeof(uint64_t) * (size_t)n * K * (size_t)(Lcap + 1));
    z.sigma = group_share(sizeof(double) * (size_t)n * W);
    z.list = group_share(sizeof(int32_t) * 2 * (size_t)n);
    z.levels = group_share((sizeof(int32_t) * 4 + sizeof(uint64_t) * K) * (size_t)(Lcap + 2));
    return z;
}

percis_status ensure_ms(percis_ctx *ctx, int W, int Lcap, int64_t nr, bool full, int groups) {
    const MsSizes z = ms_sizes(W, Lcap, nr);  // nr: vertices of the largest launch range
    ctx->ms_groups = std::max(ctx->ms_groups, groups);
    PERCIS_TRY(ensure(ctx, ctx->fq0, z.queue * groups, "frontier queue"));
    PERCIS_TRY(ensure(ctx, ctx->fq1, z.queue * groups, "frontier queue"));
    PERCIS_TRY(ensure(ctx, ctx->vis, z.vis * groups, "visited bits"));
    PERCIS_TRY(ensure(ctx, ctx->fhist, z.hist * groups, "frontier history"));
    PERCIS_TRY(ensure(ctx, ctx->sigmaW, z.sigma * groups, "lane sigma"));
    if (!full) {
        PERCIS_TRY(ensure(ctx, ctx->ms_need, z.vis * groups, "needed lanes"));
        PERCIS_TRY(ensure(ctx, ctx->ms_list, z.list * groups, "needed vertices"));
        PERCIS_TRY(ensure(ctx, ctx->ms_levels, z.levels * groups, "level counts"));
    }
    PERCIS_TRY(ensure(ctx, ctx->remaining, sizeof(int32_t) * 512 * groups, "lane remaining"));
    PERCIS_TRY(ensure(ctx, ctx->ms_ctl, sizeof(MsCtl) * groups, "ms ctl"));
    return PERCIS_OK;
}

// Group g's arguments: those of group 0 with its own share of every buffer.
MsArgs group_args(const MsArgs &a0, const MsSizes &z, int g, int64_t ap_n) {
    MsArgs a = a0;
    auto at = [g](auto *p, size_t bytes) {
        using T = decltype(p);
        return reinterpret_cast<T>(reinterpret_cast<char *>(p) + bytes * (size_t)g);
    };
    a.ctl = a0.ctl + g;
    a.fq0 = at(a0.fq0, z.queue);
    a.fq1 = at(a0.fq1, z.queue);
    a.vis = at(a0.vis, z.vis);
    a.fh = at(a0.fh, z.hist);
    a.sigma = reinterpret_cast<char *>(a0.sigma) + z.sigma * (size_t)g;
    a.need = at(a0.need, z.vis);
    a.nlist = at(a0.nlist, z.list);
    a.cont = at(a0.cont, z.levels);
    a.ncnt = at(a0.ncnt, z.levels);
    a.remaining = a0.remaining + 512 * g;
    if (a0.allpaths) {
        const int64_t w = (int64_t)a0.ap_warps * g;
        a.ap_tau = a0.ap_tau + w * ap_n;
        a.ap_stamp = a0.ap_stamp + w * ap_n;
        a.ap_list = a0.ap_list + 2 * w * ap_n;
    }
    return a;
}

struct MsLive {
    percis_ctx *ctx;
    explicit MsLive(percis_ctx *c) : ctx(c) { ctx->ms_live = true; }
    ~MsLive() { ctx->ms_live = false; }
    MsLive(const MsLive &) = delete;
    MsLive &operator=(const MsLive &) = delete;
};

void fill_common(percis_ctx *ctx, MsArgs &a, int Lcap, int K, int64_t nr) {
    a.n = ctx->n;
    a.big_count = ctx->ms_big.as<int32_t>();
    a.lsafe = a.big_count + 1;
    a.big = a.big_count + 16;
    a.need = ctx->ms_need.as<uint64_t>();
    a.nlist = ctx->ms_list.as<int32_t>();
    a.ncap = 2 * nr;
    a.cont = ctx->ms_levels.as<uint64_t>();
    a.ncnt = reinterpret_cast<int32_t *>(a.cont + (size_t)(Lcap + 2) * K);
    a.irp = ctx->directed ? ctx->irp.as<int64_t>() : ctx->rp.as<int64_t>();
    a.icol = ctx->directed ? ctx->icol.as<int32_t>() : ctx->col.as<int32_t>();
    a.vis = ctx->vis.as<uint64_t>();
    a.fh = ctx->fhist.as<uint64_t>();
    a.sigma = ctx->sigmaW.p;
    a.ctl = ctx->ms_ctl.as<MsCtl>();
    a.status = &a.ctl->status;
    a.Lcap = Lcap;
    a.budget_ns = (uint64_t)(ctx->opt.timeout_s * 1e9);
    a.rp = ctx->rp.as<int64_t>();
    a.col = ctx->col.as<int32_t>();
    a.counters = nullptr;
    a.levdeg = nullptr;
    a.fq0 = ctx->fq0.as<int32_t>();
    a.fq1 = ctx->fq1.as<int32_t>();
    a.policy = ctx->opt.direction;
    a.push_alpha = ctx->opt.push_alpha > 0.0 ? ctx->opt.push_alpha : 1.0;
}

}  // namespace

// More batches side by side are an option of speed alone: where an allocation fails, the
// memory they hold goes first (one batch at a time took a quarter of it, and a call that
// fits with that still runs).
bool ms_give_back(percis_ctx *ctx) {
    if (ctx->ms_groups <= 1) return false;
    cudaStreamSynchronize(ctx->stream);
    for (DevBuf *b : {&ctx->fq0, &ctx->fq1, &ctx->vis, &ctx->fhist, &ctx->sigmaW, &ctx->ms_need, &ctx->ms_list,
                      &ctx->ms_levels}) {
        if (b->p) cudaFree(b->p);
        *b = DevBuf{};
    }
    ctx->ms_max_groups = ctx->ms_groups / 2;
    ctx->ms_groups = 0;
    return true;
}

int choose_lanes(percis_ctx *ctx, int64_t n_sources) {
    int W = ctx->opt.lanes;
    if (W != 64 && W != 128 && W != 256 && W != 512) {
        W = 512;
        while (W > 64 && (int64_t)W / 2 >= n_sources) W /= 2;
        // keep the lane sigma array within a modest share of device memory
        size_t free_b = 0, total_b = 0;
        if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess) {
            const double nv = (double)(ctx->multi ? multi_range(ctx) : ctx->n);
            while (W > 64 && nv * W * 8.0 > 0.25 * (double)total_b) W /= 2;
        }
    }
    return W;
}

percis_status batched_phase(percis_ctx *ctx, uint64_t seed, uint32_t tag_path, int64_t count, int64_t n_sources,
                            int64_t *batches) {
    const int W = choose_lanes(ctx, n_sources);
    const int K = W / 64;
    int Lcap = std::max(ctx->levels_alloc, 32);
    // many graphs: a host plan of lane batches over vertex ranges; one graph:
    // W-lane batches over the lane count the grouping left on the device
    std::vector<LaneBatch> plan;
    int64_t nr_max = ctx->n;
    if (ctx->multi) {
        PERCIS_TRY(multi_plan_batches(ctx, n_sources, W, &plan));
        nr_max = 1;
        for (const LaneBatch &lb : plan) nr_max = std::max(nr_max, lb.nr);
    }
    if (!ctx->directed && ctx->vertex_diam > 0) {
        // no undirected shortest path has more than D + 1 edges: enough levels
        // up front (within a 16 GiB frontier history), so deep graphs need no
        // re-runs with a longer history
        const int64_t lmem = (16ll << 30) / std::max<int64_t>(1, nr_max * K * 8) - 1;
        Lcap = (int)std::max<int64_t>(Lcap, std::min<int64_t>(ctx->vertex_diam + 3, std::min<int64_t>(lmem, 1 << 20)));
    }
    const int64_t B = ctx->multi ? (int64_t)plan.size() : (n_sources + W - 1) / W;
    // batches side by side, while their state stays within 24 GiB (fewer where that cannot be
    // had: ms_give_back; the work counters and the level records are those of one at a time)
    int G = 1;
    if (!ctx->opt.instrument) {
        const MsSizes z = ms_sizes(W, Lcap, nr_max);
        const size_t each = 2 * z.queue + 2 * z.vis + z.hist + z.sigma + z.list + z.levels;
        const int most = ctx->ms_max_groups ? std::min(kMaxGroups, ctx->ms_max_groups) : kMaxGroups;
        while (G < most && G + 1 <= B && (size_t)(G + 1) * each <= (24ull << 30)) ++G;
    }
    MsLive live(ctx);
    PERCIS_TRY(prep_ms_graph(ctx, false));
    PERCIS_TRY(ensure_ms(ctx, W, Lcap, nr_max, false, G));
    ctx->levels_alloc = Lcap;
    ctx->lanes_alloc = W;
    PERCIS_TRY(ensure(ctx, ctx->found, sizeof(int32_t) * (count + 1), "found"));
    PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->ms_ctl.p, 0, sizeof(MsCtl) * G, ctx->stream));
    *batches = B;
    MsArgs a{};
    fill_common(ctx, a, Lcap, K, nr_max);
    a.lane_src = ctx->lane_src.as<int32_t>();
    a.lane_off = ctx->lane_off.as<long long>();
    a.samp_t = ctx->samp_t.as<int32_t>();
    a.samp_lane = ctx->samp_lane.as<int32_t>();
    a.sorted_samples = ctx->sorted_samples.as<int32_t>();
    a.found = ctx->found.as<int32_t>();
    a.remaining = ctx->remaining.as<int32_t>();
    a.seed = seed;
    a.tag = tag_path;
    a.kind = ctx->kind.as<int32_t>();
    a.ilen = ctx->ilen.as<int32_t>();
    a.path_off = ctx->path_off.as<long long>();
    a.arena = ctx->arena.as<int32_t>();
    a.arena_top = ctx->arena_top.as<unsigned long long>();
    a.arena_cap = ctx->arena_cap;
    a.cnt = ctx->cnt.as<unsigned long long>();
    a.full = 0;
    if (ctx->opt.instrument) {
        PERCIS_TRY(ensure(ctx, ctx->levdeg, sizeof(unsigned long long) * W * (size_t)(Lcap + 1), "level degrees"));
        a.counters = ctx->counters.as<unsigned long long>();
        a.levdeg = ctx->levdeg.as<unsigned long long>();
    }
    a.allpaths = ctx->opt.estimator == 1;
    if (a.allpaths) {
        // per-warp scratch of 20 n bytes, within a 8 GiB budget
        const int64_t n = nr_max;
        const int64_t per_warp = 20 * n;
        const int64_t warps = (int64_t)ms_grid_for(ctx, K) * (kMsBlock / 32);
        // (a group's warps have their own)
        const int64_t ap_group = std::max<int64_t>(1, std::min<int64_t>(warps, (8ll << 30) / per_warp) / G);
        const int64_t ap_warps = ap_group * G;
        if (ctx->ap_warps != ap_warps || ctx->ap_n != n) {
            ctx->ap_warps = 0;  // (an allocation may fail)
            PERCIS_TRY(ensure(ctx, ctx->ap_tau, sizeof(unsigned long long) * n * ap_warps, "all-paths tau"));
            PERCIS_TRY(ensure(ctx, ctx->ap_stamp, sizeof(int32_t) * n * ap_warps, "all-paths stamps"));
            PERCIS_TRY(ensure(ctx, ctx->ap_list, sizeof(int32_t) * 2 * n * ap_warps, "all-paths lists"));
            PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->ap_stamp.p, 0, sizeof(int32_t) * n * ap_warps, ctx->stream));
            ctx->ap_warps = ap_warps;
            ctx->ap_n = n;
            ctx->ap_epoch = 0;
        }
        if (ctx->ap_epoch > (1 << 30)) {
            PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->ap_stamp.p, 0, sizeof(int32_t) * n * ap_warps, ctx->stream));
            ctx->ap_epoch = 0;
        }
        a.ap_warps = (int32_t)ap_group;
        a.acc_ap = ctx->acc_ap.as<double>();
        a.ap_tau = ctx->ap_tau.as<unsigned long long>();
        a.ap_stamp = ctx->ap_stamp.as<int32_t>();
        a.ap_list = ctx->ap_list.as<int32_t>();
    }
    if (ctx->multi) {
        PERCIS_TRY(ensure(ctx, ctx->plan_dev, sizeof(LaneBatch) * std::max<size_t>(plan.size(), 1), "batch plan"));
        PERCIS_CUDA(ctx, cudaMemcpyAsync(ctx->plan_dev.p, plan.data(), sizeof(LaneBatch) * plan.size(),
                                         cudaMemcpyHostToDevice, ctx->stream));
        a.plan = ctx->plan_dev.as<LaneBatch>();
        a.nplan = (int32_t)plan.size();
    } else {
        a.u_dev = ctx->lane_of_v.as<long long>() + ctx->n;  // number of lanes
    }
    if (a.allpaths) {
        a.ap_epoch = ctx->ap_epoch;
        ctx->ap_epoch += (int32_t)std::min<int64_t>(count, 1 << 30) + 1;
    }
    // every batch of the phase in one persistent launch
    cudaEvent_t e0 = next_event(ctx), e1 = next_event(ctx);
    if (e0) cudaEventRecord(e0, ctx->stream);
    MsLaunch l{};
    l.groups = G;
    {
        const MsSizes z = ms_sizes(W, Lcap, nr_max);
        for (int g = 0; g < G; ++g) l.g[g] = group_args(a, z, g, nr_max);
    }
    PERCIS_TRY(launch_ms_k(ctx, K, l));
    if (e1) cudaEventRecord(e1, ctx->stream);
    return PERCIS_OK;
}

// Full traversal from nsrc <= 512 sources (inspection and exact centrality).
percis_status msbfs_full(percis_ctx *ctx, int32_t nsrc, const int32_t *sources, int32_t *dist, double *sigma) {
    ctx->sigma_mode = 0;
    int W = 64;
    while (W < nsrc) W *= 2;
    const int K = W / 64;
    int Lcap = std::max(ctx->levels_alloc, 32);
    for (int attempt = 0; attempt < 12; ++attempt) {
        MsLive live(ctx);
        PERCIS_TRY(prep_ms_graph(ctx, true));
        percis_status es = ensure_ms(ctx, W, Lcap, ctx->n, true, 1);
        if (es == PERCIS_E_OOM && ms_give_back(ctx)) es = ensure_ms(ctx, W, Lcap, ctx->n, true, 1);
        PERCIS_TRY(es);
        ctx->levels_alloc = Lcap;
        PERCIS_CUDA(ctx, cudaMemsetAsync(ctx->ms_ctl.p, 0, sizeof(MsCtl), ctx->stream));
        MsArgs a{};
        fill_common(ctx, a, Lcap, K, ctx->n);
        a.lane_src = sources;
        a.lane_base = 0;
        a.nlanes = nsrc;
        a.remaining = ctx->remaining.as<int32_t>();
        a.full = 1;
        MsLaunch l{};
        l.groups = 1;
        l.g[0] = a;
        PERCIS_TRY(launch_ms_k(ctx, K, l));
        MsCtl hc;
        PERCIS_CUDA(ctx, cudaMemcpyAsync(&hc, ctx->ms_ctl.p, sizeof(hc), cudaMemcpyDeviceToHost, ctx->stream));
        PERCIS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        if (hc.status & DEV_TIMEOUT) return set_err(ctx, PERCIS_E_TIMEOUT, "batched BFS timed out");
        if (hc.status & DEV_NEED_LEVELS) {
            Lcap *= 2;
            continue;
        }
        if ((hc.status & DEV_SIGMA_WIDE) && ctx->sigma_mode == 0) {
            ctx->sigma_mode = 1;  // counts reached 2^32: redo with 64-bit storage
            continue;
        }
        if ((hc.status & DEV_SIGMA_OVERFLOW) && ctx->sigma_mode == 1) {
            ctx->sigma_mode = 2;  // counts reached 2^53: redo with FP64 sigma
            continue;
        }
        const int levels = hc.level;
        if (!dist && !sigma) return PERCIS_OK;
        const int grid = grid_for(ctx, ctx->n * nsrc, 256);
        const void *sg = ctx->sigmaW.p;
        const uint64_t *fhp = ctx->fhist.as<uint64_t>();
        const int64_t nn = ctx->n;
#define PERCIS_EXTRACT(KK, SMM) \
    k_ms_extract<KK, SMM><<<grid, 256, 0, ctx->stream>>>(fhp, sg, nn, levels, nsrc, dist, sigma)
#define PERCIS_EXTRACT_K(SMM)            \
    switch (K) {                         \
        case 1: PERCIS_EXTRACT(1, SMM); break; \
        case 2: PERCIS_EXTRACT(2, SMM); break; \
        case 4: PERCIS_EXTRACT(4, SMM); break; \
        default: PERCIS_EXTRACT(8, SMM); break; \
    }
        if (ctx->sigma_mode == 0) {
            PERCIS_EXTRACT_K(0);
        } else if (ctx->sigma_mode == 1) {
            PERCIS_EXTRACT_K(1);
        } else {
            PERCIS_EXTRACT_K(2);
        }
#undef PERCIS_EXTRACT_K
#undef PERCIS_EXTRACT
        PERCIS_CHECK_LAUNCH(ctx, "ms extract");
        return PERCIS_OK;
    }
    return set_err(ctx, PERCIS_E_TOO_LARGE, "frontier history exceeded the level cap");
}

}  // namespace percis

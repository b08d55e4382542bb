// Exact percolation centrality (Definition 1): every vertex is a source once.
// Sources go through the batched sigma-BFS in groups of up to 512 lanes (full
// traversals); then, level by level from the deepest, the dependencies of the
// extended Brandes recurrence
//   delta_s(v) = sum over w in out(v) at the next level of
//                (sigma_sv / sigma_sw) (R(x_s - x_w) + delta_s(w))
// are pulled over out-neighbours (one warp per vertex and word of 64 sources,
// two sources a lane), and p(v) = sum_{s != v} delta_s(v) / C_v.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace percis {

namespace {

// The recurrence is carried in y_s(w) = (R(x_s - x_w) + delta_s(w)) / sigma_sw, so
// that delta_s(v) = sigma_sv * (sum of y_s(w) over the next level's w) and y_s(v) =
// R(x_s - x_v) / sigma_sv + that sum: one FP64 addition per DAG edge and source and
// one division per vertex and source (a division per edge held the FP64 pipe, ~64
// cycles a warp operation).  An item is one vertex and one word of 64 sources, so a
// vertex's words run on different warps; a warp loads 32 edges and their frontier
// words at once and takes the edges that matter four at a time.  Above kDepBlockDeg
// edges a whole block shares an item (a hub's 8 words one after the other on one warp,
// edge by edge, set the time of every launch).  Barabasi-Albert n = 3001, m = 4:
// 93.6 -> 1.9 ms in all launches, error against 64 bits 2.8e-16 -> 1.4e-16 relative.
// R(x_s - x_w) is 0 or at least 2^-53 x_s, so y is at least 2^-53 x_s / sigma.  Where that
// could be subnormal (FP64 counts, or states below kTinyState; unscaled, states of 1e-300
// lost digits from counts of 2^27 on and gave 0 from 2^78) a source's y is carried times
// the power of two that takes x_s to [2^60, 2^61), which every term of num takes out
// again, both exactly.
constexpr unsigned long long kTinyState = 123ull << 52;  // 2^-900, as bits
constexpr int kDepBlock = 256;
constexpr int64_t kDepBlockDeg = 128;

// 2^k, |k| < 1023
__device__ __forceinline__ double pow2(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }

// v 2^k, |k| < 2000
__device__ __forceinline__ double scaled(double v, int k) {
    const int lo = max(-1000, min(1000, k));
    const double r = v * pow2(lo);
    return k == lo ? r : r * pow2(k - lo);  // (a second factor for states below 2^-940 alone)
}

// the exponent of source state x's scale
template <int SM>
__device__ __forceinline__ int state_scale(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    if (SM < 2 && b - 1ull >= kTinyState) return 0;  // (x = 0 has no ramp: no scale)
    return 60 - (b >> 52 ? (int)(b >> 52) - 1023 : -1011 - __clzll((long long)b));
}

template <int K, int SM>
__global__ void __launch_bounds__(kDepBlock) k_dependency(int64_t n, const int64_t *rp, const int32_t *col,
                                                          const uint64_t *fh, int32_t L, const void *sigma_v,
                                                          double *y, const double *x, int64_t src0, int32_t nlanes,
                                                          double *num, int kn) {
    constexpr int W = 64 * K;
    constexpr int nwb = kDepBlock / 32;
    using ST = typename SigmaMode<SM>::ST;
    const ST *sigma = static_cast<const ST *>(sigma_v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nwarps = (int64_t)gridDim.x * nwb;
    const int64_t nk = n * K;
    const uint64_t *fL = fh + (int64_t)L * nk;
    const uint64_t *fN = fh + (int64_t)(L + 1) * nk;
    __shared__ double s_part[nwb][64];
    __shared__ int s_hub[nwb];

    // sum of y over the next level's vertices among edges [e, e1), 32 edges every
    // `step`; a0, a1: lanes l and l + 32 of the word
    auto gather = [&](int64_t e, int64_t e1, int64_t step, int w, uint64_t bits, double &a0, double &a1) {
        for (; e < e1; e += step) {
            int32_t c = 0;
            uint64_t m = 0ull;
            if (e + lane < e1) {
                c = __ldg(&col[e + lane]);
                m = bits & __ldg(&fN[(int64_t)c * K + w]);
            }
            unsigned nz = __ballot_sync(0xffffffffu, m != 0ull);
            while (nz) {
                double lo[4], hi[4];
                bool bl[4], bh[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int src = nz ? __ffs(nz) - 1 : 0;
                    const uint64_t f = nz ? shfl64(m, src) : 0ull;
                    const double *row = y + (int64_t)__shfl_sync(0xffffffffu, c, src) * W + 64 * w;
                    nz &= nz - 1;
                    bl[q] = (f >> lane) & 1ull;
                    bh[q] = (f >> (lane + 32)) & 1ull;
                    lo[q] = bl[q] ? __ldcg(row + lane) : 0.0;
                    hi[q] = bh[q] ? __ldcg(row + lane + 32) : 0.0;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (bl[q]) a0 += lo[q];
                    if (bh[q]) a1 += hi[q];
                }
            }
        }
    };
    // the item's results from its sums: y of its sources and its share of num (every lane
    // of the warp calls it)
    auto finish = [&](int64_t v, int w, uint64_t bits, double a0, double a1) {
        double vsum = 0.0;
        const double xv = x[v];
        const int j0 = 64 * w + lane;
        const double xs[2] = {j0 < nlanes ? x[src0 + j0] : 0.0, j0 + 32 < nlanes ? x[src0 + j0 + 32] : 0.0};
        auto half = [&](int h, int k, auto rescale) {
            const int j = j0 + 32 * h;
            if (!((bits >> (lane + 32 * h)) & 1ull) || j >= nlanes) return;
            const double a = h ? a1 : a0, sv = (double)sigma[v * W + j];
            const double ramp = xs[h] - xv;
            if constexpr (rescale) {
                y[v * W + j] = ramp > 0.0 ? a + scaled(ramp, k) / sv : a;
                vsum += scaled(sv * a, -k);
            } else {
                y[v * W + j] = ramp > 0.0 ? a + ramp / sv : a;
                vsum += sv * a;
            }
        };
        // (apart, so that ordinary states' two divisions stay side by side)
        const int k0 = state_scale<SM>(xs[0]), k1 = state_scale<SM>(xs[1]);
        if (__any_sync(0xffffffffu, (k0 | k1) != 0)) {
            half(0, k0, std::true_type{});
            half(1, k1, std::true_type{});
        } else {
            half(0, 0, std::false_type{});
            half(1, 0, std::false_type{});
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) vsum += __shfl_xor_sync(0xffffffffu, vsum, off);
        if (lane == 0 && vsum != 0.0) num[v * kn + w] += vsum;  // (this item's alone)
    };

    // a block's warps take items a grid apart (a vertex's words go to different blocks)
    for (int64_t t = 0; t < nk; t += nwarps) {
        const int64_t it = t + (int64_t)warp * gridDim.x + blockIdx.x;
        const uint64_t bits = it < nk ? fL[it] : 0ull;
        bool hub = false;
        if (bits) {
            const int64_t v = it / K;
            const int w = (int)(it - v * K);
            const int64_t e0 = rp[v], e1 = rp[v + 1];
            hub = e1 - e0 > kDepBlockDeg;
            if (!hub) {
                double a0 = 0.0, a1 = 0.0;
                gather(e0, e1, 32, w, bits, a0, a1);
                finish(v, w, bits, a0, a1);
            }
        }
        if (lane == 0) s_hub[warp] = hub;
        if (!__syncthreads_or(hub)) continue;
        unsigned hubs = 0u;
        for (int q = 0; q < nwb; ++q) hubs |= (unsigned)s_hub[q] << q;
        __syncthreads();  // (s_hub is written again by the next round)
        for (; hubs; hubs &= hubs - 1) {  // the block's hub items, all its warps on each
            const int q = __ffs(hubs) - 1;
            const int64_t hit = t + (int64_t)q * gridDim.x + blockIdx.x;
            const int64_t v = hit / K;
            const int w = (int)(hit - v * K);
            const uint64_t hb = fL[hit];
            double a0 = 0.0, a1 = 0.0;
            gather(rp[v] + 32 * warp, rp[v + 1], kDepBlock, w, hb, a0, a1);
            s_part[warp][lane] = a0;
            s_part[warp][lane + 32] = a1;
            __syncthreads();
            if (warp == 0) {
                a0 = a1 = 0.0;
                for (int p = 0; p < nwb; ++p) {
                    a0 += s_part[p][lane];
                    a1 += s_part[p][lane + 32];
                }
                finish(v, w, hb, a0, a1);
            }
            __syncthreads();
        }
    }
}

__global__ void k_iota(int32_t *a, int64_t lo, int64_t cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) a[i] = (int32_t)(lo + i);
}

// p(v) from the words' shares
__global__ void k_divide(const double *num, int kn, const double *Cv, int64_t n, double *pc) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        double t = 0.0;
        for (int w = 0; w < kn; ++w) t += num[v * kn + w];
        pc[v] = t / Cv[v];
    }
}

// Levels from the deepest (levels is the first empty one) to 1: a source takes
// nothing from itself, so level 0 is not needed.
template <int K>
percis_status dependency_levels(percis_ctx *ctx, int levels, const void *sig, double *y, int64_t src0, int32_t nlanes,
                                double *num, int kn) {
    const int grid = grid_for(ctx, ctx->n * K * 32, kDepBlock);
    auto launch = [&](auto kernel, int L) {
        kernel<<<grid, kDepBlock, 0, ctx->stream>>>(ctx->n, ctx->rp.as<int64_t>(), ctx->col.as<int32_t>(),
                                                    ctx->fhist.as<uint64_t>(), L, sig, y, ctx->x.as<double>(), src0,
                                                    nlanes, num, kn);
    };
    for (int L = levels - 1; L >= 1; --L) {
        if (ctx->sigma_mode == 2) launch(k_dependency<K, 2>, L);
        else if (ctx->sigma_mode == 1) launch(k_dependency<K, 1>, L);
        else launch(k_dependency<K, 0>, L);
        PERCIS_CHECK_LAUNCH(ctx, "dependency");
    }
    return PERCIS_OK;
}

}  // namespace

percis_status exact_pc(percis_ctx *ctx, double *pc) {
    const int64_t n = ctx->n;
    const int W = n >= 512 ? 512 : (n > 256 ? 512 : n > 128 ? 256 : n > 64 ? 128 : 64);
    const int kn = W / 64;  // words per vertex (a narrower last batch uses the first ones)
    PERCIS_TRY(ensure(ctx, ctx->pc_tmp, sizeof(double) * (size_t)n * (W + kn) + sizeof(int32_t) * 512, "exact scratch"));
    double *num = ctx->pc_tmp.as<double>();
    double *y = num + (size_t)n * kn;
    int32_t *src = (int32_t *)(y + (size_t)n * W);
    PERCIS_CUDA(ctx, cudaMemsetAsync(num, 0, sizeof(double) * n * kn, ctx->stream));
    for (int64_t lo = 0; lo < n; lo += W) {
        const int32_t cnt = (int32_t)std::min<int64_t>(W, n - lo);
        k_iota<<<1, 512, 0, ctx->stream>>>(src, lo, cnt);
        PERCIS_CHECK_LAUNCH(ctx, "iota");
        // full traversals; msbfs_full rounds the lane width up to a power of two >= cnt
        PERCIS_TRY(msbfs_full(ctx, cnt, src, nullptr, nullptr));
        MsCtl hc;
        PERCIS_CUDA(ctx, cudaMemcpyAsync(&hc, ctx->ms_ctl.p, sizeof(hc), cudaMemcpyDeviceToHost, ctx->stream));
        PERCIS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        int Wl = 64;
        while (Wl < cnt) Wl *= 2;
        const int levels = hc.level;
        percis_status st;
        switch (Wl / 64) {
            case 1: st = dependency_levels<1>(ctx, levels, ctx->sigmaW.p, y, lo, cnt, num, kn); break;
            case 2: st = dependency_levels<2>(ctx, levels, ctx->sigmaW.p, y, lo, cnt, num, kn); break;
            case 4: st = dependency_levels<4>(ctx, levels, ctx->sigmaW.p, y, lo, cnt, num, kn); break;
            default: st = dependency_levels<8>(ctx, levels, ctx->sigmaW.p, y, lo, cnt, num, kn); break;
        }
        if (st != PERCIS_OK) return st;
    }
    k_divide<<<grid_for(ctx, n, 256), 256, 0, ctx->stream>>>(num, kn, ctx->Cv.as<double>(), n, pc);
    PERCIS_CHECK_LAUNCH(ctx, "divide");
    return PERCIS_OK;
}

}  // namespace percis

// One device step = one correspondence pass of Alg. 1 / Alg. 2 plus the
// decision that follows it, in two kernels:
//   k_nn     double-float transform (Sec. 3, x = R p + t), warm start from the
//            previous correspondence, exact closest target point (Eq. 3), eight
//            lanes per query (group_nn);
//   k_accum  residual, Welsch weight and energy term (Eq. 10, Eq. 12, Eq. 16)
//            and each point's share of the alignment sums in FP64; each block
//            reduces its tile into one record (fixed shared-memory tree, no
//            atomics); the last block reduces all records in a fixed order and
//            runs solver_step() on one warp, so the iteration never leaves
//            the device.
#include <algorithm>

#include "step_common.cuh"

namespace fricp {

namespace {

constexpr int kHardWork = 64;    // rounds and scans (24 on average) above which a ticket is hard, half of it: fairly hard
constexpr int kColdRounds = 4;   // runs of up to 4 x kGroupQ queries per ticket of a first pass (see k_nn)

// Search kernel: persistent warps take runs of Morton-adjacent queries, four
// queries at a time (search_group). Writes prev[i] = this pass's correspondence
// (the next pass's warm start). The first run of a warp is its own index, the
// others come from a counter in the state, so the SMs finish together and the
// queries in flight stay in one window of the Morton order; each query's result
// depends only on the query. A warm pass takes four queries per ticket (runs of
// sixteen left the last tickets running alone: 335 us against 218 us, ellipsoids,
// M = 200,000). The first pass of a large source takes longer runs, whose queries
// start from the result of the one before, once there are 16 tickets per warp
// (eval_pass, M = 200,000: 623 us with single tickets, 635 with runs of two, 695
// with four; fricp_closest_points, M = 1M: 2.27, 1.81, 1.69 ms).
//
// A few queries (outliers about equally far from a large part of the target) walk
// ten times the average, and one that starts late runs on alone. They are the same
// ones from pass to pass, so each pass lists its hard tickets for the next, which
// takes them first. Every ticket is searched once either way. (Ellipsoids, M =
// 200,000: 197 -> 157 us; field, M = 80,000: 91 -> 82 us; thresholds of 48, 96 and
// 160: 158, 161, 169 us.)
//
// Four blocks per SM in FP64 mode (five spill: 156 -> 167 us), five in the others
// (field, M = 80,000, FP32: 80 -> 75-78 us).
template <int PREC>
__global__ void __launch_bounds__(kBlock, PREC == PREC_FP64 ? 4 : 5) k_nn(StepArgs a) {
    __shared__ StepHead h;
    __shared__ float2 s_stk[kBlock / kGroup][kGroupStack];
    if (threadIdx.x == 0) load_head(a.st, h);
    __syncthreads();
    if (h.done) return;
    const bool p2p = !fricp::variant_p2pl(h.variant);
    const int lane = threadIdx.x & 31;
    float2 *stk = s_stk[threadIdx.x / kGroup];
    const unsigned warps = gridDim.x * (kBlock / 32);
    const int step = a.st->device_steps;
    const int rounds = step == 0 ? max(1, min(kColdRounds, (int)(h.M / (16 * kGroupQ * warps)))) : 1;
    // hard tickets listed by the pass before: class 0 from the front of its list, class 1 from the back
    const int T = (int)search_tickets(h.M), par = step & 1;
    const int n0 = a.hard ? a.st->hard_n[par][0] : 0, n1 = a.hard ? a.st->hard_n[par][1] : 0, nh = n0 + n1;
    const int *list = a.hard + (size_t)par * T;
    int *list_out = a.hard + (size_t)(par ^ 1) * T;
    unsigned char *flags = reinterpret_cast<unsigned char *>(a.hard + 2 * (size_t)T);
    const unsigned char *flag = flags + (size_t)par * T;
    unsigned char *flag_out = flags + (size_t)(par ^ 1) * T;
    unsigned u = blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5);
    for (;;) {
        long long e;   // first ticket of this warp's run
        if (u < (unsigned)nh)
            e = u < (unsigned)n0 ? list[u] : list[T - 1 - (int)(u - n0)];
        else
            e = (long long)(u - nh) * rounds;
        if (e >= T) break;
        unsigned nx = 0;
        if (lane == 0) nx = warps + atomicAdd(&a.st->nn_next, 1u);
        if (nh == 0 || u < (unsigned)nh || flag[e] == 0) {
            int seed = -1;
            for (int r = 0; r < rounds && e + r < T; ++r) {
                const int i = (int)(e + r) * kGroupQ + lane / kGroup;
                int work = 0;
                seed = search_group<PREC>(a.ix, a.src, a.prev, h, i, i < h.M, p2p, stk, seed, work);
                if (a.hard && lane == 0) {
                    const int cls = work > kHardWork ? 1 : (work > kHardWork / 2 ? 2 : 0);
                    flag_out[e + r] = (unsigned char)cls;
                    if (cls) {
                        const int pos = atomicAdd(&a.st->hard_n[par ^ 1][cls - 1], 1);
                        list_out[cls == 1 ? pos : T - 1 - pos] = (int)(e + r);
                    }
                }
            }
        }
        u = __shfl_sync(0xffffffffu, nx, 0);
    }
}

// Accumulate kernel: one tile of points per block; the block that completes
// the pass reduces the records and runs the solver step.
template <int VAR, int PREC>
__global__ void __launch_bounds__(kBlock, 3) k_accum(StepArgs a) {
    constexpr int K = VAR ? kSumsP2PL : kSumsP2P;
    __shared__ StepHead h;
    __shared__ double red[K * kRedHalf];
    __shared__ double sS[K];
    __shared__ int s_last;
    if (threadIdx.x == 0) load_head(a.st, h);
    __syncthreads();
    if (h.done) return;
    if (accum_tile<VAR, PREC>(h, a.st, a.ix, a.src, a.prev, a.resid, a.partial, blockIdx.x, gridDim.x, red, &s_last,
                              a.src_nrm))
        finish_pass<K>(h, a.st, a.partial, gridDim.x, a.resid, a.trace, sS, red);
}

// ---------------------------------------------------------------------------
// Correspondence step alone (fricp_closest_points): index (original order) and
// FP64 squared distance, eight lanes per cold query (group_nn).
//
// The caller's points may come in any order, and queries of one warp that are
// far apart walk different parts of the tree: they wait for each other and share
// no lines. Large sets are therefore first dealt into the cells of a 32^3 grid
// over the target's box, in Morton order of the cells (a counting sort: count
// with ranks, scan, scatter); a warp then takes runs of neighbours, and a query
// starts from the result of the one before it in its group. The order inside a
// cell is arbitrary: a result depends only on its query. Against one thread per
// query the serial chain of dependent loads is a fifth as long (M = N = 2,000:
// 114 -> 25 us) and the boxes are read in whole lines (M = 80,000, N = 100,000:
// 1.42 -> 0.2 ms; M = N = 1M: 14.1 -> 1.4 ms).
// ---------------------------------------------------------------------------
constexpr int kCloseBlock = 128;
constexpr int kCellBits = 5;                       // per axis
constexpr int kCells = 1 << (3 * kCellBits);
constexpr int kScanBlock = 1024;

struct ClosestArgs {
    double T[12];
    float lo[3], inv[3];   // target box: cell = (x - lo) * inv, clamped
};

__device__ __forceinline__ unsigned spread5(unsigned v) {   // bits 0..4 to bits 0, 3, .., 12
    v = (v | (v << 8)) & 0x100fu;
    v = (v | (v << 4)) & 0x10c3u;
    return (v | (v << 2)) & 0x1249u;
}

// Cell of every query and its rank among the cell's.
__global__ void __launch_bounds__(256) k_cell_count(ClosestArgs a, const float *__restrict__ p, int64_t m,
                                                    int *__restrict__ hist, int2 *__restrict__ cell) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= m) return;
    const float v[3] = {p[3 * i], p[3 * i + 1], p[3 * i + 2]};
    unsigned c[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float x = fmaf((float)a.T[3 * r], v[0], fmaf((float)a.T[3 * r + 1], v[1],
                             fmaf((float)a.T[3 * r + 2], v[2], (float)a.T[9 + r])));
        c[r] = (unsigned)fminf(fmaxf((x - a.lo[r]) * a.inv[r], 0.0f), (float)((1 << kCellBits) - 1));   // NaN: 0
    }
    const int k = (int)((spread5(c[0]) << 2) | (spread5(c[1]) << 1) | spread5(c[2]));
    cell[i] = make_int2(k, atomicAdd(hist + k, 1));
}

// Exclusive scan of the cell counts, in place (one block).
__global__ void __launch_bounds__(kScanBlock) k_cell_scan(int *hist) {
    __shared__ int s_warp[kScanBlock / 32];
    constexpr int PER = kCells / kScanBlock;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int v[PER], sum = 0;
    int4 *h4 = reinterpret_cast<int4 *>(hist + t * PER);
#pragma unroll
    for (int k = 0; k < PER / 4; ++k) {
        const int4 x = h4[k];
        v[4 * k] = x.x;
        v[4 * k + 1] = x.y;
        v[4 * k + 2] = x.z;
        v[4 * k + 3] = x.w;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) sum += v[k];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        int x = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        s_warp[lane] = x;
    }
    __syncthreads();
    int run = incl - sum + (w > 0 ? s_warp[w - 1] : 0);
#pragma unroll
    for (int k = 0; k < PER / 4; ++k) {
        int4 x;
        x.x = run;
        run += v[4 * k];
        x.y = run;
        run += v[4 * k + 1];
        x.z = run;
        run += v[4 * k + 2];
        x.w = run;
        run += v[4 * k + 3];
        h4[k] = x;
    }
}

__global__ void __launch_bounds__(256) k_cell_scatter(const float *__restrict__ p, int64_t m,
                                                      const int *__restrict__ first, const int2 *__restrict__ cell,
                                                      float4 *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= m) return;
    const int2 c = cell[i];
    out[first[c.x] + c.y] = make_float4(p[3 * i], p[3 * i + 1], p[3 * i + 2], __int_as_float((int)i));
}

// `sorted`: the queries dealt by cell (.w = index), or null to take p as it is.
__global__ void __launch_bounds__(kCloseBlock) k_closest(Index ix, ClosestArgs a, const float *__restrict__ p,
                                                         const float4 *__restrict__ sorted, int64_t m, int rounds,
                                                         int64_t *__restrict__ idx, double *__restrict__ d2) {
    __shared__ float2 s_stk[kCloseBlock / kGroup][kGroupStack];
    const int lane = threadIdx.x & 31;
    const int64_t run = ((int64_t)blockIdx.x * (kCloseBlock / 32) + (threadIdx.x >> 5)) * rounds * kGroupQ;
    int seed = -1;
    for (int r = 0; r < rounds; ++r) {
        if (run + r * kGroupQ >= m) break;   // uniform in the warp
        int64_t i = run + r * kGroupQ + lane / kGroup;
        const bool live = i < m;
        float xh[3] = {0.0f, 0.0f, 0.0f}, xl[3] = {0.0f, 0.0f, 0.0f};
        float4 pp = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float bound = __int_as_float(0x7f800000);
        if (live) {
            float Rh[9], Rl[9], th[3], tl[3];
            for (int k = 0; k < 9; ++k) split_double(a.T[k], Rh[k], Rl[k]);
            for (int k = 0; k < 3; ++k) split_double(a.T[9 + k], th[k], tl[k]);
            if (sorted != nullptr) {
                pp = __ldg(sorted + i);
                i = __float_as_int(pp.w);
            } else {
                pp = make_float4(p[3 * i], p[3 * i + 1], p[3 * i + 2], 0.0f);
            }
            df_transform(Rh, Rl, th, tl, pp, xh, xl);
            if (seed >= 0) bound = point_d2f(xh, xl, __ldg(ix.pts + seed));
        }
        // a non-finite x has no closest point: position 0, as a search that accepts nothing
        const bool finite = isfinite(xh[0] + xh[1] + xh[2]);
        int work = 0;
        const int j = group_nn<PREC_FP64>(ix, xh, xl, bound, s_stk[threadIdx.x / kGroup], live && finite, work);
        if (sorted != nullptr && finite) seed = j;
        if (live && (lane & (kGroup - 1)) == 0) {
            const float4 qq = __ldg(ix.pts + max(j, 0));
            double x[3];
            for (int k = 0; k < 3; ++k) x[k] = fma(a.T[3 * k], (double)pp.x, fma(a.T[3 * k + 1], (double)pp.y, fma(a.T[3 * k + 2], (double)pp.z, a.T[9 + k])));
            const double dx = x[0] - (double)qq.x, dy = x[1] - (double)qq.y, dz = x[2] - (double)qq.z;
            idx[i] = __float_as_int(qq.w);
            d2[i] = dx * dx + dy * dy + dz * dz;
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(32) k_after_init(PairState *st, const double *median) {
    if (threadIdx.x == 0) start_after_init(st, *median);   // nu_max and the first stage, as after a block median
}

}  // namespace

// Blocks of a persistent search kernel: enough to fill every SM at that
// kernel's occupancy, and no more than the work units need (M / per_warp
// queries per warp).
template <typename K>
int persistent_blocks(K kernel, int *cache, int M, int per_warp) {
    if (*cache == 0) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, 0);
        *cache = (sms > 0 ? sms : 152) * (per_sm > 0 ? per_sm : 1);
    }
    const int warps = (M + per_warp - 1) / per_warp;
    const int need = (warps + kBlock / 32 - 1) / (kBlock / 32);
    return need < *cache ? need : *cache;
}

template <int PREC>
void launch_step_prec(const StepArgs &a, int variant, int ntiles, cudaStream_t s, cudaEvent_t mid) {
    static int nb = 0;
    k_nn<PREC><<<persistent_blocks(k_nn<PREC>, &nb, ntiles * kBlock, kGroupQ), kBlock, 0, s>>>(a);
    if (mid) cudaEventRecord(mid, s);
    if (fricp::variant_p2pl(variant))
        k_accum<1, PREC><<<ntiles, kBlock, 0, s>>>(a);
    else
        k_accum<0, PREC><<<ntiles, kBlock, 0, s>>>(a);
}

cudaError_t launch_step(const StepArgs &a, int variant, int prec, int ntiles, cudaStream_t s, cudaEvent_t mid) {
    if (prec == PREC_FP32)
        launch_step_prec<PREC_FP32>(a, variant, ntiles, s, mid);
    else if (prec == PREC_FP16)
        launch_step_prec<PREC_FP16>(a, variant, ntiles, s, mid);
    else
        launch_step_prec<PREC_FP64>(a, variant, ntiles, s, mid);
    counters().launches += 2;
    return cudaGetLastError();
}

// Queries from which on dealing them by cell (about 30 us in five launches) pays.
// Dealt / as they come, in random order: M = 32,000 116 / 89 us, 80,000 199 / 194 us,
// 200,000 462 / 494 us, 999,001 1.42 / 2.74 ms.
constexpr int64_t kSortMin = 1 << 17;

cudaError_t launch_closest(const TargetDev *t, const float *p_dev, int64_t m, const double T[12], int64_t *idx,
                           double *d2, cudaStream_t s) {
    ClosestArgs a;
    for (int k = 0; k < 12; ++k) a.T[k] = T[k];
    for (int r = 0; r < 3; ++r) {
        const float ext = t->hi[r] - t->lo[r];
        a.lo[r] = t->lo[r];
        a.inv[r] = ext > 0.0f ? (float)(1 << kCellBits) / ext : 0.0f;
    }
    const Index ix = make_index(*t);
    // scratch: cell counts, then per query its cell and rank, then the dealt queries
    char *scr = nullptr;
    const size_t cell_b = sizeof(int) * kCells, rank_b = (sizeof(int2) * (size_t)m + 15) / 16 * 16;
    if (m >= kSortMin && pool_alloc(&scr, cell_b + rank_b + sizeof(float4) * (size_t)m, s) != cudaSuccess) {
        cudaGetLastError();   // no room: search them as they come
        scr = nullptr;
    }
    const float4 *sorted = nullptr;
    if (scr != nullptr) {
        int *hist = reinterpret_cast<int *>(scr);
        int2 *cell = reinterpret_cast<int2 *>(scr + cell_b);
        float4 *out = reinterpret_cast<float4 *>(scr + cell_b + rank_b);
        const cudaError_t e = cudaMemsetAsync(hist, 0, cell_b, s);
        if (e != cudaSuccess) {
            cudaFreeAsync(scr, s);
            return e;
        }
        const unsigned nb = (unsigned)((m + 255) / 256);
        k_cell_count<<<nb, 256, 0, s>>>(a, p_dev, m, hist, cell);
        k_cell_scan<<<1, kScanBlock, 0, s>>>(hist);
        k_cell_scatter<<<nb, 256, 0, s>>>(p_dev, m, hist, cell, out);
        counters().launches += 3;
        sorted = out;
    }
    // runs of up to four rounds per warp, while they leave several blocks per slot of the GPU
    const int64_t per_round = kCloseBlock / kGroup;
    const int rounds = sorted != nullptr ? (int)std::min<int64_t>(4, std::max<int64_t>(1, m / (per_round * 4096))) : 1;
    const int64_t per_block = per_round * rounds;
    k_closest<<<(unsigned)((m + per_block - 1) / per_block), kCloseBlock, 0, s>>>(ix, a, p_dev, sorted, m, rounds, idx,
                                                                                 d2);
    counters().launches += 1;
    const cudaError_t e = cudaGetLastError();
    if (scr != nullptr) cudaFreeAsync(scr, s);
    return e;
}

cudaError_t launch_after_init(PairState *st, const double *median_dev, cudaStream_t s) {
    k_after_init<<<1, 32, 0, s>>>(st, median_dev);
    counters().launches += 1;
    return cudaGetLastError();
}

}  // namespace fricp

// Target index build, source preparation and the target's nu_min statistic.
//
// The exact closest-point query (Sec. 3, Eq. 3) runs over a complete binary
// tree of axis-aligned boxes whose leaves are buckets of kLeaf consecutive
// target points in Morton order. The tree is implicit (node i has children 2i
// and 2i+1), so building it is: bounding box -> 30-bit Morton keys -> radix sort
// -> gather into float4 -> leaf boxes -> one launch per eight tree levels, and the
// oriented boxes that the search walks (obb.cuh) for every third level.
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fricp_internal.cuh"
#include "launch_count.cuh"

namespace fricp {

namespace {

constexpr int kRedBlock = 256;

struct BoxPartial {
    float lo[3], hi[3];
    double sum[3];
    int bad;
};

// Per-block min/max/sum in a fixed order; flags NaN/Inf coordinates and normals
// that are not unit length within 1e-3.
__global__ void k_box_partial(const float *__restrict__ x, const float *__restrict__ nrm, int64_t n,
                              BoxPartial *out, int zero_normals_ok) {
    __shared__ float slo[3][kRedBlock], shi[3][kRedBlock];
    __shared__ double ssum[3][kRedBlock];
    __shared__ int sbad;
    if (threadIdx.x == 0) sbad = 0;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    double sm[3] = {0.0, 0.0, 0.0};
    int bad = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        for (int a = 0; a < 3; ++a) {
            const float v = x[3 * i + a];
            if (!isfinite(v)) bad = 1;
            lo[a] = fminf(lo[a], v);
            hi[a] = fmaxf(hi[a], v);
            sm[a] += (double)v;
        }
        if (nrm != nullptr) {
            const float n0 = nrm[3 * i], n1 = nrm[3 * i + 1], n2 = nrm[3 * i + 2];
            const float lf = fmaf(n2, n2, fmaf(n1, n1, n0 * n0));
            if (!(fabsf(lf - 1.0f) <= 1.999e-3f)) {   // not clearly unit (float: exact to 3e-7): the FP64 test decides
                const double a0 = n0, a1 = n1, a2 = n2;
                const double l2 = a0 * a0 + a1 * a1 + a2 * a2;
                if (!(fabs(l2 - 1.0) <= 2e-3) && !(zero_normals_ok && l2 == 0.0)) bad = 1;
            }
        }
    }
    __syncthreads();
    if (bad) atomicOr(&sbad, 1);
    for (int a = 0; a < 3; ++a) {
        slo[a][threadIdx.x] = lo[a];
        shi[a][threadIdx.x] = hi[a];
        ssum[a][threadIdx.x] = sm[a];
    }
    __syncthreads();
    for (int s = kRedBlock / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int a = 0; a < 3; ++a) {
                slo[a][threadIdx.x] = fminf(slo[a][threadIdx.x], slo[a][threadIdx.x + s]);
                shi[a][threadIdx.x] = fmaxf(shi[a][threadIdx.x], shi[a][threadIdx.x + s]);
                ssum[a][threadIdx.x] += ssum[a][threadIdx.x + s];
            }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        BoxPartial r;
        for (int a = 0; a < 3; ++a) {
            r.lo[a] = slo[a][0];
            r.hi[a] = shi[a][0];
            r.sum[a] = ssum[a][0];
        }
        r.bad = sbad;
        out[blockIdx.x] = r;
    }
}

// One block folds the per-block records: thread t takes records t, t+256, ...,
// then a fixed shared-memory tree (deterministic order).
__global__ void k_box_final(const BoxPartial *parts, int nparts, BoxPartial *out, BoxPartial *host_out) {
    __shared__ float slo[3][kRedBlock], shi[3][kRedBlock];
    __shared__ double ssum[3][kRedBlock];
    __shared__ int sbad[kRedBlock];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    double sm[3] = {0.0, 0.0, 0.0};
    int bad = 0;
    for (int b = threadIdx.x; b < nparts; b += kRedBlock) {
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], parts[b].lo[a]);
            hi[a] = fmaxf(hi[a], parts[b].hi[a]);
            sm[a] += parts[b].sum[a];
        }
        bad |= parts[b].bad;
    }
    for (int a = 0; a < 3; ++a) {
        slo[a][threadIdx.x] = lo[a];
        shi[a][threadIdx.x] = hi[a];
        ssum[a][threadIdx.x] = sm[a];
    }
    sbad[threadIdx.x] = bad;
    __syncthreads();
    for (int s = kRedBlock / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            for (int a = 0; a < 3; ++a) {
                slo[a][threadIdx.x] = fminf(slo[a][threadIdx.x], slo[a][threadIdx.x + s]);
                shi[a][threadIdx.x] = fmaxf(shi[a][threadIdx.x], shi[a][threadIdx.x + s]);
                ssum[a][threadIdx.x] += ssum[a][threadIdx.x + s];
            }
            sbad[threadIdx.x] |= sbad[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        BoxPartial r;
        for (int a = 0; a < 3; ++a) {
            r.lo[a] = slo[a][0];
            r.hi[a] = shi[a][0];
            r.sum[a] = ssum[a][0];
        }
        r.bad = sbad[0];
        *out = r;
        *host_out = r;   // pinned host memory: no copy of its own in the stream
    }
}

__device__ __forceinline__ unsigned expand_bits10(unsigned v) {
    v = (v * 0x00010001u) & 0xFF0000FFu;
    v = (v * 0x00000101u) & 0x0F00F00Fu;
    v = (v * 0x00000011u) & 0xC30C30C3u;
    v = (v * 0x00000005u) & 0x49249249u;
    return v;
}

// Keys from the box k_box_final wrote: the host need not wait for it.
__global__ void k_morton(const float *__restrict__ x, int64_t n, const BoxPartial *__restrict__ box,
                         unsigned *__restrict__ code, int *__restrict__ idx) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float c[3];
    for (int a = 0; a < 3; ++a) {
        const float ext = box->hi[a] - box->lo[a];
        c[a] = (x[3 * i + a] - box->lo[a]) * (ext > 0.0f ? 1.0f / ext : 0.0f);
    }
    unsigned k[3];
    for (int a = 0; a < 3; ++a) k[a] = (unsigned)fminf(fmaxf(c[a] * 1024.0f, 0.0f), 1023.0f);
    code[i] = (expand_bits10(k[0]) << 2) | (expand_bits10(k[1]) << 1) | expand_bits10(k[2]);
    idx[i] = (int)i;
}

__global__ void k_gather(const float *__restrict__ x, const float *__restrict__ nrm, const int *__restrict__ order,
                         int64_t n, float4 *__restrict__ pts, float4 *__restrict__ nout) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int o = order[i];
    pts[i] = make_float4(x[3 * (int64_t)o], x[3 * (int64_t)o + 1], x[3 * (int64_t)o + 2], __int_as_float(o));
    if (nrm != nullptr && nout != nullptr)
        nout[i] = make_float4(nrm[3 * (int64_t)o], nrm[3 * (int64_t)o + 1], nrm[3 * (int64_t)o + 2], 0.0f);
}

// Axis-aligned boxes of the tree, 256 nodes of a level per block and the levels
// above them up to eight: the bucket level (LEAF) from the points, a higher one
// from the boxes written by the launch before. One launch per eight levels (a
// launch per level, 15 of them, took 42 us for 500,000 points).
template <bool LEAF>
__global__ void __launch_bounds__(256) k_boxes(const float4 *__restrict__ pts, int64_t n, int size,
                                               float4 *__restrict__ nodes) {
    __shared__ float4 s_lo[256], s_hi[256];
    const int t = threadIdx.x;
    const int l = blockIdx.x * 256 + t;
    float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.0f);
    float4 hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.0f);
    if (l < size) {
        const int64_t node = (int64_t)size + l;
        if (LEAF) {
            const int64_t beg = (int64_t)l * kLeaf;
            const int64_t end = beg + kLeaf < n ? beg + kLeaf : n;
            for (int64_t j = beg; j < end; ++j) {
                const float4 p = pts[j];
                lo.x = fminf(lo.x, p.x); lo.y = fminf(lo.y, p.y); lo.z = fminf(lo.z, p.z);
                hi.x = fmaxf(hi.x, p.x); hi.y = fmaxf(hi.y, p.y); hi.z = fmaxf(hi.z, p.z);
            }
            nodes[2 * node] = lo;
            nodes[2 * node + 1] = hi;
        } else {
            lo = nodes[2 * node];
            hi = nodes[2 * node + 1];
        }
    }
    s_lo[t] = lo;
    s_hi[t] = hi;
    __syncthreads();
    int level = size, first = blockIdx.x * 256;   // nodes of the level, and this block's first
    for (int cnt = 128; cnt >= 1 && level > 1; cnt >>= 1) {
        level >>= 1;
        first >>= 1;
        if (t < cnt) {
            const float4 a0 = s_lo[2 * t], a1 = s_hi[2 * t], b0 = s_lo[2 * t + 1], b1 = s_hi[2 * t + 1];
            lo = make_float4(fminf(a0.x, b0.x), fminf(a0.y, b0.y), fminf(a0.z, b0.z), 0.0f);
            hi = make_float4(fmaxf(a1.x, b1.x), fmaxf(a1.y, b1.y), fmaxf(a1.z, b1.z), 0.0f);
            if (first + t < level) {
                nodes[2 * ((int64_t)level + first + t)] = lo;
                nodes[2 * ((int64_t)level + first + t) + 1] = hi;
            }
        }
        __syncthreads();
        if (t < cnt) {
            s_lo[t] = lo;
            s_hi[t] = hi;
        }
        __syncthreads();
    }
}

// Box of no points: farther than any finite bound.
__device__ __forceinline__ void empty_obb(float4 *o) {
    o[0] = make_float4(1e18f, 1e18f, 1e18f, 0.0f);
    o[8] = make_float4(1.0f, 0.0f, 0.0f, 0.0f);
    o[16] = make_float4(0.0f, 1.0f, 0.0f, 0.0f);
    o[24] = make_float4(0.0f, 0.0f, 1.0f, 0.0f);
}

// Oriented box of every bucket (obb_fit in obb.cuh), the bound obb_d2 tests.
__global__ void k_leaf_obb(const float4 *__restrict__ pts, int64_t n, int L, float4 *__restrict__ obb) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= L) return;
    float4 *o = obb_at(obb, wide_leaf(L) + l);
    const int64_t beg = (int64_t)l * kLeaf;
    const int64_t end = beg + kLeaf < n ? beg + kLeaf : n;
    if (beg >= end) {
        empty_obb(o);
        return;
    }
    float4 box[4];
    obb_fit(pts + beg, (int)(end - beg), box);
    for (int k = 0; k < 4; ++k) o[8 * k] = box[k];
}

// Oriented boxes of the patches three, six and nine levels above the buckets (128,
// 1,024 and 8,192 points), one per NT threads (obb_fit_patch). `shift` = 3, 6 or 9.
template <int NT>
__global__ void __launch_bounds__(256) k_patch_obb(const float4 *__restrict__ pts, int64_t n, int L, int shift,
                                                   const float4 *__restrict__ nodes, float4 *__restrict__ obb) {
    __shared__ float s_red[8][10];
    const int tid = threadIdx.x % NT, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int size = L >> shift;
    const int l = blockIdx.x * (blockDim.x / NT) + threadIdx.x / NT;
    const bool in = l < size;
    const int64_t beg = ((int64_t)l * kLeaf) << shift;
    const int64_t end = beg + (kLeaf << shift) < n ? beg + (kLeaf << shift) : n;
    const int cnt = in && end > beg ? (int)(end - beg) : 0;
    const int node = size + l;
    float4 *o = obb_at(obb, wide_pos(wide_first(L), size) + l);
    // sum or max over the NT threads of a patch, the same in all of them
    auto fold = [&](float *v, int k, bool mx) {
        for (int a = 0; a < k; ++a)
            for (int off = 16; off > 0; off >>= 1) {
                const float x = __shfl_xor_sync(0xffffffffu, v[a], off);
                v[a] = mx ? fmaxf(v[a], x) : v[a] + x;
            }
        if (NT > 32) {
            __syncthreads();
            if (lane == 0)
                for (int a = 0; a < k; ++a) s_red[w][a] = v[a];
            __syncthreads();
            for (int a = 0; a < k; ++a) {
                float x = s_red[0][a];
                for (int ww = 1; ww < 8; ++ww) x = mx ? fmaxf(x, s_red[ww][a]) : x + s_red[ww][a];
                v[a] = x;
            }
        }
    };
    float c[3] = {0.0f, 0.0f, 0.0f};
    if (cnt > 0) {
        const float4 lo = nodes[2 * node], hi = nodes[2 * node + 1];
        c[0] = 0.5f * lo.x + 0.5f * hi.x;
        c[1] = 0.5f * lo.y + 0.5f * hi.y;
        c[2] = 0.5f * lo.z + 0.5f * hi.z;
    }
    float4 box[4];
    obb_fit_patch(pts + beg, cnt, c, tid, NT, fold, box);
    if (!in || tid != 0) return;
    if (cnt == 0) {
        empty_obb(o);
        return;
    }
    for (int k = 0; k < 4; ++k) o[8 * k] = box[k];
}

// The levels above (few, large nodes): the axis-aligned box in the same form.
// The first level also fills the empty positions before it (`pad`).
__global__ void k_level_obb(const float4 *__restrict__ nodes, int L, int size, int pad, float4 *__restrict__ obb) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < pad) empty_obb(obb_at(obb, l));
    if (l >= size) return;
    const int node = size + l;
    float4 *o = obb_at(obb, wide_pos(wide_first(L), size) + l);
    const float4 lo = nodes[2 * node], hi = nodes[2 * node + 1];
    if (!(lo.x <= hi.x)) {
        empty_obb(o);
        return;
    }
    const float c[3] = {0.5f * lo.x + 0.5f * hi.x, 0.5f * lo.y + 0.5f * hi.y, 0.5f * lo.z + 0.5f * hi.z};
    const float l3[3] = {lo.x, lo.y, lo.z}, h3[3] = {hi.x, hi.y, hi.z};
    float h[3];
    double r2 = 0.0;
    for (int k = 0; k < 3; ++k) {
        const double e = fmax((double)h3[k] - c[k], (double)c[k] - l3[k]);
        r2 += e * e;
        h[k] = (float)e;
    }
    const double r = sqrt(r2);
    for (int k = 0; k < 3; ++k) h[k] = f32_round_up((double)h[k] * (1.0 + 1e-6) + 2e-6 * r + 1e-37);
    o[0] = make_float4(c[0], c[1], c[2], h[0]);
    o[8] = make_float4(1.0f, 0.0f, 0.0f, h[1]);
    o[16] = make_float4(0.0f, 1.0f, 0.0f, h[2]);
    o[24] = make_float4(0.0f, 0.0f, 1.0f, f32_round_up(r));
}

// Six nearest target points of every target point, the point itself excluded
// (duplicates at distance zero count), ordered by (exact FP64 squared distance,
// original index). Per point: the median of the six distances (Sec. 4.3) and,
// with normals, the median of the six distances to the point's tangent plane
// (Sec. 5); the median of six is the mean of the 3rd and 4th smallest.
//
// One warp per query point (tiny targets and ties): the query's own bucket
// is scanned first, then the siblings of its path to the root and what they
// open, two tree levels per round; lanes test boxes and bucket points in
// parallel. Pruning is in float: a box or candidate is skipped only when its
// float squared distance, shrunk by kShrink (far more than the float rounding
// of either), exceeds the current sixth-best FP64 distance rounded up to float.
// Every point that can enter the six gets its exact FP64 distance, and the six
// (kept identical in every lane) are merged one at a time in a fixed order, so
// the selection and the medians are exact.
struct Best6 {
    double d[6];
    int o[6], j[6];
    float bound;   // d[5] rounded up to float
};

// Insert (d, o, j) into the six kept in (d, o) order, if it belongs there. Fully
// unrolled with constant indices, so the six stay in registers: slot s takes
// the old entry s - 1 while that one orders after the newcomer, the newcomer at
// the first slot where it does not, and slot 0 if it orders before all.
__device__ __forceinline__ void best6_insert(Best6 &b, double d, int o, int j) {
    if (!(d < b.d[5] || (d == b.d[5] && o < b.o[5]))) return;
    bool done = false;
#pragma unroll
    for (int s = 5; s >= 1; --s) {
        const bool after = !done && (b.d[s - 1] > d || (b.d[s - 1] == d && b.o[s - 1] > o));
        const bool put = !done && !after;
        b.d[s] = after ? b.d[s - 1] : (put ? d : b.d[s]);
        b.o[s] = after ? b.o[s - 1] : (put ? o : b.o[s]);
        b.j[s] = after ? b.j[s - 1] : (put ? j : b.j[s]);
        done = done || put;
    }
    if (!done) {
        b.d[0] = d;
        b.o[0] = o;
        b.j[0] = j;
    }
    b.bound = __double2float_ru(b.d[5]);
}

// Offers bucket na's points (lanes 0-15) and, if `two`, bucket nb's (lanes
// 16-31) to the six; the point i itself is skipped.
__device__ __forceinline__ void knn6_scan(const Index &ix, int i, const float xq[3], Best6 &b, int na, int nb,
                                          bool two) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    bool cand = false;
    double d = 0.0;
    int o = 0, j = -1;
    if (lane < 16 || two) {
        j = ((lane < 16 ? na : nb) - ix.L) * kLeaf + (lane & 15);
        if (j < ix.n && j != i) {
            const float4 q = __ldg(ix.pts + j);
            const float fx = q.x - xq[0], fy = q.y - xq[1], fz = q.z - xq[2];
            if (fmaf(fz, fz, fmaf(fy, fy, fx * fx)) * kShrink <= b.bound) {
                const double a0 = (double)q.x - (double)xq[0], a1 = (double)q.y - (double)xq[1],
                             a2 = (double)q.z - (double)xq[2];
                d = a0 * a0 + a1 * a1 + a2 * a2;
                o = __float_as_int(q.w);
                cand = true;
            }
        }
    }
    unsigned cm = __ballot_sync(FULL, cand);
    while (cm) {   // merge in lane order: every lane applies the same insertions
        const int src = __ffs(cm) - 1;
        cm &= cm - 1u;
        const double dv = __shfl_sync(FULL, d, src);
        const int ov = __shfl_sync(FULL, o, src), jv = __shfl_sync(FULL, j, src);
        best6_insert(b, dv, ov, jv);
    }
}

// Returns false if the stack would overflow.
__device__ bool warp_knn6(const Index &ix, int i, const float xq[3], Best6 &b, int *stk) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float zero[3] = {0.0f, 0.0f, 0.0f};
    for (int s = 0; s < 6; ++s) {
        b.d[s] = INFINITY;
        b.o[s] = 0x7fffffff;
        b.j[s] = -1;
    }
    b.bound = INFINITY;
    int depth = 0;
    while ((1 << depth) < ix.L) ++depth;
    // the query's own bucket and its sibling bucket first: a tight bound early
    const int start = ix.L + i / kLeaf;
    knn6_scan(ix, i, xq, b, start, start ^ 1, depth > 0);   // a one-bucket tree has no sibling
    int sp;
    {
        int c = 0;
        bool pass = false;
        if (lane < depth - 1) {   // the sibling of the path node at level lane + 1 (the bucket level is done)
            c = (start >> (depth - 1 - lane)) ^ 1;
            pass = box_d2(__ldg(ix.nodes + 2 * c), __ldg(ix.nodes + 2 * c + 1), xq, zero) * kShrink <= b.bound;
        }
        const unsigned m = __ballot_sync(FULL, pass);
        if (pass) stk[__popc(m & below)] = c;
        sp = __popc(m);
    }
    __syncwarp();
    const int leaf_parent_level = depth - 1;
    while (sp > 0) {
        const int k = min(32, sp);
        const int node = (lane < k) ? stk[sp - 1 - lane] : 0;
        sp -= k;
        __syncwarp();
        int c[4] = {0, 0, 0, 0};
        bool ok[4] = {false, false, false, false};
        bool leaf_ok = false;
        if (node != 0) {
            if (node < ix.L) {
                const int level = 31 - __clz(node);
                if (level < leaf_parent_level) {
                    const float4 *bx = ix.nodes + 8 * node;
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        c[g] = 4 * node + g;
                        ok[g] = box_d2(__ldg(bx + 2 * g), __ldg(bx + 2 * g + 1), xq, zero) * kShrink <= b.bound;
                    }
                } else {
                    const float4 *bx = ix.nodes + 4 * node;
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        c[g] = 2 * node + g;
                        ok[g] = box_d2(__ldg(bx + 2 * g), __ldg(bx + 2 * g + 1), xq, zero) * kShrink <= b.bound;
                    }
                }
            } else {
                leaf_ok = box_d2(__ldg(ix.nodes + 2 * node), __ldg(ix.nodes + 2 * node + 1), xq, zero) * kShrink
                              <= b.bound &&
                          obb_d2(obb_at(ix.obb, node - ix.L + ix.leaf0), xq, zero) * kObbShrink <= b.bound;
            }
        }
        int base = sp;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const unsigned mg = __ballot_sync(FULL, ok[g]);
            if (base + __popc(mg) > kWarpStack) return false;
            if (ok[g]) stk[base + __popc(mg & below)] = c[g];
            base += __popc(mg);
        }
        sp = base;
        unsigned lm = __ballot_sync(FULL, leaf_ok);
        while (lm) {   // two buckets per pass: lanes 0-15 and 16-31
            const int la = __ffs(lm) - 1;
            lm &= lm - 1u;
            int lb = la;
            bool two = false;
            if (lm) {
                lb = __ffs(lm) - 1;
                lm &= lm - 1u;
                two = true;
            }
            const int na = __shfl_sync(FULL, node, la), nb = __shfl_sync(FULL, node, lb);
            knn6_scan(ix, i, xq, b, na, nb, two);
        }
        __syncwarp();
    }
    return true;
}

constexpr int kKnnBlock = 128;

// Per-point statistics of point i from its six nearest (Sec. 4.3, Sec. 5): the
// median of the six distances and, with normals, of the six distances to the
// point's tangent plane (the median of six: the mean of the 3rd and 4th).
__device__ void write_knn6_stats(const Index &ix, int i, const float xq[3], const Best6 &b, double *stat_d,
                                 double *stat_h) {
    const double x0 = xq[0], x1 = xq[1], x2 = xq[2];
    stat_d[i] = 0.5 * (sqrt(b.d[2]) + sqrt(b.d[3]));
    if (stat_h != nullptr) {
        const float4 ni = ix.nrm[i];
        double h[6];
        for (int s = 0; s < 6; ++s) {
            if (b.j[s] < 0) {
                h[s] = INFINITY;
                continue;
            }
            const float4 q = ix.pts[b.j[s]];
            h[s] = fabs(((double)q.x - x0) * ni.x + ((double)q.y - x1) * ni.y + ((double)q.z - x2) * ni.z);
        }
        for (int a = 1; a < 6; ++a) {   // insertion sort of six values
            const double v = h[a];
            int c = a - 1;
            while (c >= 0 && h[c] > v) {
                h[c + 1] = h[c];
                --c;
            }
            h[c + 1] = v;
        }
        stat_h[i] = 0.5 * (h[2] + h[3]);
    }
}

__global__ void __launch_bounds__(kKnnBlock) k_knn6_stats(Index ix, double *__restrict__ stat_d,
                                                          double *__restrict__ stat_h, int *__restrict__ overflow) {
    __shared__ int s_stk[kKnnBlock / 32][kWarpStack];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int wpb = kKnnBlock / 32;
    for (int i = blockIdx.x * wpb + w; i < ix.n; i += gridDim.x * wpb) {
        const float4 qi = __ldg(ix.pts + i);
        const float xq[3] = {qi.x, qi.y, qi.z};
        Best6 b;
        if (!warp_knn6(ix, i, xq, b, s_stk[w])) {
            if (lane == 0) *overflow = 1;
            continue;
        }
        if (lane == 0) write_knn6_stats(ix, i, xq, b, stat_d, stat_h);
    }
}

// Six-neighbour statistics by tiles: a warp takes the 32 Morton-consecutive
// target points of buckets 2g and 2g + 1, one per lane, each lane keeping its
// own nearest.
//   1. Each lane offers the tile's other 31 points to its list: its sixth
//      distance is then an upper bound of its true sixth distance, and R, the
//      largest over the lanes, bounds them all.
//   2. Every point within sqrt(R) of some lane's point lies within sqrt(R) of
//      the two buckets' common box (the tree node above them), so the buckets
//      whose box is within that distance of that box (walk from the node's path
//      siblings, box-to-box distance, kShrink slack) hold every candidate.
//   3. Each lane offers the points of those buckets to its list, pruning with
//      its own sixth distance.
// The lists rank by float distance (tile_near7, seven entries); a tile in which
// the seventh cannot be told from the sixth repeats it with FP64 distances
// (tile_knn6: Best6, the order and float pre-test of warp_knn6). A tile whose
// bucket list does not fit (scattered, or fewer than seven points in it) is left
// to k_knn6_rest, which gives each of its points a warp.
// With every distance and comparison in FP64, and the left-over tiles searched
// point by point by their own warp, the FP64 pipe and a few such warps were the
// bound (ellipsoids, 500,000 points: 2.48 ms); now 0.34 ms, and 0.11 ms for the
// rest. What bounds it: issue slots (55% busy, 17 of 32 lanes at work) and the
// candidates' loads, with the busiest SM 30% above the average.
constexpr int kKnnCand = 192;   // candidate buckets per tile

__device__ __forceinline__ float box_box_d2(float4 alo, float4 ahi, float4 blo, float4 bhi) {
    const float gx = fmaxf(fmaxf(alo.x - bhi.x, blo.x - ahi.x), 0.0f);
    const float gy = fmaxf(fmaxf(alo.y - bhi.y, blo.y - ahi.y), 0.0f);
    const float gz = fmaxf(fmaxf(alo.z - bhi.z, blo.z - ahi.z), 0.0f);
    return fmaf(gz, gz, fmaf(gy, gy, gx * gx));
}

__device__ __forceinline__ void knn6_offer_own(Best6 &b, float4 q, const float xq[3], int j) {
    const float fx = q.x - xq[0], fy = q.y - xq[1], fz = q.z - xq[2];
    if (fmaf(fz, fz, fmaf(fy, fy, fx * fx)) * kShrink <= b.bound) {
        const double a0 = (double)q.x - (double)xq[0], a1 = (double)q.y - (double)xq[1],
                     a2 = (double)q.z - (double)xq[2];
        best6_insert(b, a0 * a0 + a1 * a1 + a2 * a2, __float_as_int(q.w), j);
    }
}

// Buckets within sqrt(R) of the box of tile g (node P above buckets 2g, 2g + 1),
// in cand; their number, or -1 when the list or the walk's stack would overflow.
__device__ __forceinline__ int tile_candidates(const Index &ix, int g, float R, int *stk, int *cand) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int depth = 0;
    while ((1 << depth) < ix.L) ++depth;
    const int P = (ix.L >> 1) + g;
    const float4 glo = __ldg(ix.nodes + 2 * P), ghi = __ldg(ix.nodes + 2 * P + 1);
    int sp = 0, nc = 0;
    {
        int c = 0;
        bool pass = false;
        if (lane < depth - 1) {   // siblings of P's path, from the root's children down
            c = (P >> (depth - 2 - lane)) ^ 1;
            pass = box_box_d2(__ldg(ix.nodes + 2 * c), __ldg(ix.nodes + 2 * c + 1), glo, ghi) * kShrink <= R;
        }
        const unsigned m = __ballot_sync(FULL, pass);
        if (pass) stk[__popc(m & below)] = c;
        sp = __popc(m);
    }
    __syncwarp();
    while (sp > 0) {
        const int k = min(32, sp);
        const int node = (lane < k) ? stk[sp - 1 - lane] : 0;
        sp -= k;
        __syncwarp();
        int c[4] = {0, 0, 0, 0};
        bool ok[4] = {false, false, false, false};
        bool leaf = false;
        if (node != 0) {
            if (node < ix.L) {
                const int level = 31 - __clz(node);
                if (level < depth - 1) {
                    const float4 *bx = ix.nodes + 8 * node;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        c[q] = 4 * node + q;
                        ok[q] = box_box_d2(__ldg(bx + 2 * q), __ldg(bx + 2 * q + 1), glo, ghi) * kShrink <= R;
                    }
                } else {
                    const float4 *bx = ix.nodes + 4 * node;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        c[q] = 2 * node + q;
                        ok[q] = box_box_d2(__ldg(bx + 2 * q), __ldg(bx + 2 * q + 1), glo, ghi) * kShrink <= R;
                    }
                }
            } else {
                leaf = true;   // tested when it was pushed
            }
        }
        const unsigned lm = __ballot_sync(FULL, leaf);
        if (nc + __popc(lm) > kKnnCand) return -1;
        if (leaf) cand[nc + __popc(lm & below)] = node;
        nc += __popc(lm);
        int base = sp;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned mq = __ballot_sync(FULL, ok[q]);
            if (base + __popc(mq) > kWarpStack - kKnnCand) return -1;
            if (ok[q]) stk[base + __popc(mq & below)] = c[q];
            base += __popc(mq);
        }
        sp = base;
        __syncwarp();
    }
    return nc;
}

// Returns false when the candidate list or the walk's stack would overflow.
__device__ __noinline__ bool tile_knn6(const Index &ix, int g, int i, bool live, const float xq[3], Best6 &b, int *stk,
                          int *cand) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int s = 0; s < 6; ++s) {
        b.d[s] = INFINITY;
        b.o[s] = 0x7fffffff;
        b.j[s] = -1;
    }
    b.bound = INFINITY;
    const int i0 = 32 * g;
    const float4 mine = live ? __ldg(ix.pts + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int k = 1; k < 32; ++k) {   // 1. the tile's own points, nearest in Morton order first
        const int off = (k & 1) ? (k + 1) >> 1 : -(k >> 1);   // +1, -1, +2, -2, ..., -15, +16
        const int t = (lane + off) & 31;
        float4 q;
        q.x = __shfl_sync(FULL, mine.x, t);
        q.y = __shfl_sync(FULL, mine.y, t);
        q.z = __shfl_sync(FULL, mine.z, t);
        q.w = __shfl_sync(FULL, mine.w, t);
        if (live && i0 + t < ix.n) knn6_offer_own(b, q, xq, i0 + t);
    }
    float R = live ? b.bound : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) R = fmaxf(R, __shfl_xor_sync(FULL, R, o));
    if (!(R < INFINITY)) return false;
    const int nc = tile_candidates(ix, g, R, stk, cand);   // 2.
    if (nc < 0) return false;
    // 3. every lane offers the candidates' points to its own six, bucket by
    //    bucket; a lane whose own bound the bucket's boxes exceed skips it, and
    //    the warp skips a bucket no lane needs
    const float zero[3] = {0.0f, 0.0f, 0.0f};
    for (int k = 0; k < nc; ++k) {
        const int c = cand[k];
        bool need = false;
        if (live)
            need = box_d2(__ldg(ix.nodes + 2 * c), __ldg(ix.nodes + 2 * c + 1), xq, zero) * kShrink <= b.bound &&
                   obb_d2(obb_at(ix.obb, c - ix.L + ix.leaf0), xq, zero) * kObbShrink <= b.bound;
        if (!__any_sync(FULL, need)) continue;
        const int beg = (c - ix.L) * kLeaf;
        const int end = min(beg + kLeaf, ix.n);
        if (need)
            for (int j = beg; j < end; ++j) knn6_offer_own(b, __ldg(ix.pts + j), xq, j);
    }
    __syncwarp();
    return true;
}

// The 32 nearest points of a query by float distance, lane s the s-th.
struct NearK {
    float d;
    int j;
    float bound;   // upper bound of the K-th distance
    float spill;   // smallest distance that left the list
};

// Compare-exchange with lane ^ s, the smaller distance to the lower lane when
// `up`. Equal distances stay where they are, in both lanes.
__device__ __forceinline__ void near_exchange(float &d, int &j, int s, bool up) {
    const unsigned FULL = 0xffffffffu;
    const float od = __shfl_xor_sync(FULL, d, s);
    const int oj = __shfl_xor_sync(FULL, j, s);
    const bool keep_min = ((threadIdx.x & s) == 0) == up;
    if (keep_min ? od < d : od > d) {
        d = od;
        j = oj;
    }
}

__device__ __forceinline__ void near_scan(const Index &ix, const float xq[3], int skip, NearK &t, int K, int na,
                                          int nb, bool two) {
    const unsigned FULL = 0xffffffffu;
    const float INF = __int_as_float(0x7f800000);
    const int lane = threadIdx.x & 31;
    float d = INF;
    int j = -1;
    if (lane < 16 || two) {
        j = ((lane < 16 ? na : nb) - ix.L) * kLeaf + (lane & 15);
        if (j < ix.n && j != skip) {
            const float4 q = __ldg(ix.pts + j);
            const float fx = q.x - xq[0], fy = q.y - xq[1], fz = q.z - xq[2];
            d = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
            if (!(d * kShrink <= t.bound)) d = INF;
        }
    }
    unsigned cm = __ballot_sync(FULL, d < INF);
    if (cm == 0u) return;
    if (__popc(cm) <= 6) {   // a few: insert one by one
        while (cm) {
            const int src = __ffs(cm) - 1;
            cm &= cm - 1u;
            const float dv = __shfl_sync(FULL, d, src);
            const int jv = __shfl_sync(FULL, j, src);
            const unsigned gm = __ballot_sync(FULL, t.d > dv);
            const float ud = __shfl_up_sync(FULL, t.d, 1);
            const int uj = __shfl_up_sync(FULL, t.j, 1);
            t.spill = fminf(t.spill, gm == 0u ? dv : __shfl_sync(FULL, t.d, 31));
            if (gm == 0u) continue;
            const int pos = __ffs(gm) - 1;
            if (lane >= pos) {
                t.d = lane == pos ? dv : ud;
                t.j = lane == pos ? jv : uj;
            }
        }
    } else {   // sort the 32 descending, merge with the ascending list, keep the lower half
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
            for (int o = k >> 1; o > 0; o >>= 1) near_exchange(d, j, o, (lane & k) != 0);
        float out = t.d > d ? t.d : d;
        if (d < t.d) {
            t.d = d;
            t.j = j;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) near_exchange(t.d, t.j, o, true);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) out = fminf(out, __shfl_xor_sync(FULL, out, o));
        t.spill = fminf(t.spill, out);
    }
    t.bound = fminf(t.bound, __shfl_sync(FULL, t.d, K - 1));
}

// The K nearest of point i in lanes 0 .. K-1 (point `skip` left out), all of them
// within the squared distance `bound` (INF if none is known). Returns 0 if they
// are the exact K, 1 if float distances cannot tell, 2 if the stack would overflow.
//
// The point's bucket and its sibling are scanned first; then the walk of group_nn
// over the oriented boxes, by the whole warp: up to four nodes a round, eight
// children each, and the buckets within the bound two at a time, nearest first.
// Squares below it lose bits to underflow, and the float distances their relative
// error of 4e-7: such a list is left to FP64 (points about 1e-18 apart; also seven
// copies of a point).
constexpr float kNearMin = 1e-36f;
constexpr int kNearStack = kWarpStack;   // a round replaces up to 4 nodes by at most 32: below 9 levels x 32 + 8

__device__ __forceinline__ int near_knn(const Index &ix, int i, const float xq[3], int skip, int K, float bound,
                                        NearK &t, int *stk) {
    const unsigned FULL = 0xffffffffu;
    const float INF = __int_as_float(0x7f800000);
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float zero[3] = {0.0f, 0.0f, 0.0f};
    t.d = t.spill = INF;
    t.bound = bound;
    t.j = -1;
    const int own = i / kLeaf;
    near_scan(ix, xq, skip, t, K, ix.L + own, ix.L + (own ^ 1), ix.L > 1);
    int sp = 0, base = 0;
    bool live = lane >= 8 - ix.first && lane < 8;   // the first round: the nodes of the first level
    for (;;) {
        const bool leaf = base + 7 >= ix.leaf0;
        const int pos = base + (lane & 7);
        float key = INF;
        bool pass = false;
        if (live && !(leaf && ((pos - ix.leaf0) ^ own) <= 1)) {   // the two buckets scanned first are done
            key = obb_d2(obb_at(ix.obb, pos), xq, zero) * kObbShrink;
            pass = key <= t.bound;
        }
        const unsigned im = __ballot_sync(FULL, pass && !leaf);
        if (sp + __popc(im) > kNearStack) return 2;
        if (pass && !leaf) stk[sp + __popc(im & below)] = pos;
        sp += __popc(im);
        for (;;) {   // buckets, nearest first
            unsigned m[2];
#pragma unroll
            for (int two = 0; two < 2; ++two) {
                const bool in = pass && leaf && key <= t.bound;
                m[two] = __reduce_min_sync(FULL, in ? (__float_as_uint(key) & ~31u) | lane : 0xffffffffu);
                if (m[two] != 0xffffffffu && lane == (int)(m[two] & 31u)) pass = false;
            }
            if (m[0] == 0xffffffffu) break;
            const bool two = m[1] != 0xffffffffu;
            const int na = __shfl_sync(FULL, pos, m[0] & 31u), nb = __shfl_sync(FULL, pos, m[1] & 31u);
            near_scan(ix, xq, skip, t, K, ix.L + na - ix.leaf0, ix.L + nb - ix.leaf0, two);
        }
        __syncwarp();
        if (sp == 0) break;
        const int k = min(4, sp), g = lane >> 3;
        live = g < k;
        base = live ? 8 * stk[sp - 1 - g] + 8 * ix.first - 56 : 0;
        sp -= k;
        __syncwarp();
    }
    const float kth = __shfl_sync(FULL, t.d, K - 1);
    const float next = K < 32 ? __shfl_sync(FULL, t.d, K & 31) : t.spill;
    t.bound = kth;
    return !(kth >= kNearMin && kth < INF) || (next <= kth * kTieWindow && next < INF) ? 1 : 0;
}

// The same selection by float distance: each lane keeps its seven nearest, sorted.
// A float distance has a relative error below 4e-7, so the first six are the exact
// six unless the seventh lies within 2e-6 of the sixth.
struct Near7 {
    float d[7];
    int j[7];
};

__device__ __forceinline__ void near7_offer(Near7 &b, float4 q, const float xq[3], int j) {
    const float fx = q.x - xq[0], fy = q.y - xq[1], fz = q.z - xq[2];
    const float dv = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
    if (!(dv < b.d[6])) return;
#pragma unroll
    for (int s = 6; s >= 1; --s) {
        const bool in = dv < b.d[s], before = dv < b.d[s - 1];
        b.j[s] = before ? b.j[s - 1] : (in ? j : b.j[s]);
        b.d[s] = before ? b.d[s - 1] : (in ? dv : b.d[s]);
    }
    if (dv < b.d[0]) {
        b.d[0] = dv;
        b.j[0] = j;
    }
}

// Returns 0 when every lane has its exact six, 1 when float distances cannot tell
// some lane's sixth, 2 when the candidate list or the walk's stack would overflow.
__device__ __forceinline__ int tile_near7(const Index &ix, int g, int i, bool live, const float xq[3], Near7 &b,
                                           int *stk, int *cand) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int s = 0; s < 7; ++s) {
        b.d[s] = INFINITY;
        b.j[s] = -1;
    }
    const int i0 = 32 * g;
    const float4 mine = live ? __ldg(ix.pts + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int k = 1; k < 32; ++k) {   // the tile's own points, nearest in Morton order first
        const int off = (k & 1) ? (k + 1) >> 1 : -(k >> 1);   // +1, -1, +2, -2, ..., -15, +16
        const int t = (lane + off) & 31;
        float4 q;
        q.x = __shfl_sync(FULL, mine.x, t);
        q.y = __shfl_sync(FULL, mine.y, t);
        q.z = __shfl_sync(FULL, mine.z, t);
        if (live && i0 + t < ix.n) near7_offer(b, q, xq, i0 + t);
    }
    float R = live ? b.d[5] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) R = fmaxf(R, __shfl_xor_sync(FULL, R, o));
    if (!(R < INFINITY)) return 2;
    const int nc = tile_candidates(ix, g, R, stk, cand);
    if (nc < 0) return 2;
    const float zero[3] = {0.0f, 0.0f, 0.0f};
    for (int k = 0; k < nc; ++k) {
        const int c = cand[k];
        const bool need = live && obb_d2(obb_at(ix.obb, c - ix.L + ix.leaf0), xq, zero) * kObbShrink <= b.d[5];
        if (!__any_sync(FULL, need)) continue;
        const int beg = (c - ix.L) * kLeaf;
        const int end = min(beg + kLeaf, ix.n);
        if (need)
            for (int j = beg; j < end; ++j) near7_offer(b, __ldg(ix.pts + j), xq, j);
    }
    return __any_sync(FULL, live && !(b.d[6] > b.d[5] * kTieWindow && b.d[5] < INFINITY && b.d[5] >= kNearMin)) ? 1 : 0;
}

// Sort of six non-negative doubles by their bits (they order alike).
__device__ __forceinline__ void sort6(long long (&v)[6]) {
    constexpr int A[12] = {0, 1, 2, 1, 3, 0, 2, 0, 2, 4, 1, 3}, B[12] = {5, 3, 4, 2, 4, 3, 5, 1, 3, 5, 2, 4};
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const long long x = v[A[k]], y = v[B[k]];
        v[A[k]] = x < y ? x : y;
        v[B[k]] = x < y ? y : x;
    }
}

// write_knn6_stats for six neighbours in any order.
__device__ __forceinline__ void write_near6_stats(const Index &ix, int i, const float xq[3], const Near7 &b,
                                                  double *stat_d, double *stat_h) {
    const double x0 = xq[0], x1 = xq[1], x2 = xq[2];
    float4 ni = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (stat_h != nullptr) ni = ix.nrm[i];
    long long dk[6], hk[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const float4 q = __ldg(ix.pts + b.j[s]);
        const double a0 = (double)q.x - x0, a1 = (double)q.y - x1, a2 = (double)q.z - x2;
        dk[s] = __double_as_longlong(a0 * a0 + a1 * a1 + a2 * a2);
        hk[s] = __double_as_longlong(fabs(a0 * ni.x + a1 * ni.y + a2 * ni.z));
    }
    sort6(dk);
    stat_d[i] = 0.5 * (sqrt(__longlong_as_double(dk[2])) + sqrt(__longlong_as_double(dk[3])));
    if (stat_h != nullptr) {
        sort6(hk);
        stat_h[i] = 0.5 * (__longlong_as_double(hk[2]) + __longlong_as_double(hk[3]));
    }
}

// Tiles whose candidate list does not fit (a scattered tile: its 32 points lie on
// both sides of a gap of the Morton order) are left to k_knn6_rest: `rest` holds
// their numbers, rest[-1] how many.
__global__ void __launch_bounds__(kKnnBlock) k_knn6_tile(Index ix, double *__restrict__ stat_d,
                                                         double *__restrict__ stat_h, int *__restrict__ rest) {
    __shared__ int s_stk[kKnnBlock / 32][kWarpStack];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int g = blockIdx.x * (kKnnBlock / 32) + w;
    if (g >= (ix.n + 31) / 32) return;
    int *stk = s_stk[w];
    int *cand = s_stk[w] + (kWarpStack - kKnnCand);
    const int i = 32 * g + lane;
    const bool live = i < ix.n;
    float xq[3] = {0.0f, 0.0f, 0.0f};
    if (live) {
        const float4 qi = __ldg(ix.pts + i);
        xq[0] = qi.x;
        xq[1] = qi.y;
        xq[2] = qi.z;
    }
    Near7 nb;
    const int rc = tile_near7(ix, g, i, live, xq, nb, stk, cand);
    if (rc == 0) {
        if (live) write_near6_stats(ix, i, xq, nb, stat_d, stat_h);
        return;
    }
    __syncwarp();
    if (rc == 1) {   // ties: FP64 distances
        Best6 b;
        if (tile_knn6(ix, g, i, live, xq, b, stk, cand)) {
            if (live) write_knn6_stats(ix, i, xq, b, stat_d, stat_h);
            return;
        }
    }
    if (lane == 0) rest[atomicAdd(rest - 1, 1)] = g;
}

// The points of the tiles k_knn6_tile left over, one per warp: by float distance
// (near_knn), again in FP64 where that cannot tell the sixth.
__global__ void __launch_bounds__(kKnnBlock) k_knn6_rest(Index ix, double *__restrict__ stat_d,
                                                         double *__restrict__ stat_h, const int *__restrict__ rest,
                                                         int *__restrict__ overflow) {
    __shared__ int s_stk[kKnnBlock / 32][kWarpStack];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t total = 32 * (int64_t)__ldg(rest - 1);
    for (int64_t u = (int64_t)blockIdx.x * (kKnnBlock / 32) + w; u < total; u += (int64_t)gridDim.x * (kKnnBlock / 32)) {
        const int i = 32 * __ldg(rest + (u >> 5)) + (int)(u & 31);
        if (i >= ix.n) continue;   // uniform in the warp
        const float4 qi = __ldg(ix.pts + i);
        const float xq[3] = {qi.x, qi.y, qi.z};
        NearK t;
        const int rc = near_knn(ix, i, xq, i, 6, __int_as_float(0x7f800000), t, s_stk[w]);
        __syncwarp();
        if (rc != 0) {
            Best6 b;
            if (!warp_knn6(ix, i, xq, b, s_stk[w])) {
                if (lane == 0) *overflow = 1;
            } else if (lane == 0) {
                write_knn6_stats(ix, i, xq, b, stat_d, stat_h);
            }
            __syncwarp();
            continue;
        }
        // one neighbour per lane; the 3rd and 4th smallest by rank
        long long dk = 0, hk = 0;
        if (lane < 6) {
            const float4 q = __ldg(ix.pts + t.j);
            const double a0 = (double)q.x - (double)xq[0], a1 = (double)q.y - (double)xq[1],
                         a2 = (double)q.z - (double)xq[2];
            dk = __double_as_longlong(a0 * a0 + a1 * a1 + a2 * a2);
            if (stat_h != nullptr) {
                const float4 ni = __ldg(ix.nrm + i);
                hk = __double_as_longlong(fabs(a0 * ni.x + a1 * ni.y + a2 * ni.z));
            }
        }
        int rd = 0, rh = 0;
#pragma unroll
        for (int s = 0; s < 6; ++s) {
            const long long od = __shfl_sync(FULL, dk, s), oh = __shfl_sync(FULL, hk, s);
            rd += od < dk || (od == dk && s < lane);
            rh += oh < hk || (oh == hk && s < lane);
        }
        const unsigned d2 = __ballot_sync(FULL, lane < 6 && rd == 2), d3 = __ballot_sync(FULL, lane < 6 && rd == 3);
        const unsigned h2 = __ballot_sync(FULL, lane < 6 && rh == 2), h3 = __ballot_sync(FULL, lane < 6 && rh == 3);
        const double v2 = __longlong_as_double(__shfl_sync(FULL, dk, __ffs(d2) - 1));
        const double v3 = __longlong_as_double(__shfl_sync(FULL, dk, __ffs(d3) - 1));
        const double u2 = __longlong_as_double(__shfl_sync(FULL, hk, __ffs(h2) - 1));
        const double u3 = __longlong_as_double(__shfl_sync(FULL, hk, __ffs(h3) - 1));
        if (lane == 0) {
            stat_d[i] = 0.5 * (sqrt(v2) + sqrt(v3));
            if (stat_h != nullptr) stat_h[i] = 0.5 * (u2 + u3);
        }
    }
}

// ---------------------------------------------------------------------------
// Normal estimate (Sec. 6: where the surface is unknown the paper estimates
// normals from the 30 nearest neighbours): the neighbourhood of q_i is its k
// nearest points, q_i included, ordered by (exact FP64 squared distance,
// original index); the normal is the eigenvector of the smallest eigenvalue of
// the neighbourhood's covariance about its centroid, turned towards a viewpoint.
//
// k_normals: a block takes up to 32 Morton-consecutive points.
//   1. Each warp finds the K nearest of its points by float distance, one point
//      after the other (near_knn: the list sorted one entry per lane, buckets
//      merged 32 candidates at a time). Float distances have a
//      relative error below 4e-7, so the set is the exact one unless the
//      (K+1)-th lies within 2e-6 of the K-th; those points (ties, and about one
//      in 10^4 otherwise) are searched again with FP64 distances (warp_knn_k).
//   2. Each lane of the first warp takes one point: the covariance of its
//      neighbours in FP64 and its smallest eigenvector (smallest_axis).
// GB300 issues an FP64 warp instruction once in 64 cycles however many lanes it
// has, so FP64 work spread over a warp per point (distances, list comparisons,
// covariance sums, 3.0 ms of k_knn_cov for 100,000 points) was the bound; with a
// point per lane it is 1/32 of that. The kernel now keeps 57% of the issue slots
// and 33% of the FP64 pipe busy: the search's issue and latency are the bound.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double exact_d2(float4 q, const float xq[3]) {
    const double a0 = (double)q.x - (double)xq[0], a1 = (double)q.y - (double)xq[1], a2 = (double)q.z - (double)xq[2];
    return __dadd_rn(__dadd_rn(__dmul_rn(a0, a0), __dmul_rn(a1, a1)), __dmul_rn(a2, a2));
}

struct TopK {
    double d;   // lane s: the s-th smallest squared distance so far
    int o, j;   // its original index and bucket-order position
    float bound;
};

__device__ __forceinline__ void topk_scan(const Index &ix, const float xq[3], TopK &t, int K, int na, int nb,
                                          bool two) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    bool cand = false;
    double d = 0.0;
    int o = 0, j = -1;
    if (lane < 16 || two) {
        j = ((lane < 16 ? na : nb) - ix.L) * kLeaf + (lane & 15);
        if (j < ix.n) {
            const float4 q = __ldg(ix.pts + j);
            const float fx = q.x - xq[0], fy = q.y - xq[1], fz = q.z - xq[2];
            if (fmaf(fz, fz, fmaf(fy, fy, fx * fx)) * kShrink <= t.bound) {
                d = exact_d2(q, xq);
                o = __float_as_int(q.w);
                cand = true;
            }
        }
    }
    unsigned cm = __ballot_sync(FULL, cand);
    while (cm) {   // insert in lane order
        const int src = __ffs(cm) - 1;
        cm &= cm - 1u;
        const double dv = __shfl_sync(FULL, d, src);
        const int ov = __shfl_sync(FULL, o, src), jv = __shfl_sync(FULL, j, src);
        // non-negative doubles order as their bits: no FP64 comparison
        const long long td = __double_as_longlong(t.d), cd = __double_as_longlong(dv);
        const bool greater = lane < K && (td > cd || (td == cd && t.o > ov));
        const unsigned gm = __ballot_sync(FULL, greater);
        if (gm == 0u) continue;   // not among the K nearest
        const int pos = __ffs(gm) - 1;
        const double ud = __shfl_up_sync(FULL, t.d, 1);
        const int uo = __shfl_up_sync(FULL, t.o, 1), uj = __shfl_up_sync(FULL, t.j, 1);
        if (lane == pos) {
            t.d = dv;
            t.o = ov;
            t.j = jv;
        } else if (lane > pos && lane < K) {
            t.d = ud;
            t.o = uo;
            t.j = uj;
        }
        t.bound = __double2float_ru(__shfl_sync(FULL, t.d, K - 1));
    }
}

// The K nearest by (FP64 distance, original index). Returns false if the stack
// would overflow.
__device__ __noinline__ bool warp_knn_k(const Index &ix, int i, const float xq[3], int K, TopK &t, int *stk) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const float zero[3] = {0.0f, 0.0f, 0.0f};
    t.d = INFINITY;
    t.o = 0x7fffffff;
    t.j = -1;
    t.bound = INFINITY;
    int depth = 0;
    while ((1 << depth) < ix.L) ++depth;
    const int start = ix.L + i / kLeaf;
    topk_scan(ix, xq, t, K, start, start ^ 1, depth > 0);   // the point's bucket and its sibling first
    int sp;
    {
        int c = 0;
        bool pass = false;
        if (lane < depth - 1) {
            c = (start >> (depth - 1 - lane)) ^ 1;
            pass = box_d2(__ldg(ix.nodes + 2 * c), __ldg(ix.nodes + 2 * c + 1), xq, zero) * kShrink <= t.bound;
        }
        const unsigned m = __ballot_sync(FULL, pass);
        if (pass) stk[__popc(m & below)] = c;
        sp = __popc(m);
    }
    __syncwarp();
    const int leaf_parent_level = depth - 1;
    while (sp > 0) {
        const int k = min(32, sp);
        const int node = (lane < k) ? stk[sp - 1 - lane] : 0;
        sp -= k;
        __syncwarp();
        int c[4] = {0, 0, 0, 0};
        bool ok[4] = {false, false, false, false};
        bool leaf_ok = false;
        if (node != 0) {
            if (node < ix.L) {
                const int level = 31 - __clz(node);
                if (level < leaf_parent_level) {
                    const float4 *bx = ix.nodes + 8 * node;
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        c[g] = 4 * node + g;
                        ok[g] = box_d2(__ldg(bx + 2 * g), __ldg(bx + 2 * g + 1), xq, zero) * kShrink <= t.bound;
                    }
                } else {
                    const float4 *bx = ix.nodes + 4 * node;
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        c[g] = 2 * node + g;
                        ok[g] = box_d2(__ldg(bx + 2 * g), __ldg(bx + 2 * g + 1), xq, zero) * kShrink <= t.bound;
                    }
                }
            } else {
                leaf_ok = box_d2(__ldg(ix.nodes + 2 * node), __ldg(ix.nodes + 2 * node + 1), xq, zero) * kShrink
                              <= t.bound &&
                          obb_d2(obb_at(ix.obb, node - ix.L + ix.leaf0), xq, zero) * kObbShrink <= t.bound;
            }
        }
        int base = sp;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const unsigned mg = __ballot_sync(FULL, ok[g]);
            if (base + __popc(mg) > kWarpStack) return false;
            if (ok[g]) stk[base + __popc(mg & below)] = c[g];
            base += __popc(mg);
        }
        sp = base;
        unsigned lm = __ballot_sync(FULL, leaf_ok);
        while (lm) {   // two buckets per pass: lanes 0-15 and 16-31
            const int la = __ffs(lm) - 1;
            lm &= lm - 1u;
            int lb = la;
            bool two = false;
            if (lm) {
                lb = __ffs(lm) - 1;
                lm &= lm - 1u;
                two = true;
            }
            const int na = __shfl_sync(FULL, node, la), nb = __shfl_sync(FULL, node, lb);
            topk_scan(ix, xq, t, K, na, nb, two);
        }
        __syncwarp();
    }
    return true;
}

// Eigenvector of the smallest eigenvalue of the symmetric matrix e (xx, xy, xz,
// yy, yz, zz) by cyclic Jacobi rotations in FP64.
__device__ __noinline__ void jacobi_axis(const double e[6], double n[3]) {
    double a[3][3], V[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
    a[0][0] = e[0];
    a[0][1] = a[1][0] = e[1];
    a[0][2] = a[2][0] = e[2];
    a[1][1] = e[3];
    a[1][2] = a[2][1] = e[4];
    a[2][2] = e[5];
    const int P[3] = {0, 0, 1}, Qi[3] = {1, 2, 2};
    for (int sweep = 0; sweep < 32; ++sweep) {
        const double off = fabs(a[0][1]) + fabs(a[0][2]) + fabs(a[1][2]);
        const double diag = fabs(a[0][0]) + fabs(a[1][1]) + fabs(a[2][2]);
        if (!(off > 1e-18 * diag)) break;
        for (int r = 0; r < 3; ++r) {
            const int pp = P[r], qq = Qi[r];
            if (a[pp][qq] == 0.0) continue;
            const double th = (a[qq][qq] - a[pp][pp]) / (2.0 * a[pp][qq]);
            const double tt = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
            const double cs = 1.0 / sqrt(tt * tt + 1.0), sn = tt * cs;
            for (int k = 0; k < 3; ++k) {   // a <- J^T a J
                const double akp = a[k][pp], akq = a[k][qq];
                a[k][pp] = cs * akp - sn * akq;
                a[k][qq] = sn * akp + cs * akq;
            }
            for (int k = 0; k < 3; ++k) {
                const double apk = a[pp][k], aqk = a[qq][k];
                a[pp][k] = cs * apk - sn * aqk;
                a[qq][k] = sn * apk + cs * aqk;
            }
            for (int k = 0; k < 3; ++k) {   // V <- V J
                const double vkp = V[k][pp], vkq = V[k][qq];
                V[k][pp] = cs * vkp - sn * vkq;
                V[k][qq] = sn * vkp + cs * vkq;
            }
        }
    }
    int m = 0;
    if (a[1][1] < a[m][m]) m = 1;
    if (a[2][2] < a[m][m]) m = 2;
    for (int k = 0; k < 3; ++k) n[k] = V[k][m];
}

// The same vector (any length) when the two smaller eigenvalues are apart: float
// Jacobi rotations, then two Rayleigh quotient steps in FP64, n <- adj(A - s I) n
// with s = n.A n / n.n. A step cubes the float error (below 1e-2 where the gap
// exceeds 1e-4 of the largest eigenvalue), so two give the FP64 eigenvector, in
// about 100 FP64 instructions instead of 1,300. Smaller gaps take jacobi_axis.
__device__ __forceinline__ void smallest_axis(const double e[6], double n[3]) {
    const double sc = e[0] + e[3] + e[5];
    const float is = 1.0f / (float)sc;
    const float f[6] = {(float)e[0] * is, (float)e[1] * is, (float)e[2] * is,
                        (float)e[3] * is, (float)e[4] * is, (float)e[5] * is};
    float A[3][3] = {{f[0], f[1], f[2]}, {f[1], f[3], f[4]}, {f[2], f[4], f[5]}}, V[3][3];
    jacobi3f(A, V);
    const float l0 = A[0][0], l1 = A[1][1], l2 = A[2][2];
    const float lo = fminf(l0, fminf(l1, l2)), hi = fmaxf(l0, fmaxf(l1, l2));
    const float mid = fmaxf(fminf(l0, l1), fminf(fmaxf(l0, l1), l2));
    if (!(mid - lo > 1e-4f * hi) || !(is > 1e-30f && is < 1e30f)) {
        jacobi_axis(e, n);
        return;
    }
    const bool m1 = l1 == lo, m2 = l2 == lo;
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] = (double)(m2 ? V[k][2] : (m1 ? V[k][1] : V[k][0]));
    const double ds = (double)is;
    const double xx = e[0] * ds, xy = e[1] * ds, xz = e[2] * ds, yy = e[3] * ds, yz = e[4] * ds, zz = e[5] * ds;
#pragma unroll
    for (int step = 0; step < 2; ++step) {
        const double n2 = fma(n[2], n[2], fma(n[1], n[1], n[0] * n[0]));
        double u[3] = {fma(xz, n[2], fma(xy, n[1], xx * n[0])), fma(yz, n[2], fma(yy, n[1], xy * n[0])),
                       fma(zz, n[2], fma(yz, n[1], xz * n[0]))};
        const double inv = (double)(1.0f / (float)n2);   // the quotient to float accuracy of |n|^2, refined once
        const double r = inv * fma(-n2, inv, 2.0);
        const double s = fma(n[2], u[2], fma(n[1], u[1], n[0] * u[0])) * r;
        const double a = xx - s, b = yy - s, c = zz - s;
        const double c00 = fma(b, c, -(yz * yz)), c01 = fma(xz, yz, -(xy * c)), c02 = fma(xy, yz, -(xz * b));
        const double c11 = fma(a, c, -(xz * xz)), c12 = fma(xy, xz, -(a * yz)), c22 = fma(a, b, -(xy * xy));
        u[0] = fma(c02, n[2], fma(c01, n[1], c00 * n[0]));
        u[1] = fma(c12, n[2], fma(c11, n[1], c01 * n[0]));
        u[2] = fma(c22, n[2], fma(c12, n[1], c02 * n[0]));
        // back to about unit length (any positive factor does)
        const float q = (float)fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]));
        const double g = (double)rsqrtf(q);
#pragma unroll
        for (int k = 0; k < 3; ++k) n[k] = u[k] * g;
    }
}

// Normals of 4 x `per_warp` (up to 8) Morton-consecutive points per block, turned
// so that n . (viewpoint - q) >= 0, written at the original index. Consecutive
// points are close: the K nearest of one lie within its K-th distance plus the
// step to the next, which bounds the next one's search from the start.
constexpr int kNormalsPerWarp = 8;

__global__ void __launch_bounds__(kKnnBlock) k_normals(Index ix, int K, int per_warp, double v0, double v1, double v2,
                                                       float *__restrict__ out, int *__restrict__ overflow) {
    __shared__ int s_stk[kKnnBlock / 32][kWarpStack];   // kNearStack of it, but warp_knn_k takes all
    __shared__ int s_nbr[32][33];
    const float INF = __int_as_float(0x7f800000);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t b0 = (int64_t)blockIdx.x * (kKnnBlock / 32) * per_warp;
    float bound = INF;
    float last[3] = {0.0f, 0.0f, 0.0f};
    for (int p = 0; p < per_warp; ++p) {
        const int64_t i = b0 + w * per_warp + p;
        if (i >= ix.n) break;   // uniform in the warp
        const float4 qi = __ldg(ix.pts + i);
        const float xq[3] = {qi.x, qi.y, qi.z};
        if (bound < INF) {
            const float dx = xq[0] - last[0], dy = xq[1] - last[1], dz = xq[2] - last[2];
            const float r = sqrtf(bound) + sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
            bound = r * r * (1.0f + 1e-5f);
        }
        NearK t;
        int rc = near_knn(ix, (int)i, xq, -1, K, bound, t, s_stk[w]);
        bound = t.bound;
        last[0] = xq[0];
        last[1] = xq[1];
        last[2] = xq[2];
        __syncwarp();
        if (rc == 1) {
            TopK e;
            rc = warp_knn_k(ix, (int)i, xq, K, e, s_stk[w]) ? 0 : 2;
            t.j = e.j;
        }
        if (rc == 2 && lane == 0) *overflow = 1;
        s_nbr[w * per_warp + p][lane] = rc == 2 ? (int)i : t.j;
        __syncwarp();
    }
    __syncthreads();
    const int64_t i = b0 + lane;
    if (w != 0 || lane >= (kKnnBlock / 32) * per_warp || i >= ix.n) return;
    const float4 qi = __ldg(ix.pts + i);
    const double x = qi.x, y = qi.y, z = qi.z;
    // sums of the differences to the point and of their products
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, e[6] = {0, 0, 0, 0, 0, 0};
    for (int k = 0; k < K; ++k) {
        const float4 q = __ldg(ix.pts + s_nbr[lane][k]);
        const double d0 = (double)q.x - x, d1 = (double)q.y - y, d2 = (double)q.z - z;
        s0 += d0;
        s1 += d1;
        s2 += d2;
        e[0] = fma(d0, d0, e[0]);
        e[1] = fma(d0, d1, e[1]);
        e[2] = fma(d0, d2, e[2]);
        e[3] = fma(d1, d1, e[3]);
        e[4] = fma(d1, d2, e[4]);
        e[5] = fma(d2, d2, e[5]);
    }
    const double ik = 1.0 / (double)K;
    e[0] = fma(-s0 * ik, s0, e[0]);
    e[1] = fma(-s0 * ik, s1, e[1]);
    e[2] = fma(-s0 * ik, s2, e[2]);
    e[3] = fma(-s1 * ik, s1, e[3]);
    e[4] = fma(-s1 * ik, s2, e[4]);
    e[5] = fma(-s2 * ik, s2, e[5]);
    double n[3];
    smallest_axis(e, n);
    const double inv = 1.0 / sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    const double side = n[0] * (v0 - x) + n[1] * (v1 - y) + n[2] * (v2 - z);
    const double sg = side < 0.0 ? -inv : inv;
    const int o = __float_as_int(qi.w);
    out[3 * (size_t)o] = (float)(n[0] * sg);
    out[3 * (size_t)o + 1] = (float)(n[1] * sg);
    out[3 * (size_t)o + 2] = (float)(n[2] * sg);
}

// Grid-wide form of block_median_pair for large n (the nu_min medians of a
// whole target): the same eight 8-bit radix passes over the IEEE bit patterns,
// but each pass's two histograms are built by every block (shared-memory
// histograms folded into MedianState::hist with one atomic per bin and block). Counts do not depend on the
// order of the atomics, so the result is the one block_median_pair gives.
// One launch per radix pass: the last block to fold its histograms locates each
// rank's bin and clears the histograms for the next pass. Two arrays of n values
// (the point and the plane statistic) are taken side by side, blockIdx.y each
// (500,000 points, both statistics: 34 launches 162 us, 9 launches 86 us).
// Launch order: k_median_init, then for shift = 56, 48, ..., 0 one
// k_median_pass; the last writes 0.5 * (lo + hi) to out[blockIdx.y].
struct MedianState {
    unsigned long long prefix[2];
    int k[2];
    unsigned int done;   // blocks that folded their histograms in this pass
    unsigned int pad;
    unsigned int hist[2][256];
};

__global__ void k_median_init(MedianState *st, int n) {
    st += blockIdx.x;
    for (int b = threadIdx.x; b < 512; b += blockDim.x) (&st->hist[0][0])[b] = 0u;
    if (threadIdx.x == 0) {
        st->prefix[0] = st->prefix[1] = 0ull;
        st->k[0] = (n - 1) / 2;
        st->k[1] = n / 2;
        st->done = 0u;
    }
}

__global__ void __launch_bounds__(256) k_median_pass(const double *v0, const double *v1, int n, MedianState *st,
                                                     int shift, double *out) {
    __shared__ unsigned int hist[2][256];
    __shared__ bool s_last;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double *v = blockIdx.y ? v1 : v0;
    st += blockIdx.y;
    for (int b = threadIdx.x; b < 512; b += blockDim.x) (&hist[0][0])[b] = 0u;
    __syncthreads();
    const unsigned long long p0 = st->prefix[0], p1 = st->prefix[1];
    const unsigned long long mask = (shift == 56) ? 0ull : (~0ull << (shift + 8));
    // every lane runs every round (the peer match is warp-wide)
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        unsigned long long key = ~0ull;
        if (i < n) key = (unsigned long long)__double_as_longlong(__ldcg(v + i));
        const int bin = (int)((key >> shift) & 255ull);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const bool match = i < n && (key & mask) == (r ? p1 : p0);
            const unsigned peers = __match_any_sync(FULL, match ? bin : -1);
            if (match && lane == __ffs(peers) - 1) atomicAdd(&hist[r][bin], (unsigned)__popc(peers));
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 512; b += blockDim.x) {
        const unsigned c = (&hist[0][0])[b];
        if (c) atomicAdd(&st->hist[0][0] + b, c);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (w < 2) {   // warp r finds the bin holding its rank (as block_median_pair)
        unsigned c[8], sum = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            c[q] = __ldcg(&st->hist[w][8 * lane + q]);
            sum += c[q];
        }
        unsigned incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        const unsigned excl = incl - sum;
        const unsigned k = (unsigned)st->k[w];
        const unsigned owner = __ballot_sync(FULL, excl <= k && k < incl);
        if (lane == __ffs(owner) - 1) {
            unsigned cum = excl;
            int q = 0;
            for (; q < 7; ++q) {
                if (cum + c[q] > k) break;
                cum += c[q];
            }
            st->k[w] = (int)(k - cum);
            st->prefix[w] |= (unsigned long long)(8 * lane + q) << shift;
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 512; b += blockDim.x) (&st->hist[0][0])[b] = 0u;   // for the next pass
    if (threadIdx.x == 0) {
        st->done = 0u;
        if (shift == 0)
            out[blockIdx.y] =
                0.5 * (__longlong_as_double((long long)st->prefix[0]) + __longlong_as_double((long long)st->prefix[1]));
    }
}

// Bounding box, sum and validity of n points, on the device (parts: freed by the
// caller on s) and in pinned host memory of this thread, which wait_box waits for:
// what is queued in between runs meanwhile. Every start_box that succeeded is
// followed by a wait_box before the next.
struct BoxStage {
    BoxPartial *h = nullptr;
    cudaEvent_t ev = nullptr;
};

BoxStage &box_stage() {
    thread_local BoxStage b;
    if (b.h == nullptr && cudaMallocHost(&b.h, sizeof(BoxPartial)) != cudaSuccess) b.h = nullptr;
    if (b.ev == nullptr && cudaEventCreateWithFlags(&b.ev, cudaEventDisableTiming) != cudaSuccess) b.ev = nullptr;
    return b;
}

cudaError_t start_box(const float *x, const float *nrm, int64_t n, cudaStream_t s, BoxPartial **parts_out,
                      const BoxPartial **box_out, int zero_normals_ok = 0) {
    BoxStage &st = box_stage();
    if (st.h == nullptr || st.ev == nullptr) return cudaErrorMemoryAllocation;
    int nb = (int)std::min<int64_t>((n + kRedBlock - 1) / kRedBlock, 1024);
    if (nb < 1) nb = 1;
    BoxPartial *parts = nullptr;
    cudaError_t e = pool_alloc(&parts, sizeof(BoxPartial) * (nb + 1), s);
    if (e != cudaSuccess) return e;
    k_box_partial<<<nb, kRedBlock, 0, s>>>(x, nrm, n, parts, zero_normals_ok);
    k_box_final<<<1, kRedBlock, 0, s>>>(parts, nb, parts + nb, st.h);
    counters().launches += 2;
    e = cudaGetLastError();
    counters().d2h += sizeof(BoxPartial);
    if (e == cudaSuccess) e = cudaEventRecord(st.ev, s);
    if (e != cudaSuccess) {
        cudaFreeAsync(parts, s);
        return e;
    }
    *parts_out = parts;
    *box_out = parts + nb;
    return cudaSuccess;
}

cudaError_t wait_box(BoxPartial *res) {
    BoxStage &st = box_stage();
    const cudaError_t e = cudaEventSynchronize(st.ev);
    if (e == cudaSuccess) *res = *st.h;
    return e;
}

// Kernels one sort of n keys launches, for the launch counter (0 if unknown: the
// stream cannot be captured). A call whose size lies outside the ranges seen costs a
// capture of the sort (eval_pass on 20,000 and 19,999 points in turn, captured in
// every call 205 us, in none 194 us; on 2,000 and 1,999, whose sort is two kernels,
// 137 and 137 us).
int64_t sort_launches(void *tmp, size_t tb, unsigned *code, unsigned *code2, int *idx, int *idx2, int n,
                      cudaStream_t s) {
    thread_local host::LaunchMemo memo;
    int64_t k = memo.find(n);
    if (k < 0) {
        k = host::captured_kernels(s, [&] {
            return cub::DeviceRadixSort::SortPairs(tmp, tb, code, code2, idx, idx2, n, 0, 30, s);
        });
        if (k >= 0) memo.add(n, k);
    }
    return k > 0 ? k : 0;
}

// Morton order of n points: returns the permutation (device, caller frees).
cudaError_t morton_order(const float *x, int64_t n, const BoxPartial *box, cudaStream_t s, int **order_out) {
    unsigned *code = nullptr, *code2 = nullptr;
    int *idx = nullptr, *idx2 = nullptr;
    void *tmp = nullptr;
    size_t tb = 0;
    cudaError_t e = pool_alloc(&code, 4 * n, s);
    if (e == cudaSuccess) e = pool_alloc(&code2, 4 * n, s);
    if (e == cudaSuccess) e = pool_alloc(&idx, 4 * n, s);
    if (e == cudaSuccess) e = pool_alloc(&idx2, 4 * n, s);
    if (e == cudaSuccess) {
        k_morton<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, n, box, code, idx);
        counters().launches += 1;
        e = cub::DeviceRadixSort::SortPairs(nullptr, tb, code, code2, idx, idx2, (int)n, 0, 30, s);
    }
    if (e == cudaSuccess) e = pool_alloc(&tmp, tb > 0 ? tb : 16, s);
    if (e == cudaSuccess) {
        counters().launches += sort_launches(tmp, tb, code, code2, idx, idx2, (int)n, s);
        e = cub::DeviceRadixSort::SortPairs(tmp, tb, code, code2, idx, idx2, (int)n, 0, 30, s);
    }
    if (tmp) cudaFreeAsync(tmp, s);
    if (code) cudaFreeAsync(code, s);
    if (code2) cudaFreeAsync(code2, s);
    if (idx) cudaFreeAsync(idx, s);
    if (e != cudaSuccess) {
        if (idx2) cudaFreeAsync(idx2, s);
        return e;
    }
    *order_out = idx2;
    return cudaGetLastError();
}

// Oriented boxes of all the levels of the walk, of points in the buckets of `nodes`.
void launch_oriented(const float4 *pts, int64_t n, int L, const float4 *nodes, float4 *obb, cudaStream_t s) {
    k_leaf_obb<<<(L + 127) / 128, 128, 0, s>>>(pts, n, L, obb);
    counters().launches += 1;
    const int first = wide_first(L);
    for (int shift = 3; (L >> shift) >= first; shift += 3) {
        const int size = L >> shift;
        if (shift == 3)
            k_patch_obb<32><<<(size + 7) / 8, 256, 0, s>>>(pts, n, L, shift, nodes, obb);
        else if (shift <= 9)
            k_patch_obb<256><<<size, 256, 0, s>>>(pts, n, L, shift, nodes, obb);
        else
            k_level_obb<<<(size + 127) / 128, 128, 0, s>>>(nodes, L, size, 0, obb);
        counters().launches += 1;
    }
    if (first < 8) {
        k_level_obb<<<1, 32, 0, s>>>(nodes, L, 0, 8 - first, obb);
        counters().launches += 1;
    }
}

}  // namespace

cudaError_t build_target(const float *q_dev, const float *n_dev, int64_t n, cudaStream_t s, TargetDev *t,
                         int *bad_input) {
    BoxPartial *parts = nullptr;
    const BoxPartial *box = nullptr;
    cudaError_t e = start_box(q_dev, n_dev, n, s, &parts, &box);
    if (e != cudaSuccess) return e;
    t->n = n;
    t->has_normals = n_dev != nullptr;
    const int64_t buckets = (n + kLeaf - 1) / kLeaf;
    int L = 1;
    while (L < buckets) L *= 2;
    t->L = L;
    t->E_Q = -1.0;
    t->H_Q = -1.0;
    int *order = nullptr;
    e = morton_order(q_dev, n, box, s, &order);
    cudaFreeAsync(parts, s);
    BoxPartial bx;
    const cudaError_t eb = wait_box(&bx);
    if (e == cudaSuccess) e = eb;
    if (e != cudaSuccess || bx.bad) {   // bad coordinates: their keys and order are of no use
        if (order) cudaFreeAsync(order, s);
        *bad_input = e == cudaSuccess;
        return e;
    }
    *bad_input = 0;
    for (int a = 0; a < 3; ++a) {
        t->lo[a] = bx.lo[a];
        t->hi[a] = bx.hi[a];
        t->centroid[a] = bx.sum[a] / (double)n;
    }
    e = pool_alloc(&t->pts, sizeof(float4) * n, s);
    if (e == cudaSuccess && n_dev) e = pool_alloc(&t->nrm, sizeof(float4) * n, s);
    if (e == cudaSuccess) e = pool_alloc(&t->nodes, sizeof(float4) * 4 * ((size_t)L + oriented_boxes(L)), s);
    if (e == cudaSuccess) {
        t->obb = t->nodes + 4 * (size_t)L;
        k_gather<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(q_dev, n_dev, order, n, t->pts, t->nrm);
        k_boxes<true><<<(L + 255) / 256, 256, 0, s>>>(t->pts, n, L, t->nodes);
        counters().launches += 2;
        for (int size = L / 256; size > 1; size /= 256) {
            k_boxes<false><<<(size + 255) / 256, 256, 0, s>>>(t->pts, n, size, t->nodes);
            counters().launches += 1;
        }
        launch_oriented(t->pts, n, L, t->nodes, t->obb, s);
        e = cudaGetLastError();
    }
    cudaFreeAsync(order, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    return cudaSuccess;
}

// FP16 storage of the target: each point as half-precision offsets in
// [0, 1] of its bucket's bounding box (a degenerate box axis stores 0), so a
// decoded point lo + u (hi - lo) stays inside the box the tree tests.
__global__ void k_encode16(const float4 *__restrict__ pts, const float4 *__restrict__ nodes, int n, int L,
                           ushort4 *__restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const float4 p = pts[j];
    const int leaf = L + j / kLeaf;
    const float4 lo = nodes[2 * leaf], hi = nodes[2 * leaf + 1];
    const float ex = hi.x - lo.x, ey = hi.y - lo.y, ez = hi.z - lo.z;
    const float ux = ex > 0.0f ? fminf(fmaxf((p.x - lo.x) / ex, 0.0f), 1.0f) : 0.0f;
    const float uy = ey > 0.0f ? fminf(fmaxf((p.y - lo.y) / ey, 0.0f), 1.0f) : 0.0f;
    const float uz = ez > 0.0f ? fminf(fmaxf((p.z - lo.z) / ez, 0.0f), 1.0f) : 0.0f;
    out[j] = make_ushort4(__half_as_ushort(__float2half_rn(ux)), __half_as_ushort(__float2half_rn(uy)),
                          __half_as_ushort(__float2half_rn(uz)), 0);
}

// The points as the search decodes them.
__global__ void k_decode16(Index ix, float4 *__restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < ix.n) out[j] = target_point<PREC_FP16>(ix, j);
}

cudaError_t build_fp16_storage(TargetDev *t, cudaStream_t s) {
    if (t->pts16) return cudaSuccess;
    ushort4 *p = nullptr;
    float4 *obb = nullptr, *dec = nullptr;
    cudaError_t e = pool_alloc(&p, sizeof(ushort4) * (size_t)t->n, s);
    if (e == cudaSuccess) e = pool_alloc(&obb, sizeof(float4) * 4 * oriented_boxes(t->L), s);
    if (e == cudaSuccess) e = pool_alloc(&dec, sizeof(float4) * (size_t)t->n, s);
    if (e == cudaSuccess) {
        const unsigned nb = (unsigned)((t->n + 255) / 256);
        k_encode16<<<nb, 256, 0, s>>>(t->pts, t->nodes, (int)t->n, t->L, p);
        Index ix = make_index(*t);
        ix.pts16 = p;
        k_decode16<<<nb, 256, 0, s>>>(ix, dec);
        counters().launches += 2;
        launch_oriented(dec, t->n, t->L, t->nodes, obb, s);
        e = cudaGetLastError();
    }
    if (dec) cudaFreeAsync(dec, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        if (p) cudaFreeAsync(p, s);
        if (obb) cudaFreeAsync(obb, s);
        return e;
    }
    t->obb16 = obb;
    t->pts16 = p;
    return cudaSuccess;
}

cudaError_t launch_median(const double *v, const double *v2, int n, void *scratch, double *out_dev, cudaStream_t s) {
    static_assert(2 * sizeof(MedianState) <= (size_t)kMedianScratchBytes, "median scratch");
    MedianState *mst = static_cast<MedianState *>(scratch);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int arrays = v2 != nullptr ? 2 : 1;
    const unsigned mblocks = (unsigned)std::min<int64_t>(((int64_t)n + 255) / 256, (int64_t)(sms > 0 ? sms : 152) * 4);
    k_median_init<<<arrays, 256, 0, s>>>(mst, n);
    for (int shift = 56; shift >= 0; shift -= 8)
        k_median_pass<<<dim3(mblocks, arrays), 256, 0, s>>>(v, v2, n, mst, shift, out_dev);
    counters().launches += 9;
    return cudaGetLastError();
}

cudaError_t target_nu_stats(TargetDev *t, cudaStream_t s) {
    if (t->E_Q >= 0.0 && (!t->has_normals || t->H_Q >= 0.0)) return cudaSuccess;
    if (t->n < 7) {   // fewer than six neighbours: statistic undefined, use 0 (clamped later)
        t->E_Q = 0.0;
        t->H_Q = 0.0;
        return cudaSuccess;
    }
    double *sd = nullptr, *sh = nullptr, *out = nullptr;
    void *mst = nullptr;
    cudaError_t e = pool_alloc(&sd, sizeof(double) * t->n, s);
    if (e == cudaSuccess) e = pool_alloc(&mst, kMedianScratchBytes, s);
    if (e == cudaSuccess && t->has_normals) e = pool_alloc(&sh, sizeof(double) * t->n, s);
    if (e == cudaSuccess) e = pool_alloc(&out, 3 * sizeof(double), s);
    int *flag = reinterpret_cast<int *>(out + 2);
    if (e == cudaSuccess) e = cudaMemsetAsync(out, 0, 3 * sizeof(double), s);
    if (e == cudaSuccess) {
        const Index ix = make_index(*t);
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int64_t blocks = std::min<int64_t>((t->n + kKnnBlock / 32 - 1) / (kKnnBlock / 32),
                                                 (int64_t)(sms > 0 ? sms : 152) * 16);
        if (t->L >= 4) {
            const int64_t tiles = (t->n + 31) / 32;
            int *rest = nullptr;
            e = pool_alloc(&rest, sizeof(int) * (size_t)(tiles + 1), s);
            if (e == cudaSuccess) e = cudaMemsetAsync(rest, 0, sizeof(int), s);
            if (e == cudaSuccess) {
                k_knn6_tile<<<(unsigned)((tiles + kKnnBlock / 32 - 1) / (kKnnBlock / 32)), kKnnBlock, 0, s>>>(
                    ix, sd, sh, rest + 1);
                k_knn6_rest<<<(sms > 0 ? sms : 152) * 8, kKnnBlock, 0, s>>>(ix, sd, sh, rest + 1, flag);
                counters().launches += 1;
            }
            if (rest) cudaFreeAsync(rest, s);
        } else {
            k_knn6_stats<<<(unsigned)blocks, kKnnBlock, 0, s>>>(ix, sd, sh, flag);
        }
        counters().launches += 1;
        if (e == cudaSuccess) e = launch_median(sd, sh, (int)t->n, mst, out, s);
        double h[3] = {0.0, 0.0, 0.0};
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, out, 3 * sizeof(double), cudaMemcpyDeviceToHost, s);
        counters().d2h += 3 * sizeof(double);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        int overflow = 0;
        std::memcpy(&overflow, &h[2], sizeof(int));
        if (e == cudaSuccess && overflow) e = cudaErrorLaunchOutOfResources;   // search stack: never expected
        if (e == cudaSuccess) {
            t->E_Q = h[0];
            t->H_Q = sh ? h[1] : -1.0;
        }
    }
    if (sd) cudaFreeAsync(sd, s);
    if (sh) cudaFreeAsync(sh, s);
    if (out) cudaFreeAsync(out, s);
    if (mst) cudaFreeAsync(mst, s);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

cudaError_t estimate_normals(const TargetDev *t, int k, const double viewpoint[3], float *out_dev, cudaStream_t s,
                             int *overflow_out) {
    const int K = (int)std::min<int64_t>(k, t->n);
    int *flag = nullptr;
    cudaError_t e = pool_alloc(&flag, sizeof(int), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(flag, 0, sizeof(int), s);
    if (e == cudaSuccess) {
        const Index ix = make_index(*t);
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        // 32 points per block fill the lanes of its FP64 part; fewer while that leaves an SM less than two blocks
        int per_warp = kNormalsPerWarp;
        while (per_warp > 1 && t->n < (int64_t)2 * (kKnnBlock / 32) * per_warp * (sms > 0 ? sms : 152)) per_warp /= 2;
        const int64_t per_block = (int64_t)per_warp * (kKnnBlock / 32);
        k_normals<<<(unsigned)((t->n + per_block - 1) / per_block), kKnnBlock, 0, s>>>(
            ix, K, per_warp, viewpoint[0], viewpoint[1], viewpoint[2], out_dev, flag);
        counters().launches += 1;
        e = cudaGetLastError();
    }
    int h = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    counters().d2h += sizeof(int);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (flag) cudaFreeAsync(flag, s);
    *overflow_out = h;
    return e;
}

cudaError_t prepare_source(const float *p_dev, int64_t m, cudaStream_t s, float4 *src_out, float lo[3],
                           float hi[3], int *bad_input, const float *n_dev, float4 *nrm_out) {
    BoxPartial *parts = nullptr;
    const BoxPartial *box = nullptr;
    cudaError_t e = start_box(p_dev, n_dev, m, s, &parts, &box, 1);   // a zero source normal: no normal at that point
    if (e != cudaSuccess) return e;
    int *order = nullptr;
    e = morton_order(p_dev, m, box, s, &order);
    cudaFreeAsync(parts, s);
    BoxPartial bx;
    if (e != cudaSuccess) {
        wait_box(&bx);
        return e;
    }
    k_gather<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(p_dev, n_dev, order, m, src_out, nrm_out);
    counters().launches += 1;
    e = cudaGetLastError();
    cudaFreeAsync(order, s);
    const cudaError_t eb = wait_box(&bx);
    if (e == cudaSuccess) e = eb;
    if (e != cudaSuccess) return e;
    *bad_input = bx.bad;
    for (int a = 0; a < 3; ++a) {
        lo[a] = bx.lo[a];
        hi[a] = bx.hi[a];
    }
    return cudaSuccess;
}

}  // namespace fricp

// Internal declarations shared by the CUDA translation units of libfricp.
//
// Data layout in HBM (one target set Q, one registration):
//   pts   float4[n]      target points in Morton order; .w holds the original index bits
//   nrm   float4[n]      target normals in the same order (point-to-plane only)
//   nodes float4[4L]     complete binary box tree over L (power of two) buckets of
//                        kLeaf consecutive points; node i in [1, 2L) has its box at
//                        nodes[2i] (lo) and nodes[2i+1] (hi), so the two children of
//                        node i sit in one aligned 64-byte line nodes[4i .. 4i+3].
//                        Leaf l is node L + l; empty buckets have an inverted box.
//   obb   float4[4W]     oriented box of every bucket and of every third level above
//                        the buckets (W = wide_leaf(L) + L rounded up to eights, same
//                        allocation, after the nodes): centre c and half-extents h along three orthonormal
//                        axes a_k fitted to the bucket's points, as
//                        (c, h0) (a0, h1) (a1, h2) (a2, r), r the bucket's radius;
//                        eight boxes together, one float4 of each at a time (obb_at)
//   src   float4[M]      source points in Morton order, .w = original index bits
//   PairState            one registration's solver state (FP64), ~2 KB
//   partial double[T][K] per-tile reduction records (T = ceil(M / kBlock) tiles)
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/fricp.h"
#include "obb.cuh"

#define FRICP_HD __host__ __device__

namespace fricp {

constexpr int kBlock = 256;        // threads per step block = source points per tile
constexpr int kLeaf = 16;          // target points per bucket
constexpr int kMaxM = 5;           // largest Anderson history m
constexpr int kSumsP2P = 17;       // W, W p (3), W q (3), W p q^T (9), E
constexpr int kSumsP2PL = 28;      // g z z^T (21), g z B (6), E
constexpr int kMaxSums = 28;

// Relative slack of the box pruning test: a bucket is skipped only when its box
// distance exceeds the best distance by more than the float rounding of either.
constexpr float kShrink = 1.0f - 4e-6f;

// exp(-a) is 0.0 in FP64 for a > 745.14: a Welsch point-to-point residual with
// d^2 / (2 nu^2) >= kWelschCut has weight 0 and psi 1 exactly.
constexpr double kWelschCut = 750.0;

// Precision of a registration's search and per-point terms (fricp_params.precision):
//   PREC_FP64  candidates screened in float and re-ranked in double-float: the FP64
//              argmin, ties to the lowest original index; per-point terms in FP64;
//   PREC_FP32  transform, distances and weights in float (ties to the lowest
//              original index among equal float distances); sums and solve in FP64;
//   PREC_FP16  as PREC_FP32 on target coordinates stored as 16-bit offsets in their
//              bucket's box (8 B per point); ties to the lowest bucket-order position.
enum Prec : int { PREC_FP64 = 0, PREC_FP32 = 1, PREC_FP16 = 2 };

// Variant families: point-to-plane (the Alg. 2 scheme, 28 sums) and robust
// (Welsch weights and nu stages).
__host__ __device__ inline bool variant_p2pl(int v) {
    return v == FRICP_P2PL_WELSCH_AA || v == FRICP_P2PL_AA || v == FRICP_SYM_WELSCH_AA;
}
__host__ __device__ inline bool variant_robust(int v) {
    return v == FRICP_P2P_WELSCH_AA || v == FRICP_P2PL_WELSCH_AA || v == FRICP_SYM_WELSCH_AA;
}
// The symmetric objective: the point-to-plane scheme on a residual that also
// carries the source point's normal.
__host__ __device__ inline bool variant_sym(int v) { return v == FRICP_SYM_WELSCH_AA; }

struct Index {
    const float4 *pts;
    const float4 *nrm;
    const float4 *nodes;
    const ushort4 *pts16;   // FP16 storage (x, y, z as half offsets in the bucket box), or null
    int n;
    int L;
    const float4 *obb;      // oriented boxes of the buckets and of every third level above them
    int first;              // wide_first(L)
    int leaf0;              // wide_leaf(L)
    const float4 *obb16;    // the same boxes of the points as FP16 storage decodes them, or null
};

enum Phase : int {
    PH_INIT = 0,          // pass at T0 storing per-point residuals, then the nu_max median
    PH_STAGE_START = 1,   // pass at T^(k-1) with the new nu: first alignment of a stage
    PH_ITER = 2,          // pass at T^(k): energy check at the head of an inner iteration
    PH_ITER_REVERTED = 3, // pass at T' after a failed energy check (Alg. 1)
    PH_CAPCHECK = 4,      // pass at the iterate carried out of a stage on the cap
    PH_LS = 5,            // Alg. 2 line-search trial
    PH_EVAL = 6,          // single evaluation (fricp_eval_pass)
    PH_DONE = 7
};

struct PairState {
    // ---- problem (host-written before the first step)
    int variant;
    int m;
    int max_iters;
    int cap_first;
    int cap_max;
    int max_ls;
    int M;
    int ntiles;
    int trace_cap;
    int nu_max_given;
    int prec;          // Prec
    double eps;
    double nu_max;
    double nu_min;
    double s;          // normalisation scale
    double c[3];       // normalisation centre (centroid of Q), caller units
    // ---- machine
    unsigned int counter;   // last-block ticket of the running step
    unsigned int nn_next;   // next ticket of the search kernel
    int phase;
    int done;
    int status;
    int n_body;             // inner bodies run in this stage: k - k_start - 1
    int cap;                // current I_nu
    int eval_counts;        // the pending pass is a new correspondence computation
    int capexit;            // the running line search started from a cap check
    int ls_l;
    int hlen;
    int hard_n[2][2];       // hard tickets listed for the passes of either parity, by class (k_nn)
    int init_median_ext;    // the first pass leaves the nu_max median to the host's grid-wide select (k_after_init)
    double nu;
    double E_prev;
    double tau;
    double E_best;
    // Alg. 1 transforms, normalised coordinates: R row-major (9) then t (3)
    double Tk[12], Tp[12], Tprev[12];
    double logTk[6], logTp[6];   // log of Tk / Tp, kept with them (one log per step)
    // Alg. 2 parameters xi = [delta; u]
    double xk[6], xprev[6], xstar[6], xeval[6], xbest[6];
    double sys_best[kMaxSums];
    // transform the next pass applies to the source, caller units: x = Re p + te
    double Re[9];
    double te[3];
    // derived from Re, te and nu for the search and per-point kernels (set_head_cache):
    // float splits hi + lo of Re and te, 1 / (2 nu^2) and the Welsch cap radius^2 in caller units
    float hRh[9], hRl[9], hth[3], htl[3];
    float hcut2;
    double hinv2nu2;
    double hnu;   // nu that hinv2nu2 and hcut2 belong to (0: not set)
    // Anderson history, oldest first: G^(k-j), F^(k-j)
    double Gh[kMaxM + 1][6];
    double Fh[kMaxM + 1][6];
    // counters
    int iterations, corr_passes, aa_accepted, reverts, ls_trials, stages, device_steps, trace_len;
    double final_energy;
    double eval_out[48];    // PH_EVAL result: E, T' or xi*, then the reduced sums
    // normalised transform of the pass requested last (what a step record reports)
    double Teval[12];
    // per-pass records (fricp_register_recorded), or null
    fricp_step_record *rec;
    int rec_cap, rec_len;
};

struct StepArgs {
    PairState *st;
    Index ix;
    const float4 *src;     // M sorted source points
    const float4 *src_nrm = nullptr;   // M source normals in the same order (symmetric objective), or null
    int *prev;             // M: correspondence (sorted target index) of the last pass, -1 if none;
                           //    the search kernel overwrites it with this pass's correspondence
    int *hard = nullptr;   // hard_ints(M): lists and flags of the hard tickets (k_nn), or null: plain order
    double *partial;       // ntiles * kMaxSums
    double *resid;         // M per-point residuals (PH_INIT)
    double *trace;         // trace_cap energies
};

// ---------------------------------------------------------------------------
// Exact nearest neighbour (Sec. 3, Eq. 3) over the bucket tree.
//
// Precision: the search never touches the FP64 pipe (a few FP64 units per SM
// on this GPU). x = R p + t is formed in double-float arithmetic (a float pair
// hi + lo, error-free products and sums, about 2^-44 relative), so xh = hi and
// xl = lo carry x far beyond float precision. A candidate's float squared
// distance uses (xh - q) + xl, rounding only relative to the difference itself
// (relative error < 4e-7 however far x is from the origin). Candidates whose
// float distance is within 2e-6 of the smallest are ranked by their double-float
// squared distance, and the winner is the lexicographic minimum of (that
// distance, original index): the exact argmin up to ties closer than about 1e-10
// relative, ties to the lowest index. The bucket-pruning bound keeps a slack
// (kObbShrink), so a bucket that may hold the winner is never skipped.
//
// Warm start: a query may start from any target point (the previous pass's
// correspondence); its distance is a true upper bound, so the result is the
// same argmin, found with far fewer node visits.
// ---------------------------------------------------------------------------
constexpr float kTieWindow = 1.0f + 2e-6f;

// One lane's candidates under the full ranking (the tie path of group_nn).
struct NNLane {
    float xh[3], xl[3];
    float bestf;             // float bound (smallest float distance seen)
    float best_hi, best_lo;  // double-float squared distance of the winner
    int best_j;
    int best_orig;
};

// Error-free transformations (Knuth two-sum, FMA two-product) and a
// double-float sum renormalised so that |lo| <= ulp(hi) / 2.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void df_add(float &h, float &l, float bh, float bl) {
    float s, e;
    two_sum(h, bh, s, e);
    e += l + bl;
    h = s + e;
    l = e - (h - s);
}

// x = R p + t in double-float from float splits of the FP64 R and t.
__device__ __forceinline__ void df_transform(const float Rh[9], const float Rl[9], const float th[3],
                                             const float tl[3], float4 p, float xh[3], float xl[3]) {
    const float pv[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float h = th[a], l = tl[a];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float ph = Rh[3 * a + j] * pv[j];
            float pe = fmaf(Rh[3 * a + j], pv[j], -ph);
            pe = fmaf(Rl[3 * a + j], pv[j], pe);
            df_add(h, l, ph, pe);
        }
        xh[a] = h;
        xl[a] = l;
    }
}

// Split an FP64 value into a float pair (host or device set-up code).
FRICP_HD inline void split_double(double v, float &h, float &l) {
    h = (float)v;
    l = (float)(v - (double)h);
}
__device__ __forceinline__ float axis_gap(float lo, float hi, float xh, float xl) {
    return fmaxf(fmaxf((lo - xh) - xl, (xh - hi) + xl), 0.0f);
}

__device__ __forceinline__ float box_d2(float4 lo, float4 hi, const float xh[3], const float xl[3]) {
    const float a = axis_gap(lo.x, hi.x, xh[0], xl[0]);
    const float b = axis_gap(lo.y, hi.y, xh[1], xl[1]);
    const float c = axis_gap(lo.z, hi.z, xh[2], xl[2]);
    return fmaf(c, c, fmaf(b, b, a * a));
}

// Squared distance from x = xh + xl to a bucket's oriented box (obb_fit,
// obb_eval in obb.cuh): at most (1 + 8e-6) times the squared distance to the
// bucket's nearest point. A bucket is skipped only when this distance, shrunk by
// kObbShrink, still exceeds the bound: it can never hold a point inside the tie
// window.
constexpr float kObbShrink = 1.0f - 2e-5f;

// Oriented box w of the array: its four float4 are 8 apart (eight boxes are
// stored together, first all their centres, then each axis: eight lanes testing
// a node's eight children then read whole 128-byte lines).
template <class T>
__device__ __forceinline__ T *obb_at(T *obb, int w) {
    return obb + ((size_t)(w >> 3) * 32 + (w & 7));
}

__device__ __forceinline__ float obb_d2(const float4 *o, const float xh[3], const float xl[3]) {
    return obb_eval(__ldg(o), __ldg(o + 8), __ldg(o + 16), __ldg(o + 24), xh, xl);
}

// Float squared distance from x = xh + xl to target point p.
__device__ __forceinline__ float point_d2f(const float xh[3], const float xl[3], float4 p) {
    const float dx = (xh[0] - p.x) + xl[0];
    const float dy = (xh[1] - p.y) + xl[1];
    const float dz = (xh[2] - p.z) + xl[2];
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// Squared distance in double-float: (xh - q) is split exactly by two-sum, xl
// added, each difference squared by two-product.
__device__ __forceinline__ void cand_d2_df(const NNLane &q, float4 p, float &hi, float &lo) {
    const float pv[3] = {p.x, p.y, p.z};
    hi = 0.0f;
    lo = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float s, e;
        two_sum(q.xh[a], -pv[a], s, e);
        e += q.xl[a];
        const float dh = s + e;
        const float dl = e - (dh - s);
        const float sq = dh * dh;
        float sqe = fmaf(dh, dh, -sq);
        sqe = fmaf(2.0f * dh, dl, sqe);
        df_add(hi, lo, sq, sqe);
    }
}

__device__ __forceinline__ void nn_init(NNLane &q, const float xh[3], const float xl[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        q.xh[a] = xh[a];
        q.xl[a] = xl[a];
    }
    q.bestf = __int_as_float(0x7f800000);
    q.best_hi = __int_as_float(0x7f800000);
    q.best_lo = 0.0f;
    q.best_j = -1;
    q.best_orig = 0x7fffffff;
}

// Make candidate p (sorted index j) the current winner unconditionally.
template <int PREC = PREC_FP64>
__device__ __forceinline__ void nn_seed(NNLane &q, float4 p, int j) {
    q.bestf = point_d2f(q.xh, q.xl, p);
    if (PREC == PREC_FP64) {
        cand_d2_df(q, p, q.best_hi, q.best_lo);
    } else {
        q.best_hi = q.bestf;
        q.best_lo = 0.0f;
    }
    q.best_j = j;
    q.best_orig = __float_as_int(p.w);
}

// Target point j as the search and the per-point terms see it at precision PREC
// (.w: the tie-break key: original index, or the bucket-order position for FP16).
template <int PREC>
__device__ __forceinline__ float4 target_point(const Index &ix, int j) {
    if (PREC != PREC_FP16) return __ldg(ix.pts + j);
    const ushort4 h = __ldg(ix.pts16 + j);
    const int leaf = ix.L + j / kLeaf;
    const float4 lo = __ldg(ix.nodes + 2 * leaf), hi = __ldg(ix.nodes + 2 * leaf + 1);
    float4 r;
    r.x = fmaf(__half2float(__ushort_as_half(h.x)), hi.x - lo.x, lo.x);
    r.y = fmaf(__half2float(__ushort_as_half(h.y)), hi.y - lo.y, lo.y);
    r.z = fmaf(__half2float(__ushort_as_half(h.z)), hi.z - lo.z, lo.z);
    r.w = __int_as_float(j);
    return r;
}

// (double-float d^2, original index) lexicographic order; both pairs are
// renormalised, so (hi, lo) order is the order of hi + lo.
__device__ __forceinline__ bool lex_less(float ha, float la, int oa, float hb, float lb, int ob) {
    return ha < hb || (ha == hb && (la < lb || (la == lb && oa < ob)));
}

// Offer p to the lane: ranked when within the tie window of the lane's bound.
template <int PREC = PREC_FP64>
__device__ __forceinline__ void nn_offer(NNLane &q, float4 p, int j) {
    const float d = point_d2f(q.xh, q.xl, p);
    if (d <= q.bestf * kTieWindow) {
        float hi = d, lo = 0.0f;
        if (PREC == PREC_FP64) cand_d2_df(q, p, hi, lo);
        const int o = __float_as_int(p.w);
        if (lex_less(hi, lo, o, q.best_hi, q.best_lo, q.best_orig)) {
            q.best_hi = hi;
            q.best_lo = lo;
            q.best_j = j;
            q.best_orig = o;
        }
        q.bestf = fminf(q.bestf, d);
    }
}

constexpr int kWarpStack = 1024;  // walk stack of a warp in the neighbour kernels; a round grows it by <= 96

// ---------------------------------------------------------------------------
// Group search: kGroup lanes per query, 32 / kGroup queries per warp. The binary
// box tree is walked three levels at a time: the eight descendants of a node
// three levels down are nodes 8 i .. 8 i + 7, and each lane of the group tests
// kGroupC of their boxes. A tree whose depth is not a multiple of three starts
// with the remainder (2 or 4 nodes).
//   - inner nodes: the nearest child within the bound is entered at once, the
//     others are pushed with their distance on the group's stack;
//   - buckets are scanned nearest first, the lanes sharing the points, and the
//     group's bound (and with it the buckets still waiting) is refreshed after
//     each;
//   - a pop looks at the top kGroup entries together and drops those the bound
//     has overtaken.
// The set of points offered is every point that can beat the bound, so the
// result is the exact argmin of the serial search, ties included. All 32 lanes
// run every warp-wide primitive; a group without a query (`live` false) only
// takes part in them. A path holds at most kGroupDepth inner levels, each
// leaving at most seven entries, so the stack cannot overflow.
//
// The boxes tested are the oriented ones, at every level (wide_box): on a
// surface an axis-aligned box of a tilted patch is as thick as the patch is
// wide, and a query a little off the surface is inside the boxes of all the
// patches around it. FP16 storage has boxes of its own, fitted to the decoded
// points (ellipsoids, M = 200,000: 204 us a pass; on the axis-aligned boxes, which
// hold both, about 600).
//
// What bounds it: issue slots (74% busy; about 95 instructions a round and 60 a
// bucket, 16 rounds and 8 buckets for four warm-started queries that stay
// together), then the L1 latency of each round's loads. Measured (ellipsoids,
// N = 500,000, M = 200,000, FP64, mean over a registration's passes): two
// queries per warp over the axis-aligned boxes 357 us, this 157 us (196 us
// before k_nn took the hard tickets first); with four lanes per query (two
// children each) 172 us. On the way: storing the boxes in eights, so that the L1
// serves whole lines, 377 -> 335 us; the oriented boxes above the buckets take
// the rounds per query from 20.5 to 14.8.
// ---------------------------------------------------------------------------
constexpr int kGroup = 8;                         // lanes per query
constexpr int kGroupQ = 32 / kGroup;              // queries per warp
constexpr int kGroupC = 8 / kGroup;               // children per lane
// Tickets of k_nn (kGroupQ queries each) over M queries, and the ints of their
// lists and flags: per parity of the pass, a list of T tickets and T flag bytes.
FRICP_HD inline int64_t search_tickets(int64_t M) { return (M + kGroupQ - 1) / kGroupQ; }
FRICP_HD inline int64_t hard_ints(int64_t M) { return 2 * (search_tickets(M) + (search_tickets(M) + 3) / 4); }
constexpr int kGroupDepth = 9;                    // inner levels of a tree over 2^30 points: ceil(26 / 3)
constexpr int kGroupStack = 7 * kGroupDepth + 1;  // stack entries per group
constexpr unsigned kGroupMask = (1u << kGroup) - 1u;

// Order of the oriented boxes: level by level from the top, each a multiple of
// three above the buckets; the first level has wide_first(L) nodes, at positions
// 8 - wide_first(L) .. 7 (empty boxes before them), and the children of the node
// at position p are at wide_child(first, p) .. + 7. Buckets start at wide_leaf(L).
FRICP_HD inline int wide_first(int L) {
    int depth = 0;
    while ((1 << depth) < L) ++depth;
    return 1 << (depth == 0 ? 0 : (depth - 1) % 3 + 1);
}
FRICP_HD inline int wide_pos(int first, int level_size) { return (level_size - first) / 7 + 8 - first; }
FRICP_HD inline int wide_leaf(int L) { return wide_pos(wide_first(L), L); }
FRICP_HD inline int wide_child(int first, int p) { return 8 * p + 8 * first - 56; }
// Oriented boxes stored for L buckets: those of all levels, rounded up to eights.
inline size_t oriented_boxes(int L) { return (size_t)((wide_leaf(L) + L + 7) / 8) * 8; }

// Walk the tree for the point x = xh + xl of this group, offering every point of
// every bucket within `bound` to `offer(j, p)`, which returns the smallest float
// distance this lane was offered so far. `work` counts the warp's rounds and bucket
// scans.
template <int PREC, class Offer>
__device__ __forceinline__ void group_walk(const Index &ix, const float xh[3], const float xl[3], float &bound,
                                           float2 *stk, bool live, int &work, Offer offer) {
    const float4 *obb = PREC == PREC_FP16 ? ix.obb16 : ix.obb;
    const unsigned FULL = 0xffffffffu;
    const float INF = __int_as_float(0x7f800000), OUT = __int_as_float(0x7fc00000);   // OUT: not within any bound
    const int lane = threadIdx.x & 31;
    const int gl = lane & (kGroup - 1);
    const int gs = lane & ~(kGroup - 1);
    const unsigned below = (1u << gl) - 1u;
    const int leaf0 = ix.leaf0;                   // position of the first bucket
    int base = 0;                                 // first of the eight boxes this round tests
    int cnt = live ? ix.first : 0;                // how many of them are nodes: eight after the first round, whose
                                                  // positions begin with 8 - first empty boxes that must not be entered
    int sp = 0;
    while (__any_sync(FULL, cnt != 0)) {
        ++work;
        const bool leaf = base + 7 >= leaf0;
        float key[kGroupC];
        unsigned near = 0xffffffffu;
#pragma unroll
        for (int c = 0; c < kGroupC; ++c) {
            const int g = gl + c * kGroup;
            key[c] = OUT;
            if (g >= 8 - cnt) {
                key[c] = obb_d2(obb + ((size_t)(base >> 3) * 32 + g), xh, xl) * kObbShrink;
                if (key[c] <= bound) near = min(near, (__float_as_uint(key[c]) & ~7u) | g);
                else key[c] = OUT;
            }
        }
#pragma unroll
        for (int o = 1; o < kGroup; o <<= 1) near = min(near, __shfl_xor_sync(FULL, near, o));
        const bool any = near != 0xffffffffu;
        int w = near & 7;
        int node = -1;
        if (any && !leaf) node = base + w;   // enter the nearest, push the others
#pragma unroll
        for (int c = 0; c < kGroupC; ++c) {
            const int g = gl + c * kGroup;
            const bool push = any && !leaf && key[c] <= bound && g != w;
            const unsigned m = (__ballot_sync(FULL, push) >> gs) & kGroupMask;
            if (push) stk[sp + __popc(m & below)] = make_float2(key[c], __int_as_float(base + g));
            sp += __popc(m);
        }
        bool scan = any && leaf;
        while (__any_sync(FULL, scan)) {   // the nearest bucket, then the others that stay within the bound
            float d = INF;
            ++work;
            if (scan) {
                const int j0 = (base + w - leaf0) * kLeaf + gl;
#pragma unroll
                for (int t = 0; t < kLeaf / kGroup; ++t) {
                    const int j = j0 + t * kGroup;
                    if ((unsigned)j < (unsigned)ix.n) d = offer(j, target_point<PREC>(ix, j));
                }
            }
            bound = fminf(bound, d);
#pragma unroll
            for (int o = 1; o < kGroup; o <<= 1) bound = fminf(bound, __shfl_xor_sync(FULL, bound, o));
            unsigned m = 0;
#pragma unroll
            for (int c = 0; c < kGroupC; ++c) {
                if (gl + c * kGroup == w) key[c] = OUT;
                m |= ((__ballot_sync(FULL, scan && key[c] <= bound) >> gs) & kGroupMask) << (c * kGroup);
            }
            scan = m != 0u;
            w = __ffs(m) - 1;
        }
        __syncwarp();
        while (__any_sync(FULL, node < 0 && sp > 0)) {   // pop
            const int k = min(kGroup, sp);
            const float2 e = gl < k ? stk[sp - 1 - gl] : make_float2(OUT, 0.0f);
            const unsigned ok = (__ballot_sync(FULL, e.x <= bound) >> gs) & kGroupMask;
            const int f = __ffs(ok) - 1;
            const int top = __shfl_sync(FULL, __float_as_int(e.y), gs + max(f, 0));
            if (node < 0) {
                sp -= ok ? f + 1 : k;
                if (ok) node = top;
            }
        }
        __syncwarp();
        cnt = node < 0 ? 0 : 8;
        base = 8 * node + 8 * ix.first - 56;
    }
}

// Closest point of a group's query: its bucket-order index, or -1 if no target
// point lies within `bound` (a squared float distance; the distance to a known
// target point for a warm start).
//
// The walk ranks by float distance only: each lane keeps its nearest point and
// the distance of its second nearest. Unless another point lies within the tie
// window of the smallest float distance, the nearest is the winner; ties inside
// the window are ranked as the serial search ranks them, by double-float distance
// and original index, over the lanes' nearest points, or, when a lane has seen
// two such points, by a second walk within the window.
template <int PREC>
__device__ __forceinline__ int group_nn(const Index &ix, const float xh[3], const float xl[3], float bound,
                                        float2 *stk, bool live, int &work) {
    const unsigned FULL = 0xffffffffu;
    const float INF = __int_as_float(0x7f800000);
    const int lane = threadIdx.x & 31;
    const int gs = lane & ~(kGroup - 1);
    const float limit = PREC == PREC_FP64 ? bound * kTieWindow : bound;
    float d1 = INF, d2 = INF;
    int j1 = -1;
    group_walk<PREC>(ix, xh, xl, bound, stk, live, work, [&](int j, float4 p) {
        const float d = point_d2f(xh, xl, p);
        d2 = fminf(d2, fmaxf(d1, d));
        if (d < d1) j1 = j;
        d1 = fminf(d1, d);
        return d1;
    });
    float best = d1;
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) best = fminf(best, __shfl_xor_sync(FULL, best, o));
    const float win = PREC == PREC_FP64 ? best * kTieWindow : best;
    const bool found = live && best <= limit && best < INF;
    const unsigned m1 = (__ballot_sync(FULL, found && d1 <= win) >> gs) & kGroupMask;
    const unsigned m2 = (__ballot_sync(FULL, found && d2 <= win) >> gs) & kGroupMask;
    int j = __shfl_sync(FULL, j1, gs + (m1 ? __ffs(m1) - 1 : 0));
    if (!found) j = -1;
    const bool tie = m2 != 0u || __popc(m1) > 1;
    if (__any_sync(FULL, tie)) {   // rare
        NNLane q;
        nn_init(q, xh, xl);
        const bool again = m2 != 0u;
        if (tie && !again && d1 <= win) nn_seed<PREC>(q, target_point<PREC>(ix, j1), j1);
        if (__any_sync(FULL, again)) {
            float bd = win;
            if (again) q.bestf = best;
            group_walk<PREC>(ix, xh, xl, bd, stk, again, work, [&](int jj, float4 p) {
                nn_offer<PREC>(q, p, jj);
                return win;
            });
        }
#pragma unroll
        for (int o = 1; o < kGroup; o <<= 1) {
            const float oh = __shfl_xor_sync(FULL, q.best_hi, o);
            const float ol = __shfl_xor_sync(FULL, q.best_lo, o);
            const int oo = __shfl_xor_sync(FULL, q.best_orig, o);
            const int oj = __shfl_xor_sync(FULL, q.best_j, o);
            if (lex_less(oh, ol, oo, q.best_hi, q.best_lo, q.best_orig)) {
                q.best_hi = oh;
                q.best_lo = ol;
                q.best_orig = oo;
                q.best_j = oj;
            }
        }
        if (tie) j = q.best_j;
    }
    return j;
}

// ---------------------------------------------------------------------------
// Host-side launchers (index.cu, step.cu). All return cudaError_t.
// ---------------------------------------------------------------------------
struct TargetDev {
    int64_t n;
    int L;
    int has_normals;
    float4 *pts;
    float4 *nrm;
    float4 *nodes;    // 4L float4 of boxes, then the oriented boxes (one allocation)
    float4 *obb;      // = nodes + 4L
    ushort4 *pts16;   // FP16 storage and the oriented boxes of its points, built on first use (build_fp16_storage)
    float4 *obb16;
    double centroid[3];
    float lo[3], hi[3];
    // nu_min statistics in caller units (median over q of the median 6-NN distance,
    // resp. plane distance); < 0 until computed.
    double E_Q, H_Q;
};

inline Index make_index(const TargetDev &t) {
    return Index{t.pts, t.nrm, t.nodes, t.pts16, (int)t.n, t.L, t.obb, wide_first(t.L), wide_leaf(t.L), t.obb16};
}

// Per-thread accounting behind fricp_counters (defined in api.cu).
struct Counters {
    int64_t launches, h2d, d2h;
};
Counters &counters();

// Defined in api.cu: the device view of a target handle, and the message that
// fricp_last_error returns on this thread.
const TargetDev *target_dev(const fricp_target *t);
void set_last_error(const char *msg);

// Stream-ordered device memory from the library's own pool (api.cu). Freed with
// cudaFreeAsync; the pool keeps up to kPoolKeep bytes across synchronisations.
constexpr size_t kPoolKeep = (size_t)256 << 20;
cudaError_t pool_alloc_bytes(void **p, size_t bytes, cudaStream_t s);
size_t pool_idle_bytes();   // held by the current device's pool and in no use: not free to the driver, free to the library
template <class T>
inline cudaError_t pool_alloc(T **p, size_t bytes, cudaStream_t s) {
    return pool_alloc_bytes(reinterpret_cast<void **>(p), bytes, s);
}

cudaError_t build_target(const float *q_dev, const float *n_dev, int64_t n, cudaStream_t s,
                         TargetDev *t, int *bad_input);
cudaError_t target_nu_stats(TargetDev *t, cudaStream_t s);
cudaError_t estimate_normals(const TargetDev *t, int k, const double viewpoint[3], float *out_dev, cudaStream_t s,
                             int *overflow_out);
cudaError_t build_fp16_storage(TargetDev *t, cudaStream_t s);
// Source points in Morton order (and, when n_dev is given, their normals in the
// same order into nrm_out; a normal that is neither zero nor unit length within
// 1e-3 counts as bad input).
cudaError_t prepare_source(const float *p_dev, int64_t m, cudaStream_t s, float4 *src_out,
                           float lo[3], float hi[3], int *bad_input, const float *n_dev = nullptr,
                           float4 *nrm_out = nullptr);
cudaError_t launch_closest(const TargetDev *t, const float *p_dev, int64_t m, const double T[12],
                           int64_t *idx, double *d2, cudaStream_t s);
// One device step: the closest-point search kernel, then the accumulate/solve
// kernel. When `mid` is given it is recorded between the two.
cudaError_t launch_step(const StepArgs &a, int variant, int prec, int ntiles, cudaStream_t s,
                        cudaEvent_t mid = nullptr);
// Median of n non-negative doubles (the mean of the two middle order
// statistics, exact) by a grid-wide 8-bit radix select, of v and, when v2 is
// given, of v2 beside it; `scratch` holds kMedianScratchBytes of device memory,
// the results land in out_dev[0] and out_dev[1].
constexpr int kMedianScratchBytes = 8192;
cudaError_t launch_median(const double *v, const double *v2, int n, void *scratch, double *out_dev, cudaStream_t s);
// After a first pass run with init_median_ext: nu_max from the median at
// *median_dev and the first nu stage (start_after_init).
cudaError_t launch_after_init(PairState *st, const double *median_dev, cudaStream_t s);

}  // namespace fricp

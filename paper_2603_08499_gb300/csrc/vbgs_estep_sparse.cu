// vbgs_estep_sparse.cu -- the CUDA-core E-step and statistics contraction over
// the pairs that matter.
//
// Few of the N x K responsibilities differ from zero: with t = ln K + 37, a
// point has 2 to 36 components with r_nk >= e^-t on the mixture and room
// workloads (0.01% to 4% of the components), and a point loses at most e^-37
// ~ 1e-16 of its mass without the others.  The two passes below find those
// pairs with certified FP32 bounds and spend the form's arithmetic on them
// alone, in both CUDA-core forms:
//   FP64: 1.25 TFLOP/s on this part, one warp instruction per 64 cycles and SM
//         sub-partition whatever its active lanes, so surviving pairs are
//         queued and evaluated 32 at a time, one per lane.
//   FP32: the sums run over the survivors in the order, and with the
//         operations, of the dense passes; a term below e^-37 / K of the sum
//         does not change its FP32 rounding, so the results are the dense
//         ones.
// Three nested tests, all in log2 units and all certified upper bounds of the
// FP32 and FP64 values of the logit (kSlack covers the rounding of the points,
// of the record and of the FP32 quadratic form):
//   1. box of 32 points against the summary of 32 components (lanes take the
//      32 groups of a warp's turn), then against each of those components;
//   2. a pair's position rows (9 of the 27 products), voted over the warp's
//      32 points: i.i.d. colours (the mixture workload) defeat the boxes, the
//      position part alone still rules out nine pairs in ten;
//   3. the pair's full FP32 logit.
// Points and components come in Morton order (unless the caller keeps its
// own), which keeps the boxes small.
// Measured (GB300; pass 1 and pass 2, us a launch), dense -> sparse:
//   FP64, 10,000 points, K = 1,000 (mixture):  1,226 + 2,105 -> 84 + 100
//   FP64, 8,294 points, K = 50,000 (room):    44,100 + 8,650 -> 64 + 101
//   FP32, 36,000 points, K = 50,000 (room):    3,472 +   982 -> 116 + 190
//   FP32, 6,500 points, K = 1,500 (mixture):      52 +   110 -> 67 + 49
// and once per frame the seeds of pass 1: 33, 76 and 117.  Bound: the FP64 pipe
// (about 54 instructions per 32 listed pairs in pass 1, 1.7 + 1 a pair in pass
// 2) on the mixture; latency of the record and box loads on the room.
#include "vbgs_internal.cuh"
#include "vbgs_pair.cuh"
#include <cooperative_groups.h>
#include <algorithm>
#include <cmath>

namespace cg = cooperative_groups;

namespace vbgs {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxPoints = 1 << 24;   // a list entry packs a point index and a component slot
constexpr int kMaxFeatures = 1 << 20; // 235 MB of features
constexpr int kMaxSupers = 256;       // pass 2's masks of eight components stay within 8.3 KB
constexpr int kMaxComps = 1 << 20;    // pass 1's marks (FP32 form) within 128 KB
constexpr int kP2Warps = 8;
constexpr int kCluster = 8;             // blocks a cluster, at most

// Rounding slack.  With |d y| <= e, |y + d y|^2 >= |y|^2 (1 - 1/64) - 63 e^2.
// y = M (x - m) in FP32 is off by at most e = 2^-20 |M|_F (|x| + |m|): 2^-23
// (|x| + |m|) per difference, and 9 further roundings per row.  63/2 e^2 <=
// 33 * 2^-40 * 2 |M|^2 (|x|^2 + |m|^2), and the quadratic term keeps the
// factor 62/64 (the last 1/64 covers the rounding of the sum of squares).
constexpr float kSlack = 6.1e-11f;
constexpr float kQuadLo = 0.484375f;   // 1/2 * 62/64
constexpr float kQuadHi = 0.515625f;   // 1/2 * 66/64

// Arrays of one E-step.  Point side: N padded to Np = 32 G; groups of 32
// points, super groups of 32 groups.  Component side: K padded to Kp = 32 Kg.
// Everything is stored field-major so that 32 lanes read 32 neighbours.
struct SpView {
    const double *X;       // N x 8
    double *phi;           // N x 28: [1, x, upper(x x^T)] (FP64 form; null: too many points)
    int N, Np, G, S;
    float *xf;             // 6 x Np: the points in FP32
    float *gbox, *gx2;     // 12 x G boxes (lo, hi), G largest |x|^2
    float *sbox, *sx2;     // 12 x S, S: the same over 32 groups
    float *thr, *gthr;     // Np, G: lse - t (log2 units), its minimum over a group
    int *sthr;             // S: its minimum over a super group (ordered integer)
    float *lse2f;          // Np: lse in log2 units (FP32 form)
    int *best;             // Np: a component with (nearly) the largest logit of the point
    int K, Kp, Kg;
    float *cb;             // 11 x Kp: m (6), c + slack, lp, lc, la, slack per |x|^2
    float *cg;             // 17 x Kg: lo (6), hi (6), then max, min, min, min, max of the last five
    const double *rec;
    const float *rec32;
    float t2;              // t in log2 units
    int *heavy, *nheavy;   // pass 2: components left to the clusters (K), their number
};

__device__ __forceinline__ int f2ord(float f) { const int i = __float_as_int(f); return i >= 0 ? i : i ^ 0x7fffffff; }
__device__ __forceinline__ float ord2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// Upper bound of the logits between a box of points and a box of means
// (a single mean: mlo = mhi) with the smallest precisions lp, lc, la.
__device__ __forceinline__ float box_bound(const float lo[6], const float hi[6], const float mlo[6], const float mhi[6],
                                           float chi, float lp, float lc, float la)
{
    float dp = 0.f, dc = 0.f;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float o = fmaxf(fmaxf(lo[i] - mhi[i], mlo[i] - hi[i]), 0.f);
        dp = fmaf(o, o, dp);
        const float oc = fmaxf(fmaxf(lo[3 + i] - mhi[3 + i], mlo[3 + i] - hi[3 + i]), 0.f);
        dc = fmaf(oc, oc, dc);
    }
    return chi - kQuadLo * fmaxf(fmaxf(lp * dp, lc * dc), la * (dp + dc));
}

__device__ __forceinline__ float comp_bound(const SpView &V, int k, const float lo[6], const float hi[6], float x2)
{
    float m[6];
#pragma unroll
    for (int i = 0; i < 6; i++) m[i] = V.cb[(size_t)i * V.Kp + k];
    const float *p = V.cb + (size_t)6 * V.Kp + k;
    return box_bound(lo, hi, m, m, fmaf(p[(size_t)4 * V.Kp], x2, p[0]), p[V.Kp], p[(size_t)2 * V.Kp], p[(size_t)3 * V.Kp]);
}

__device__ __forceinline__ float group_bound(const SpView &V, int q, const float lo[6], const float hi[6], float x2)
{
    float a[6], b[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        a[i] = V.cg[(size_t)i * V.Kg + q];
        b[i] = V.cg[(size_t)(6 + i) * V.Kg + q];
    }
    const float *p = V.cg + (size_t)12 * V.Kg + q;
    return box_bound(lo, hi, a, b, fmaf(p[(size_t)4 * V.Kg], x2, p[0]), p[V.Kg], p[(size_t)2 * V.Kg], p[(size_t)3 * V.Kg]);
}

// Feature f of 28: the product of columns ia, ib of [1, x].
__device__ __forceinline__ void feature_cols(int f, int &ia, int &ib)
{
    ia = f >= 1 && f < 7 ? f : 0;
    ib = 0;
    int u = 7;
#pragma unroll
    for (int a = 0; a < 6; a++)
#pragma unroll
        for (int b = a; b < 6; b++, u++)
            if (f == u) { ia = a + 1; ib = b + 1; }
}

// Points to FP32, boxes per 32 and per 1,024 points.  One block per super
// group, a warp per group: latency bound (one pass over 64 N bytes).
__global__ void __launch_bounds__(1024) k_sp_points(SpView V)
{
    pdl_wait();
    __shared__ float sh[13][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, s = blockIdx.x, g = s * 32 + w;
    float b[13];
#pragma unroll
    for (int i = 0; i < 6; i++) { b[i] = INFINITY; b[6 + i] = -INFINITY; }
    b[12] = 0.f;
    if (g < V.G) {
        const int n = g * 32 + lane;
        const double *x = V.X + (size_t)min(n, V.N - 1) * VBGS_XS;
        float x2 = 0.f;
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const float v = (float)x[i];
            V.xf[(size_t)i * V.Np + n] = v;
            x2 = fmaf(v, v, x2);
            b[i] = -warp_max(-v);
            b[6 + i] = warp_max(v);
        }
        b[12] = warp_max(x2) * 1.000001f;
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < 12; i++) V.gbox[(size_t)i * V.G + g] = b[i];
            V.gx2[g] = b[12];
        }
    }
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 13; i++) sh[i][w] = b[i];
    __syncthreads();
    if (w < 13) {
        const float v = sh[w][lane];
        const float r = w < 6 ? warp_min(v) : warp_max(v);
        if (lane == 0) (w < 12 ? V.sbox[(size_t)w * V.S + s] : V.sx2[s]) = r;
    }
}

// The features of every point, once per frame: pass 2 then spends one FP64
// instruction a pair on its statistics instead of two.
__global__ void __launch_bounds__(256) k_sp_features(SpView V)
{
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= (int64_t)V.N * 28) return;
    const int n = (int)(i / 28), f = (int)(i - (int64_t)n * 28);
    int ia, ib;
    feature_cols(f, ia, ib);
    const double *x = V.X + (size_t)n * VBGS_XS;
    const double a = ia ? x[ia - 1] : 1.0;
    V.phi[i] = ib ? a * x[ib - 1] : a;
}

// Bound terms of every component and of every 32 (a warp each); also resets
// the super groups' threshold minima and the heavy count for the passes that
// follow.
__global__ void __launch_bounds__(128) k_sp_comps(SpView V)
{
    pdl_wait();
    const int lane = threadIdx.x & 31, q = blockIdx.x * 4 + (threadIdx.x >> 5);
    for (int s = blockIdx.x * 128 + threadIdx.x; s < V.S; s += gridDim.x * 128) V.sthr[s] = 0x7fffffff;
    if (blockIdx.x == 0 && threadIdx.x == 0) *V.nheavy = 0;
    if (q >= V.Kg) return;
    const int k = q * 32 + lane;
    const bool valid = k < V.K;
    float r[VBGS_REC];   // a 128-byte row per lane, eight loads in flight (K = 50,000: 9.3 -> 4.9 us)
    {
        const float4 *r4 = reinterpret_cast<const float4 *>(V.rec32 + (size_t)min(k, V.K - 1) * VBGS_REC);
#pragma unroll
        for (int i = 0; i < VBGS_REC / 4; i++) {
            const float4 f = r4[i];
            r[4 * i] = f.x; r[4 * i + 1] = f.y; r[4 * i + 2] = f.z; r[4 * i + 3] = f.w;
        }
    }
    float m2 = 0.f, M2 = 0.f, v[11];
#pragma unroll
    for (int i = 0; i < 6; i++) { v[i] = r[i]; m2 = fmaf(v[i], v[i], m2); }
#pragma unroll
    for (int i = 0; i < 21; i++) M2 = fmaf(r[6 + i], r[6 + i], M2);
    v[10] = kSlack * M2;
    v[6] = r[27] + fabsf(r[27]) * 2.5e-7f + v[10] * m2;
    v[7] = r[28]; v[8] = r[29]; v[9] = r[30];
    if (valid)
#pragma unroll
        for (int i = 0; i < 11; i++) V.cb[(size_t)i * V.Kp + k] = v[i];
    float o[17];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        o[i] = -warp_max(valid ? -v[i] : -INFINITY);
        o[6 + i] = warp_max(valid ? v[i] : -INFINITY);
    }
    o[12] = warp_max(valid ? v[6] : -INFINITY);
#pragma unroll
    for (int i = 0; i < 3; i++) o[13 + i] = warp_min(valid ? v[7 + i] : INFINITY);
    o[16] = warp_max(valid ? v[10] : 0.f);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 17; i++) V.cg[(size_t)i * V.Kg + q] = o[i];
}

// The walk of pass 1 and of its seed kernel: a block holds 32 points, one per
// lane of every warp, and its warps share the components in units of 32, 16
// or 8 neighbours (nsub units a group, so that few components still occupy
// every warp).  Lanes test 32 units at a time against the block's box, then
// each point against the unit's group (a box across a jump of the Morton order
// reaches groups that none of its points does), then the unit's components
// against the box.  Candidates collect in shared memory; the records of kStage
// of them are staged with one latency and take the pair tests.
constexpr int kP1Warps = 16;    // at most
constexpr int kStage = 16;      // records staged at once
constexpr int kWalkBytes = kStage * 112 + 512;   // shared memory of a warp: records, candidates

struct Walk {
    float *stage;     // kStage x 28
    int *cand;        // 64 components
    float *candc;     // 64: c + slack
    int nc = 0;

    __device__ Walk(unsigned char *smem, int W, int w)
    {
        stage = reinterpret_cast<float *>(smem) + w * kStage * 28;
        cand = reinterpret_cast<int *>(smem + (size_t)W * kStage * 112) + w * 64;
        candc = reinterpret_cast<float *>(smem + (size_t)W * (kStage * 112 + 256)) + w * 64;
    }
    // the records of candidates [0, cnt)
    __device__ __forceinline__ void stage_in(const SpView &V, int cnt, int lane)
    {
        __syncwarp();
        for (int i = lane; i < cnt * 7; i += 32) {
            const int c = i / 7, f = i - 7 * c;
            reinterpret_cast<float4 *>(stage)[i] =
                reinterpret_cast<const float4 *>(V.rec32 + (size_t)cand[c] * VBGS_REC)[f];
        }
        __syncwarp();
    }
    __device__ __forceinline__ void push(const SpView &V, bool in, int k, float x2, int lane)
    {
        const unsigned m = __ballot_sync(kFull, in);
        if (in) {
            const int at = nc + __popc(m & ((1u << lane) - 1u));
            cand[at] = k;
            candc[at] = fmaf(V.cb[(size_t)10 * V.Kp + k], x2, V.cb[(size_t)6 * V.Kp + k]);
        }
        nc += __popc(m);
    }
    // drop the kStage candidates just tested
    __device__ __forceinline__ void shift(int lane)
    {
        nc -= kStage;
        const int k = cand[kStage + lane];
        const float c = candc[kStage + lane];
        __syncwarp();
        if (lane < nc) { cand[lane] = k; candc[lane] = c; }
        __syncwarp();
    }
    // Every candidate whose bounds reach thr (per lane; bthr its minimum, kept
    // by test(cnt), which takes candidates [0, cnt)).  Warp tw of TW.
    template <typename Test>
    __device__ __forceinline__ void run(const SpView &V, int nsub, int tw, int TW, const float x[6], const float lo[6],
                                        const float hi[6], float x2, bool valid, const float &thr, const float &bthr,
                                        int lane, Test &&test)
    {
        const int units = V.Kg * nsub, ucomp = 32 / nsub;
        for (int u0 = 0; u0 < units; u0 += 32 * TW) {
            const int u = u0 + lane * TW + tw;
            unsigned m1 = __ballot_sync(kFull, u < units && !(group_bound(V, min(u / nsub, V.Kg - 1), lo, hi, x2) < bthr));
            while (m1) {
                const int uu = u0 + (__ffs(m1) - 1) * TW + tw;
                m1 &= m1 - 1;
                const int q = uu / nsub, k = q * 32 + lane, kc = min(k, V.K - 1), b0 = uu % nsub * ucomp;
                if (!__any_sync(kFull, valid && !(group_bound(V, q, x, x, x2) < thr))) continue;
                push(V, lane >= b0 && lane < b0 + ucomp && k < V.K && !(comp_bound(V, kc, lo, hi, x2) < bthr), k, x2, lane);
                while (nc >= kStage) {
                    test(kStage);
                    shift(lane);
                }
            }
        }
        if (nc) test(nc);
        nc = 0;
    }
};

// The component with the largest FP32 logit of every point, where no earlier
// E-step of the frame has left one (SpView::best): pass 1's thresholds start
// from it, and how close they are decides how many pairs it tests.
//   1. every warp takes its kSeedUnits units with the largest bounds (the best
//      of each lane's share), and each lane the component with the largest
//      bound among them; the block scores these;
//   2. branch and bound: the walk over all components whose bound reaches a
//      point's largest logit so far, shared by the block as (logit, component).
// A bound never lies below the FP32 logit, so the result is the exact maximum
// (ties to the lower component) whatever the order of the updates.
constexpr int kSeedWarps = 8, kSeedUnits = 4;

__global__ void __launch_bounds__(kSeedWarps * 32) k_sp_seed(SpView V, int nsub)
{
    pdl_wait();
    constexpr int W = kSeedWarps;
    __shared__ __align__(16) unsigned char sraw[W * kWalkBytes];
    __shared__ unsigned long long sbest[32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = blockIdx.x, n = g * 32 + lane;
    const bool valid = n < V.N;
    Walk K(sraw, W, w);
    float x[6], lo[6], hi[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        x[i] = V.xf[(size_t)i * V.Np + n];
        lo[i] = V.gbox[(size_t)i * V.G + g];
        hi[i] = V.gbox[(size_t)(6 + i) * V.G + g];
    }
    const float x2 = V.gx2[g];
    if (threadIdx.x < 32) sbest[threadIdx.x] = 0ull;
    __syncthreads();
    auto pack = [](float l, int k) {   // larger logit, then lower component
        return (unsigned long long)((unsigned)f2ord(l) ^ 0x80000000u) << 32 | (unsigned)~k;
    };
    auto logit_of = [](unsigned long long p) { return ord2f((int)((unsigned)(p >> 32) ^ 0x80000000u)); };
    unsigned long long mine = pack(-INFINITY, 0);
    // 1. (bounds and logits without NaN: a non-finite point)
    float ub = -INFINITY;
    int bu = -1;
    const int units = V.Kg * nsub, ucomp = 32 / nsub;
    for (int u = lane * W + w; u < units; u += 32 * W) {
        const float v = fmaxf(group_bound(V, u / nsub, lo, hi, x2), -INFINITY);
        if (v > ub || bu < 0) { ub = v; bu = u; }
    }
    float cu = -INFINITY;
    int ck = -1;
    for (int i = 0; i < kSeedUnits; i++) {
        const float top = warp_max(bu >= 0 ? ub : -INFINITY);
        const unsigned m = __ballot_sync(kFull, bu >= 0 && ub == top);
        if (!m) break;
        const int src = __ffs(m) - 1, u = __shfl_sync(kFull, bu, src);
        if (lane == src) bu = -1;
        const int k = u / nsub * 32 + lane, b0 = u % nsub * ucomp;
        if (lane >= b0 && lane < b0 + ucomp && k < V.K) {
            const float v = fmaxf(comp_bound(V, k, lo, hi, x2), -INFINITY);
            if (v > cu || ck < 0) { cu = v; ck = k; }
        }
    }
    auto score = [&](int cnt) {
        K.stage_in(V, cnt, lane);
        for (int i = 0; i < cnt; i++) {
            const unsigned long long p = pack(fmaxf(logit<float>(K.stage + i * 28, x), -INFINITY), K.cand[i]);
            mine = p > mine ? p : mine;
        }
    };
    K.push(V, ck >= 0, ck, x2, lane);
    while (K.nc >= kStage) {
        score(kStage);
        K.shift(lane);
    }
    if (K.nc) score(K.nc);
    K.nc = 0;
    atomicMax(&sbest[lane], mine);
    __syncthreads();
    // 2.
    mine = *(volatile unsigned long long *)&sbest[lane];
    float thr = valid ? logit_of(mine) : INFINITY, bthr = warp_min(thr);
    K.run(V, nsub, w, W, x, lo, hi, x2, valid, thr, bthr, lane, [&](int cnt) {
        K.stage_in(V, cnt, lane);
        for (int i = 0; i < cnt; i++) {
            const float *r = K.stage + i * 28, c = K.candc[i];
            float q = quad_pos(r, x);
            if (!__any_sync(kFull, valid && !(c - kQuadLo * q < thr))) continue;
            q = quad_rest(r, x, q);
            const unsigned long long p = pack(fmaxf(fmaf(-0.5f, q, r[27]), -INFINITY), K.cand[i]);
            if (p > mine) {
                mine = p;
                atomicMax(&sbest[lane], p);
            }
        }
        const unsigned long long p = *(volatile unsigned long long *)&sbest[lane];
        mine = p > mine ? p : mine;
        if (valid) thr = logit_of(mine);
        bthr = warp_min(thr);
    });
    __syncthreads();
    if (w == 0) V.best[n] = (int)~(unsigned)sbest[lane];
}

// Pass 1: lse_n.  A point's threshold lse - t starts from the logit of its
// component `best` and rises with the largest certified logit each warp meets.
//   FP64: the pairs found go to the warp's list.  The block then evaluates the
//     pairs that also reach the final threshold, from the lists of all its
//     warps, in full batches of 32, one pair per lane: sum_k exp(l_k - ref)
//     with ref the largest certified logit (a term above e^64 first moves the
//     reference).  Terms of one point are added in list order.  A cluster of
//     up to eight blocks shares the units of one point group when the groups
//     alone do not spread over the SMs (their FP64 pipes): 313 blocks leave
//     some SMs three and others two; the sums meet in the first block.
//   FP32: the components found are marked, and each warp then takes whole K
//     splits of the dense pass (kps components) over the marks, lanes keeping
//     their online (max, sum); the partials are merged in FP64.
// The component of the largest certified logit replaces `best` for the next
// iteration.
constexpr int kList = 384;      // pairs a warp lists before it evaluates some itself
struct P1Args {
    int nsub;
    int kps, nsplit;       // FP32
    double2 *part;         // FP32: nsplit x N
    double *lse, *lse_part, *sum_out;
    unsigned int *done;
    unsigned long long *pairs;
};
__host__ __device__ constexpr size_t p1_warp_bytes(bool f64)
{
    return (size_t)kWalkBytes + 256 + (f64 ? 512 + kList * 8 : 0);
}

template <typename T>
__global__ void __launch_bounds__(kP1Warps * 32, 2) k_sp_pass1(SpView V, P1Args A)
{
    pdl_wait();
    constexpr bool kF64 = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double sx[32 * 6], red[kP1Warps], bref[32], bsum[32];
    __shared__ int scount[kP1Warps], bkm[32];
    __shared__ float bmx[32];
    __shared__ bool last;
    cg::cluster_group cluster = cg::this_cluster();
    const int nblk = kF64 ? (int)cluster.num_blocks() : 1, rank = kF64 ? (int)cluster.block_rank() : 0;
    const int W = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = blockIdx.x / nblk;
    // per warp: the walk's, largest certified logits; FP64: references, sums, list (pair, upper bound)
    Walk K(smem_raw, W, w);
    float *sm = reinterpret_cast<float *>(smem_raw + (size_t)W * kWalkBytes);
    int *sk = reinterpret_cast<int *>(sm + W * 32);
    double *sref = reinterpret_cast<double *>(sk + W * 32), *ssum = sref + W * 32;
    uint2 *list = reinterpret_cast<uint2 *>(ssum + W * 32);                // FP64: W x kList
    unsigned *mark = reinterpret_cast<unsigned *>(sk + W * 32);            // FP32: Kg words
    const int n = g * 32 + lane;
    const bool valid = n < V.N;
    float x[6], lo[6], hi[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        x[i] = V.xf[(size_t)i * V.Np + n];
        lo[i] = V.gbox[(size_t)i * V.G + g];
        hi[i] = V.gbox[(size_t)(6 + i) * V.G + g];
    }
    const float x2 = V.gx2[g];
    int km = V.best[n];
    // the largest certified logit: a lower bound of the exact one (FP64 form:
    // c less the slack, the quadratic form inflated) or the FP32 value itself
    float mx;
    {
        const float *r = V.rec32 + (size_t)km * VBGS_REC;
        if (kF64) {
            const float q = quad_rest(r, x, quad_pos(r, x));
            mx = 2.f * r[27] - fmaf(V.cb[(size_t)10 * V.Kp + km], x2, V.cb[(size_t)6 * V.Kp + km]) - kQuadHi * q;
        } else {
            mx = logit<float>(r, x);
        }
    }
    if constexpr (kF64) {
        for (int i = threadIdx.x; i < 192; i += blockDim.x)
            sx[i] = V.X[(size_t)min(g * 32 + i / 6, V.N - 1) * VBGS_XS + i % 6];
        ssum[w * 32 + lane] = 0.0;
        sref[w * 32 + lane] = (double)(mx * 0.693147f);
    } else {
        for (int i = threadIdx.x; i < V.Kg; i += blockDim.x) mark[i] = 0u;
    }
    __syncthreads();
    float thr = valid ? mx - V.t2 : INFINITY;
    float bthr = warp_min(thr);
    unsigned npair = 0;
    bool early = false;   // FP64: this warp has evaluated pairs before the end of its walk

    double *ref = sref + w * 32, *sum = ssum + w * 32;
    uint2 *mylist = list + w * kList;
    // FP64: one listed pair per lane (act), into this warp's references and sums
    auto evaluate = [&](bool act, unsigned e) {
        const int k = (int)(e >> 5), p = (int)(e & 31u);
        double x6[6], r[28];
#pragma unroll
        for (int i = 0; i < 6; i++) x6[i] = sx[p * 6 + i];
        const double2 *rp = reinterpret_cast<const double2 *>(V.rec + (size_t)k * VBGS_REC);
#pragma unroll
        for (int i = 0; i < 14; i++) { const double2 v = rp[i]; r[2 * i] = v.x; r[2 * i + 1] = v.y; }
        const double l = logit<double>(r, x6);
        double rf = ref[p];
        unsigned over = __ballot_sync(kFull, act && l > rf + 64.0);
        if (over) {
            for (int i = 0; i < 32; i++) {
                const double le = __shfl_sync(kFull, l, i);
                const int pe = __shfl_sync(kFull, p, i);
                if (lane == 0 && (over >> i & 1u) && le > ref[pe] + 64.0) { sum[pe] *= exp(ref[pe] - le); ref[pe] = le; }
            }
            __syncwarp();
            rf = ref[p];
        }
        const double v = exp(l - rf);
        // add the terms point by point, in list order
        const unsigned peers = __match_any_sync(kFull, act ? p : 32 + lane);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        const int ranks = __reduce_max_sync(kFull, act ? rank : 0);
        for (int i = 0; i <= ranks; i++) {
            if (act && rank == i) sum[p] += v;
            __syncwarp();
        }
    };

    // ---- walk ----
    int ln = 0;
    K.run(V, A.nsub, rank * W + w, W * nblk, x, lo, hi, x2, valid, thr, bthr, lane, [&](int cnt) {
        K.stage_in(V, cnt, lane);
        for (int i = 0; i < cnt; i++) {
            const int k = K.cand[i];
            const float *r = K.stage + i * 28, c = K.candc[i];
            float qd = quad_pos(r, x);
            if (!__any_sync(kFull, valid && !(c - kQuadLo * qd < thr))) continue;
            qd = quad_rest(r, x, qd);
            const float up = c - kQuadLo * qd;
            const bool surv = valid && !(up < thr);
            const unsigned ms = __ballot_sync(kFull, surv);
            if (!ms) continue;
            const float l = kF64 ? 2.f * r[27] - c - kQuadHi * qd : fmaf(-0.5f, qd, r[27]);
            if (valid && l > mx) {
                mx = l;
                km = k;
                thr = mx - V.t2;
            }
            if constexpr (kF64) {
                if (surv) mylist[ln + __popc(ms & ((1u << lane) - 1u))] =
                    make_uint2((unsigned)k << 5 | (unsigned)lane, __float_as_uint(up));
                ln += __popc(ms);
                if (ln > kList - 32) {
                    __syncwarp();
                    ln -= 32;
                    evaluate(true, mylist[ln + lane].x);
                    npair += 32;
                    early = true;
                }
            } else {
                if (lane == 0) atomicOr(&mark[k >> 5], 1u << (k & 31));
            }
        }
        bthr = warp_min(thr);
        __syncwarp();
    });

    // the block's largest certified logits
    sm[w * 32 + lane] = mx;
    sk[w * 32 + lane] = km;
    __syncthreads();
    for (int i = 0; i < W; i++)
        if (sm[i * 32 + lane] > mx) { mx = sm[i * 32 + lane]; km = sk[i * 32 + lane]; }
    if (kF64 && nblk > 1) {   // and the cluster's
        if (w == 0) { bmx[lane] = mx; bkm[lane] = km; }
        cluster.sync();
        for (int i = 0; i < nblk; i++) {
            const float v = cluster.map_shared_rank(bmx, i)[lane];
            if (v > mx) { mx = v; km = cluster.map_shared_rank(bkm, i)[lane]; }
        }
    }

    // ---- sums ----
    if constexpr (kF64) {
        if (!early) ref[lane] = (double)(mx * 0.693147f);
        // keep the listed pairs that reach the final threshold
        const float fthr = valid ? mx - V.t2 : INFINITY;
        int kept = 0;
        for (int i0 = 0; i0 < ln; i0 += 32) {
            const uint2 e = mylist[min(i0 + lane, ln - 1)];
            const bool keep = !(__uint_as_float(e.y) < __shfl_sync(kFull, fthr, e.x & 31u)) && i0 + lane < ln;
            const unsigned m = __ballot_sync(kFull, keep);
            if (keep) mylist[kept + __popc(m & ((1u << lane) - 1u))] = e;
            kept += __popc(m);
            __syncwarp();
        }
        if (lane == 0) scount[w] = kept;
        __syncthreads();
        // batches of 32 over the concatenated lists, dealt to the warps
        int total = 0;
        for (int i = 0; i < W; i++) total += scount[i];
        for (int b = w * 32; b < total; b += W * 32) {
            int at = b + lane, i = 0;
            const bool act = at < total;
            if (!act) at = total - 1;
            while (at >= scount[i]) at -= scount[i++];
            evaluate(act, list[i * kList + at].x);
            npair += min(32, total - b);
        }
    } else {
        for (int s = w; s < A.nsplit; s += W) {
            const int k0 = s * A.kps, k1 = min(V.K, k0 + A.kps);
            float m = -INFINITY, sum32 = 0.f;
            for (int q0 = k0 >> 5; q0 * 32 < k1; q0 += 32) {
                const unsigned mk = (q0 + lane) * 32 < k1 ? mark[q0 + lane] : 0u;
                unsigned m1 = __ballot_sync(kFull, mk != 0u);
                while (m1) {
                    const int b = __ffs(m1) - 1, kb = (q0 + b) * 32;
                    m1 &= m1 - 1;
                    unsigned m2 = __shfl_sync(kFull, mk, b);
                    if (kb < k0) m2 &= kFull << (k0 - kb);
                    if (kb + 32 > k1) m2 &= kFull >> (kb + 32 - k1);
                    while (m2) {
                        const int at = __popc(m2 & ((1u << lane) - 1u));
                        const bool sel = (m2 >> lane & 1u) && at < kStage;
                        __syncwarp();
                        if (sel) K.cand[at] = kb + lane;
                        const unsigned ms = __ballot_sync(kFull, sel);
                        m2 &= ~ms;
                        const int cnt = __popc(ms);
                        K.stage_in(V, cnt, lane);
                        npair += 32 * cnt;
                        for (int i = 0; i < cnt; i++) {
                            const float l = logit<float>(K.stage + i * 28, x);
                            if (l > m) {
                                sum32 = fmaf(sum32, ex2_approx(m - l), 1.f);
                                m = l;
                            } else {
                                sum32 += ex2_approx(l - m);
                            }
                        }
                    }
                }
            }
            if (valid) {
                double2 o = make_double2(-INFINITY, 0.0);
                if (!(sum32 == 0.f)) o = make_double2((double)m / (double)Arith<float>::lse_scale(), (double)sum32);
                A.part[(size_t)s * V.N + n] = o;
            }
        }
    }
    __syncthreads();

    // ---- merge ----
    if constexpr (kF64) {
        // (reference, sum) pairs of the block's warps, then of the cluster's blocks
        auto merge = [&](int cnt, auto &&rf, auto &&sf, double &R, double &s) {
            R = rf(0);
            s = 0.0;
            bool same = true;
            for (int i = 1; i < cnt; i++) same = same && __double_as_longlong(rf(i)) == __double_as_longlong(R);
            if (__all_sync(kFull, same)) {
                for (int i = 0; i < cnt; i++) s += sf(i);
            } else {
                for (int i = 1; i < cnt; i++) R = fmax(R, rf(i));
                for (int i = 0; i < cnt; i++) s += sf(i) * exp(rf(i) - R);
            }
        };
        double R, s;
        if (w == 0) {
            merge(W, [&](int i) { return sref[i * 32 + lane]; }, [&](int i) { return ssum[i * 32 + lane]; }, R, s);
            bref[lane] = R;
            bsum[lane] = s;
        }
        if (nblk > 1) {
            cluster.sync();
            if (rank == 0 && w == 0) {
                merge(nblk, [&](int i) { return cluster.map_shared_rank(bref, i)[lane]; },
                      [&](int i) { return cluster.map_shared_rank(bsum, i)[lane]; }, R, s);
                bref[lane] = R;   // (only this block's own entry, read above)
                bsum[lane] = s;
            }
            cluster.sync();   // the sums are read before their blocks leave
        }
        if (w == 0) __syncwarp();
    }
    if (w == 0 && rank == 0) {
        double R = -INFINITY, s = 0.0, v = 0.0;
        if constexpr (kF64) {
            R = bref[lane];
            s = bsum[lane];
        } else if (valid) {
            for (int j = 0; j < A.nsplit; j++) R = fmax(R, A.part[(size_t)j * V.N + n].x);
            for (int j = 0; j < A.nsplit; j++) {
                const double2 p = A.part[(size_t)j * V.N + n];
                if (p.y > 0.0) s += p.y * exp(p.x - R);
            }
        }
        float t = INFINITY;
        if (valid) {
            v = R + log(s);
            A.lse[n] = v;
            const float l2 = (float)(v * 1.4426950408889634);
            t = l2 - fabsf(l2) * 2.5e-7f - V.t2;
            if (!kF64) V.lse2f[n] = (float)(v * (double)Arith<float>::lse_scale());
        }
        V.thr[n] = t;
        V.best[n] = km;
        t = warp_min(t);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
        if (lane == 0) {
            V.gthr[g] = t;
            atomicMin(&V.sthr[g >> 5], f2ord(t));
            if (A.lse_part) A.lse_part[g] = v;
        }
    }
    if (A.pairs && lane == 0) atomicAdd(A.pairs, (unsigned long long)npair);
    if (!A.sum_out || rank) return;
    // the groups' sums, added in order by the last block to finish
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(A.done, 1u) == (unsigned)V.G - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t = 0.0;
    for (int i = threadIdx.x; i < V.G; i += blockDim.x) t += __ldcg(A.lse_part + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(kFull, t, o);
    if (lane == 0) red[w] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int i = 0; i < W; i++) tot += red[i];
        *A.sum_out = tot;
        *A.done = 0u;
    }
}

// Pass 2: Delta S.  Pairs are found per component (its record) over the point
// groups whose box bound reaches their threshold, with the next group's points
// in flight, and listed; 32 are evaluated at once: r = exp(l - lse) one pair
// per lane, then the statistics with one feature per lane, pair after pair.
// FP64: a block's lists are evaluated together, in full batches.  FP32: a warp
// takes whole N splits of the dense pass, whose sums are FP32.  The sums of a
// component stay on chip; its FP64 sums are added in a fixed order.
//   wide: a block of eight warps per eight neighbouring components.  A warp
//     tests one component against the super groups and groups of points (bit
//     masks); then every warp walks its share (FP64: groups g = w mod 8).  Most
//     components of a large map reach a few groups or none.  One that reaches
//     more than kHeavy groups goes to a list instead: a block held by it would
//     outlast the rest of the grid.
//   single: a cluster of up to eight blocks of four warps per component (of
//     that list, or all of them when there are few); each of the 32 warps takes
//     every 32nd group (FP32: split), the blocks' sums meet in the first
//     block over distributed shared memory.
constexpr int kHeavy = 32;
constexpr int kOneWarps = 4;
struct P2Args {
    int nps, nsplit;       // FP32: points per split, splits
    int nw, nzw;           // mask words per component, words of the mask of nonzero words
    const double *lse;
    bool anchored;         // FP32 form: moments about the record's mean
    const int *kperm;
    double *dS;
    int *heavy, *nheavy;   // positions of the heavy components, their number; null: every component is single
    unsigned long long *pairs;
};

// A component's sums s (feature per lane) to its row of Delta S; anchored:
// moments about m, shifted to raw moments: S1 = S1' + N m,
// S2 = S2' + m S1'^T + S1' m^T + N m m^T.
__device__ __forceinline__ void write_row(const SpView &V, const P2Args &A, int p, double s, bool any,
                                          const float *m, int lane)
{
    if (A.anchored && any) {
        int ia, ib;
        feature_cols(lane, ia, ib);
        const double nn = __shfl_sync(kFull, s, 0);
        const double sa1 = __shfl_sync(kFull, s, ia), sb1 = __shfl_sync(kFull, s, ib);
        const double aa = ia ? (double)m[ia - 1] : 0.0, ab = ib ? (double)m[ib - 1] : 0.0;
        if (ib) s += aa * sb1 + sa1 * ab + nn * aa * ab;
        else if (ia) s += nn * aa;
    }
    if (lane < 28) A.dS[(size_t)(A.kperm ? A.kperm[p] : p) * 28 + lane] = s;
}

// One pair per lane, point n under the record r: its responsibility and its
// row of [1, x] (FP32 form: d, x about the record's mean) and, in the FP32
// form, w times that row.  FP64 with the feature table: w and n only.
template <typename T>
__device__ __forceinline__ void weigh(const SpView &V, const double *__restrict__ lse, const T *r, int n, T *ws, int *ns, T *xs)
{
    T xv[6], ref;
    if constexpr (sizeof(T) == 8) {
        const double2 *xp = reinterpret_cast<const double2 *>(V.X + (size_t)n * VBGS_XS);
#pragma unroll
        for (int i = 0; i < 3; i++) { const double2 v = xp[i]; xv[2 * i] = v.x; xv[2 * i + 1] = v.y; }
        ref = lse[n];
    } else {
#pragma unroll
        for (int i = 0; i < 6; i++) xv[i] = V.xf[(size_t)i * V.Np + n];
        ref = V.lse2f[n];
    }
    const T w = Arith<T>::expd(logit<T>(r, xv) - ref);
    if constexpr (sizeof(T) == 8) {
        *ws = w;
        *ns = n;
        if (V.phi) return;
        xs[0] = 1.0;
#pragma unroll
        for (int i = 0; i < 6; i++) xs[1 + i] = xv[i];
    } else {
        xs[0] = 1.f;
        ws[0] = w;
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const float d = xv[i] - r[i];
            xs[1 + i] = d;
            ws[1 + i] = w * d;
        }
    }
}
// Pair e's term of feature (ia, ib) added to acc, the dense passes'
// operations.  FP64: fma(w, x_a x_b); FP32: fma(w d_a, d_b), d_b = 1 for the
// lower orders (an exact sum).
template <typename T>
__device__ __forceinline__ T add_pair(const SpView &V, T acc, const T *ws, const int *ns, const T *xs, int e, int ia,
                                      int ib, int lane)
{
    if constexpr (sizeof(T) == 8) {
        const double p = V.phi ? V.phi[(size_t)ns[e] * 28 + min(lane, 27)] : xs[e * 7 + ia] * xs[e * 7 + ib];
        return fma(ws[e], p, acc);
    } else {
        return fmaf(ws[e * 7 + ia], xs[e * 7 + ib], acc);
    }
}
template <typename T>
__global__ void __launch_bounds__(kP2Warps * 32, 4) k_sp_pass2(SpView V, P2Args A)
{
    pdl_wait();
    constexpr bool kF64 = sizeof(T) == 8;
    constexpr int W = kP2Warps, C = kP2Warps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double sacc[W * C * 28];
    __shared__ T srec[C * 28];
    __shared__ float srec32[C * 28], schi[C], sb[C];
    __shared__ T sx[W][32 * 7], sw[W][32 * (kF64 ? 1 : 7)];   // rows of 7: [1, x]; w (times the row)
    __shared__ unsigned sq[W][64];
    __shared__ int stag[W][64], sn[W][32];
    __shared__ unsigned used[W];     // bit c: warp w holds a sum of component c
    __shared__ int scount[W];
    __shared__ bool sheavy[C];
    unsigned *mask = reinterpret_cast<unsigned *>(smem_raw), *nz = mask + C * A.nw;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, p0 = blockIdx.x * C;
    for (int i = threadIdx.x; i < C * (A.nw + A.nzw); i += W * 32) mask[i] = 0u;
    for (int i = threadIdx.x; i < C * 28; i += W * 32) {
        const int p = min(p0 + i / 28, V.K - 1);
        srec32[i] = V.rec32[(size_t)p * VBGS_REC + i % 28];
        srec[i] = kF64 ? (T)V.rec[(size_t)p * VBGS_REC + i % 28] : (T)srec32[i];
    }
    if (threadIdx.x < C) {
        const int p = min(p0 + (int)threadIdx.x, V.K - 1);
        schi[threadIdx.x] = V.cb[(size_t)6 * V.Kp + p];
        sb[threadIdx.x] = V.cb[(size_t)10 * V.Kp + p];
    }
    if (lane == 0) used[w] = 0u;
    // ---- point groups per component (one per warp) ----
    bool any = false;
    {
        const int p = p0 + w;
        float m[6], chi = 0.f, lp = 0.f, lc = 0.f, la = 0.f, B = 0.f;
        if (p < V.K) {
#pragma unroll
            for (int i = 0; i < 6; i++) m[i] = V.cb[(size_t)i * V.Kp + p];
            chi = V.cb[(size_t)6 * V.Kp + p]; lp = V.cb[(size_t)7 * V.Kp + p]; lc = V.cb[(size_t)8 * V.Kp + p];
            la = V.cb[(size_t)9 * V.Kp + p]; B = V.cb[(size_t)10 * V.Kp + p];
        }
        __syncthreads();   // the masks are clear
        int reached = 0;
        if (p < V.K) {
            auto reaches = [&](const float *box, int stride, int at, float xx, float t) {
                float lo[6], hi[6];
#pragma unroll
                for (int i = 0; i < 6; i++) {
                    lo[i] = box[(size_t)i * stride + at];
                    hi[i] = box[(size_t)(6 + i) * stride + at];
                }
                return !(box_bound(lo, hi, m, m, fmaf(B, xx, chi), lp, lc, la) < t);
            };
            for (int s0 = 0; s0 < V.S; s0 += 32) {
                const int s = min(s0 + lane, V.S - 1);
                unsigned m1 = __ballot_sync(kFull, s0 + lane < V.S && reaches(V.sbox, V.S, s, V.sx2[s], ord2f(V.sthr[s])));
                while (m1) {
                    const int sg = s0 + __ffs(m1) - 1;
                    m1 &= m1 - 1;
                    const int g = sg * 32 + lane, gc = min(g, V.G - 1);
                    const unsigned b = __ballot_sync(kFull, g < V.G && reaches(V.gbox, V.G, gc, V.gx2[gc], V.gthr[gc]));
                    reached += __popc(b);
                    if (b && lane == 0) {
                        mask[w * A.nw + sg] = b;
                        nz[w * A.nzw + (sg >> 5)] |= 1u << (sg & 31);
                    }
                }
            }
        }
        const bool heavy = reached > kHeavy;
        any = reached > 0 && !heavy;
        __syncwarp();
        if (heavy)
            for (int i = lane; i < A.nzw; i += 32) nz[w * A.nzw + i] = 0u;
        if (lane == 0) {
            sheavy[w] = heavy;
            if (heavy) A.heavy[atomicAdd(A.nheavy, 1)] = p;
        }
    }
    const bool work = __syncthreads_or(any);

    if (work) {
        unsigned *q = sq[w];
        int *tag = stag[w];
        T *xs = sx[w], *ws = sw[w];
        int *ns = sn[w];
        int qn = 0, cur = -1, curc = 0, ia, ib;
        unsigned mine = 0, npair = 0;
        T acc = T(0);
        feature_cols(lane, ia, ib);
        auto flush = [&]() {
            if (cur < 0) return;
            if (lane < 28) {
                double *d = sacc + (w * C + curc) * 28 + lane;
                *d = (mine >> curc & 1u) ? *d + (double)acc : (double)acc;
            }
            mine |= 1u << curc;
            acc = T(0);
        };
        auto add = [&](int e, int t, int c) {
            if (t != cur) {
                flush();
                cur = t;
                curc = c;
            }
            acc = add_pair(V, acc, ws, ns, xs, e, ia, ib, lane);
        };
        auto weigh_at = [&](unsigned e) {
            weigh<T>(V, A.lse, srec + (e >> 24) * 28, (int)(e & 0xffffffu), ws + lane * (kF64 ? 1 : 7), ns + lane, xs + lane * 7);
        };
        auto evaluate = [&](int cnt) {
            __syncwarp();
            if (lane < cnt) weigh_at(q[lane]);
            __syncwarp();
            if (cnt == 32 && tag[0] == cur && tag[31] == cur) {   // one sum for all (tags come in runs)
#pragma unroll 8
                for (int e = 0; e < 32; e++) acc = add_pair(V, acc, ws, ns, xs, e, ia, ib, lane);
            } else {
                for (int e = 0; e < cnt; e++) add(e, tag[e], (int)(q[e] >> 24));
            }
            npair += cnt;
            __syncwarp();
        };
        // the warp's groups in order: component c, group g, points [na, nb), tag
        int cc = -1, c = 0, g = 0, j = 0, na = 0, nb = V.N, tg = 0, si = 0;
        unsigned nzb = 0u, bits = 0u;
        auto next_group = [&]() -> bool {
            for (;;) {
                if (bits) {
                    g = si * 32 + __ffs(bits) - 1;
                    bits &= bits - 1;
                    return true;
                }
                if constexpr (kF64) {
                    if (nzb) {
                        si = (si & ~31) + __ffs(nzb) - 1;
                        nzb &= nzb - 1;
                        bits = mask[c * A.nw + si] & (0x01010101u << w);
                        continue;
                    }
                    si = cc < 0 ? 0 : (si & ~31) + 32;   // the next word of nz, or the next component
                    if (cc < 0 || si >= A.nw) {
                        if (++cc >= C) return false;
                        c = (cc + w) % C;
                        tg = c;
                        si = 0;
                    }
                    nzb = nz[c * A.nzw + (si >> 5)];
                } else {
                    // splits (w + c) mod W, + W, ... of each component
                    const int s1 = cc < 0 || j >= A.nsplit ? -1 : (nb - 1) >> 10;
                    if (++si > s1 || cc < 0) {
                        if (cc >= 0) j += W;
                        while (cc < 0 || j >= A.nsplit) {
                            if (++cc >= C) return false;
                            c = (cc + w) % C;
                            j = (w + c) % W;
                        }
                        na = j * A.nps;
                        nb = (int)min((long long)V.N, (long long)(j + 1) * A.nps);
                        tg = c * A.nsplit + j;
                        si = na >> 10;
                    }
                    if (!(nz[c * A.nzw + (si >> 5)] >> (si & 31) & 1u)) continue;
                    bits = mask[c * A.nw + si];
                    if (si == na >> 10) bits &= kFull << ((na >> 5) & 31);
                    if (si == (nb - 1) >> 10) bits &= kFull >> (31 - (((nb - 1) >> 5) & 31));
                }
            }
        };
        float xn[6], tn = 0.f, x2n = 0.f;
        auto fetch = [&]() {
            const int n = g * 32 + lane;
#pragma unroll
            for (int i = 0; i < 6; i++) xn[i] = V.xf[(size_t)i * V.Np + n];
            tn = V.thr[n];
            x2n = V.gx2[g];
        };
        bool more = next_group();
        if (more) fetch();
        while (more) {
            float x[6];
#pragma unroll
            for (int i = 0; i < 6; i++) x[i] = xn[i];
            const float t = tn, ch = fmaf(sb[c], x2n, schi[c]);
            const int n = g * 32 + lane, cv = c, tv = tg;
            const bool in = n >= na && n < nb;
            more = next_group();
            if (more) fetch();
            const float *r = srec32 + cv * 28;
            float qd = quad_pos(r, x);
            if (!__any_sync(kFull, in && !(ch - kQuadLo * qd < t))) continue;
            qd = quad_rest(r, x, qd);
            const bool surv = in && !(ch - kQuadLo * qd < t);
            const unsigned ms = __ballot_sync(kFull, surv);
            if (!ms) continue;
            if (surv) {
                const int at = qn + __popc(ms & ((1u << lane) - 1u));
                q[at] = ((unsigned)cv << 24) | (unsigned)n;
                tag[at] = tv;
            }
            qn += __popc(ms);
            if (qn >= 32) {
                evaluate(32);
                qn -= 32;
                const unsigned tq = q[32 + lane];
                const int tt = tag[32 + lane];
                __syncwarp();
                if (lane < qn) { q[lane] = tq; tag[lane] = tt; }
            }
        }
        // the rest of the lists
        if constexpr (kF64) {
            if (lane == 0) scount[w] = qn;
            __syncthreads();
            int total = 0;
            for (int i = 0; i < W; i++) total += scount[i];
            for (int b = w * 32; b < total; b += W * 32) {
                const int cnt = min(32, total - b);
                int at = b + min(lane, cnt - 1), i = 0;
                while (at >= scount[i]) at -= scount[i++];
                const unsigned e = sq[i][at];
                __syncwarp();
                if (lane < cnt) weigh_at(e);
                __syncwarp();
                for (int k = 0; k < cnt; k++) {
                    const int ce = (int)(__shfl_sync(kFull, e, k) >> 24);
                    add(k, ce, ce);
                }
                npair += cnt;
            }
        } else {
            if (qn) evaluate(qn);
        }
        flush();
        if (lane == 0) used[w] = mine;
        if (A.pairs && lane == 0 && npair) atomicAdd(A.pairs, (unsigned long long)npair);
        __syncthreads();
    }

    // ---- sums of the warps ----
    const int p = p0 + w;
    if (p >= V.K || sheavy[w]) return;
    double s = 0.0;
    bool first = true;
    for (int i = 0; i < W; i++)
        if (used[i] >> w & 1u) {
            const double v = lane < 28 ? sacc[(i * C + w) * 28 + lane] : 0.0;
            s = first ? v : s + v;
            first = false;
        }
    write_row(V, A, p, s, !first, srec32 + w * 28, lane);
}

template <typename T>
__global__ void __launch_bounds__(kOneWarps * 32, 8) k_sp_pass2_one(SpView V, P2Args A)
{
    pdl_wait();
    constexpr bool kF64 = sizeof(T) == 8;
    constexpr int W = kOneWarps, kList2 = 64;
    __shared__ double sacc[W * 28], ssum[2][28];
    __shared__ T srec[28];
    __shared__ float srec32[28];
    __shared__ T sx[W][32 * 7], sw[W][32 * (kF64 ? 1 : 7)];
    __shared__ int sq[W][kList2], stag[W][kList2], sn[W][32], scount[W];
    cg::cluster_group cluster = cg::this_cluster();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = (int)cluster.block_rank();
    const int nblk = (int)cluster.num_blocks(), rw = rank * W + w, nw = nblk * W, ncl = gridDim.x / nblk;
    const int todo = A.heavy ? *A.nheavy : V.K;
    int ia, ib;
    feature_cols(lane, ia, ib);
    // A block goes on to the cluster's next component as soon as its own sums
    // are out; it waits for the others only before it writes the sums after
    // those (two buffers), the first block's warp 0 before it adds them.
    int buf = 0;
    bool pending = false;
    for (int e = blockIdx.x / nblk; e < todo; e += ncl, buf ^= 1) {
        const int p = A.heavy ? A.heavy[e] : e;
        if (threadIdx.x < 28) {
            srec32[threadIdx.x] = V.rec32[(size_t)p * VBGS_REC + threadIdx.x];
            srec[threadIdx.x] = kF64 ? (T)V.rec[(size_t)p * VBGS_REC + threadIdx.x] : (T)srec32[threadIdx.x];
        }
        float m[6];
#pragma unroll
        for (int i = 0; i < 6; i++) m[i] = V.cb[(size_t)i * V.Kp + p];
        const float chi = V.cb[(size_t)6 * V.Kp + p], lp = V.cb[(size_t)7 * V.Kp + p], lc = V.cb[(size_t)8 * V.Kp + p],
                    la = V.cb[(size_t)9 * V.Kp + p], B = V.cb[(size_t)10 * V.Kp + p];
        __syncthreads();
        int *q = sq[w], *tag = stag[w], *ns = sn[w];
        T *xs = sx[w], *ws = sw[w];
        T acc = T(0);
        double total = 0.0;
        auto weigh_at = [&](int n) { weigh<T>(V, A.lse, srec, n, ws + lane * (kF64 ? 1 : 7), ns + lane, xs + lane * 7); };
        int qn = 0, cur = -1;
        unsigned npair = 0;
        auto flush = [&]() {
            if (cur >= 0) total += (double)acc;
            acc = T(0);
        };
        auto evaluate = [&](int cnt) {
            __syncwarp();
            if (lane < cnt) weigh_at(q[lane]);
            __syncwarp();
            if (cnt == 32 && (kF64 || (tag[0] == cur && tag[31] == cur))) {
#pragma unroll 8
                for (int i = 0; i < 32; i++) acc = add_pair(V, acc, ws, ns, xs, i, ia, ib, lane);
            } else {
                for (int i = 0; i < cnt; i++) {
                    if (!kF64 && tag[i] != cur) {
                        flush();
                        cur = tag[i];
                    }
                    acc = add_pair(V, acc, ws, ns, xs, i, ia, ib, lane);
                }
            }
            npair += cnt;
            __syncwarp();
        };
        // lanes test 32 groups g(lane); the pairs of those that reach their
        // threshold, points [na, nb), go to the list
        auto visit = [&](int gl, bool on, int na, int nb, int tg) {
            const int gc = min(gl, V.G - 1);
            float lo[6], hi[6];
#pragma unroll
            for (int i = 0; i < 6; i++) {
                lo[i] = V.gbox[(size_t)i * V.G + gc];
                hi[i] = V.gbox[(size_t)(6 + i) * V.G + gc];
            }
            const float xl = V.gx2[gc];
            unsigned bits = __ballot_sync(kFull, on && !(box_bound(lo, hi, m, m, fmaf(B, xl, chi), lp, lc, la) < V.gthr[gc]));
            if (!bits) return;
            float xn[6], tn, x2n;
            int g;
            auto fetch = [&]() {
                const int b = __ffs(bits) - 1;
                bits &= bits - 1;
                g = __shfl_sync(kFull, gl, b);
                x2n = __shfl_sync(kFull, xl, b);
                const int n = g * 32 + lane;
#pragma unroll
                for (int i = 0; i < 6; i++) xn[i] = V.xf[(size_t)i * V.Np + n];
                tn = V.thr[n];
            };
            fetch();
            for (bool more = true; more;) {
                float x[6];
#pragma unroll
                for (int i = 0; i < 6; i++) x[i] = xn[i];
                const float t = tn, ch = fmaf(B, x2n, chi);
                const int n = g * 32 + lane;
                const bool in = n >= na && n < nb;
                more = bits != 0u;
                if (more) fetch();
                float qd = quad_pos(srec32, x);
                if (!__any_sync(kFull, in && !(ch - kQuadLo * qd < t))) continue;
                qd = quad_rest(srec32, x, qd);
                const bool surv = in && !(ch - kQuadLo * qd < t);
                const unsigned ms = __ballot_sync(kFull, surv);
                if (!ms) continue;
                if (surv) {
                    const int at = qn + __popc(ms & ((1u << lane) - 1u));
                    q[at] = n;
                    tag[at] = tg;
                }
                qn += __popc(ms);
                if (qn >= 32) {
                    evaluate(32);
                    qn -= 32;
                    const int tq = q[32 + lane], tt = tag[32 + lane];
                    __syncwarp();
                    if (lane < qn) { q[lane] = tq; tag[lane] = tt; }
                }
            }
        };
        if constexpr (kF64) {
            cur = 0;
            for (int g0 = rw; g0 < V.G; g0 += 32 * nw) {
                const int gl = g0 + lane * nw;
                visit(gl, gl < V.G, 0, V.N, 0);
            }
            // the rest of the block's lists
            if (lane == 0) scount[w] = qn;
            __syncthreads();
            int rest = 0;
            for (int i = 0; i < W; i++) rest += scount[i];
            for (int b = w * 32; b < rest; b += W * 32) {
                const int cnt = min(32, rest - b);
                int at = b + min(lane, cnt - 1), i = 0;
                while (at >= scount[i]) at -= scount[i++];
                const int n = sq[i][at];
                __syncwarp();
                if (lane < cnt) weigh_at(n);
                __syncwarp();
#pragma unroll 4
                for (int k = 0; k < cnt; k++) acc = add_pair(V, acc, ws, ns, xs, k, ia, ib, lane);
                npair += cnt;
            }
            total = (double)acc;
        } else {
            for (int j = rw; j < A.nsplit; j += nw) {
                const int na = j * A.nps, nb = (int)min((long long)V.N, (long long)(j + 1) * A.nps);
                for (int g0 = na >> 5; g0 * 32 < nb; g0 += 32) visit(g0 + lane, (g0 + lane) * 32 < nb, na, nb, j);
            }
            if (qn) evaluate(qn);
            flush();
        }
        if (A.pairs && lane == 0 && npair) atomicAdd(A.pairs, (unsigned long long)npair);
        if (lane < 28) sacc[w * 28 + lane] = total;
        __syncthreads();
        if (pending) cluster.barrier_wait();
        if (threadIdx.x < 28) {
            double t = sacc[threadIdx.x];
            for (int i = 1; i < W; i++) t += sacc[i * 28 + threadIdx.x];
            ssum[buf][threadIdx.x] = t;
        }
        cluster.barrier_arrive();
        pending = rank != 0 || w != 0;
        if (!pending) {
            cluster.barrier_wait();
            double t = 0.0;
            if (lane < 28)
                for (int i = 0; i < nblk; i++) t += cluster.map_shared_rank(ssum[buf], i)[lane];
            write_row(V, A, p, t, true, srec32, lane);
        }
    }
    if (pending) cluster.barrier_wait();
    cluster.sync();   // the last sums are read before their blocks leave
}

inline size_t even(size_t v) { return (v + 3) & ~size_t(3); }

} // namespace

// phi: with the FP64 form's feature table (kMaxFeatures points at most).
size_t sparse_scratch_floats(int64_t N, int K, bool phi)
{
    const size_t Np = (size_t)((N + 31) / 32) * 32, G = Np / 32, S = (G + 31) / 32;
    const size_t Kp = (size_t)((K + 31) / 32) * 32, Kg = Kp / 32;
    return even(9 * Np) + even(14 * G) + even(14 * S) + even(11 * Kp) + even(17 * Kg) + even(Kp + 4) +
           (phi ? 56 * (size_t)N : 0);
}
bool sparse_phi(int64_t N, int precision) { return precision == VBGS_FP64 && N <= kMaxFeatures; }

bool sparse_fits(int64_t N, int K) { return N > 0 && N <= kMaxPoints && K <= kMaxComps; }

int sparse_set_attributes()
{
    static const bool ok = [] {
        const int s64 = (int)(kP1Warps * p1_warp_bytes(true)), s32 = (int)(kP1Warps * p1_warp_bytes(false) + kMaxComps / 8);
        return cudaFuncSetAttribute(k_sp_pass1<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, s64) == cudaSuccess &&
               cudaFuncSetAttribute(k_sp_pass1<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, s32) == cudaSuccess;
    }();
    return ok ? 0 : -1;
}

int launch_estep_sparse(const EstepBuffers &B, int precision, bool want_stats, int kps, int p1_splits, int64_t nps,
                        int p2_splits, int num_sms, unsigned int *done, cudaStream_t st, Prof *pf)
{
    const bool f64 = precision == VBGS_FP64;
    SpView V;
    V.X = B.X;
    V.N = (int)B.N;
    V.G = (V.N + 31) / 32;
    V.Np = V.G * 32;
    V.S = (V.G + 31) / 32;
    V.K = B.K;
    V.Kg = (V.K + 31) / 32;
    V.Kp = V.Kg * 32;
    float *f = B.sparse;
    V.xf = f;
    V.thr = f + (size_t)6 * V.Np;
    V.lse2f = V.thr + V.Np;
    V.best = reinterpret_cast<int *>(V.lse2f + V.Np);
    f += even((size_t)9 * V.Np);
    V.gbox = f;
    V.gx2 = f + (size_t)12 * V.G;
    V.gthr = V.gx2 + V.G;
    f += even((size_t)14 * V.G);
    V.sbox = f;
    V.sx2 = f + (size_t)12 * V.S;
    V.sthr = reinterpret_cast<int *>(V.sx2 + V.S);
    f += even((size_t)14 * V.S);
    V.cb = f;
    V.cg = f + even((size_t)11 * V.Kp);
    V.heavy = reinterpret_cast<int *>(V.cg + even((size_t)17 * V.Kg));
    V.nheavy = V.heavy + V.Kp;
    V.phi = B.sparse_phi ? reinterpret_cast<double *>(V.heavy + even((size_t)V.Kp + 4)) : nullptr;
    V.rec = B.rec;
    V.rec32 = B.rec32;
    V.t2 = (float)((std::log((double)std::max(V.K, 1)) + 37.0) * 1.4426950408889634) + 1e-3f;

    int launches = 3;
    pf->begin(VBGS_PROF_PLAN, st);
    launch_pdl(k_sp_comps, (V.Kg + 3) / 4, 128, 0, st, V);
    pf->end(st);
    if (!B.same_points) {
        pf->begin(VBGS_PROF_PLAN, st);
        launch_pdl(k_sp_points, V.S, 1024, 0, st, V);
        pf->end(st);
        launches++;
        if (V.phi && want_stats) {
            pf->begin(VBGS_PROF_PLAN, st);
            launch_pdl(k_sp_features, (unsigned)(((int64_t)V.N * 28 + 255) / 256), 256, 0, st, V);
            pf->end(st);
            launches++;
        }
    }
    // FP64: four warps a block, and a cluster per point group until the grid
    // holds five blocks an SM: fewer leave the FP64 pipe idle in the tail, more
    // cut the lists into partly filled batches (clusters of 1 / 2 / 4 / 8, us a
    // launch: 313 groups 96 / 94 / 84 / 102, 386 groups 173 / 147 / 154 / 183,
    // 254 groups of the room 107 / 76 / 64 / 86).  FP32: one block per group, with warps enough
    // for about four a sub-partition (more would cut the grid into two waves).
    // Component groups are cut into units until every warp has a few.
    int W = 4, cl = 1;
    if (f64)
        while (cl < kCluster && V.G * cl < 5 * num_sms && 8 * cl <= 4 * V.Kg) cl *= 2;
    else
        while (W < kP1Warps && (int64_t)V.G * W < 4 * (int64_t)num_sms * 4 && 2 * W <= 4 * V.Kg) W *= 2;
    int nsub = 1;
    while (nsub < 4 && V.Kg * nsub < 4 * W * cl) nsub *= 2;
    if (!B.same_points) {
        int sub = 1;
        while (sub < 4 && V.Kg * sub < 4 * kSeedWarps) sub *= 2;
        pf->begin(VBGS_PROF_PLAN, st);
        launch_pdl(k_sp_seed, V.G, kSeedWarps * 32, 0, st, V, sub);
        pf->end(st);
        launches++;
    }
    const size_t sh1 = (size_t)W * p1_warp_bytes(f64) + (f64 ? 0 : (size_t)V.Kg * 4);
    P1Args a1{nsub, kps, p1_splits, reinterpret_cast<double2 *>(B.part), B.lse, B.lse_part,
              B.lse_part ? B.scal + SC_SUM_LSE : nullptr, done, pf->on ? pf->d_pairs + 1 : nullptr};
    if (sparse_set_attributes()) return -1;
    pf->begin(VBGS_PROF_PASS1, st);
    if (f64) launch_pdl_cluster(k_sp_pass1<double>, V.G * cl, W * 32, cl, sh1, st, V, a1);
    else     launch_pdl(k_sp_pass1<float>, V.G, W * 32, sh1, st, V, a1);
    pf->end(st);
    if (!want_stats) return cudaGetLastError() == cudaSuccess ? launches - 1 : -1;

    // Eight components a block while that still gives two blocks an SM (and
    // the masks of all points fit); fewer components take a cluster each.
    P2Args a2{};
    a2.nps = (int)nps;
    a2.nsplit = p2_splits;
    a2.nw = V.S;
    a2.nzw = (V.S + 31) / 32;
    a2.lse = B.lse;
    a2.anchored = !f64;
    a2.kperm = B.kperm;
    a2.dS = B.dS;
    a2.pairs = pf->on ? pf->d_pairs : nullptr;
    const bool wide = (V.K + 7) / 8 >= 2 * num_sms && V.S <= kMaxSupers;
    if (wide) {
        pf->begin(VBGS_PROF_PASS2, st);
        a2.heavy = V.heavy;
        a2.nheavy = V.nheavy;
        const size_t sh2 = (size_t)(a2.nw + a2.nzw) * 4 * kP2Warps;
        if (f64) launch_pdl(k_sp_pass2<double>, (V.K + 7) / 8, kP2Warps * 32, sh2, st, V, a2);
        else     launch_pdl(k_sp_pass2<float>, (V.K + 7) / 8, kP2Warps * 32, sh2, st, V, a2);
        pf->end(st);
        launches++;
    }
    pf->begin(VBGS_PROF_PASS2, st);
    // A round of blocks (eight resident an SM), whose clusters take turns.
    // FP64: clusters of eight while there are few components, smaller ones as
    // soon as they would need over four rounds, since a block evaluates its
    // lists in batches of 32 pairs and small shares leave the batches part
    // filled (clusters of 1 / 2 / 4 / 8, us a launch: K = 64 45 / 28 / 21 / 20,
    // K = 1,000 129 / 103 / 98 / 124, K = 1,777 196 / 169 / 199 / 279); the
    // heavy components of a wide map take four (2 / 4 / 8: 36 / 30 / 37).
    // FP32: a warp per split is all a component can use, with a few pairs each,
    // so clusters of two from 300 components on (1 / 2 / 4 / 8: K = 300 57 / 36 /
    // 39 / 41, K = 700 51 / 45 / 47 / 57, K = 1,500 55 / 49 / 67 / 101, K = 2,200
    // 56 / 58 / 79 / 138); the heavy components of a wide map are enough to fill
    // the chip alone (132 / 145 / 195 / 299).
    cl = kCluster;
    auto crowded = [&]() {
        if (wide) return f64 ? cl > 4 : true;
        return (int64_t)V.K * cl > (f64 || cl <= 2 ? 32 : 4) * num_sms || (!f64 && cl / 2 * kOneWarps >= p2_splits);
    };
    while (cl > 1 && crowded()) cl /= 2;
    const int clusters = std::max(1, std::min(8 * num_sms / cl, V.K));
    if (f64) launch_pdl_cluster(k_sp_pass2_one<double>, clusters * cl, kOneWarps * 32, cl, 0, st, V, a2);
    else     launch_pdl_cluster(k_sp_pass2_one<float>, clusters * cl, kOneWarps * 32, cl, 0, st, V, a2);
    pf->end(st);
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

} // namespace vbgs

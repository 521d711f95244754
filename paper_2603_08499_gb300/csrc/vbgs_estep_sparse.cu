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
//   FP64, 10,000 points, K = 1,000 (mixture):  1,226 + 2,105 -> 107 + 172
//   FP64, 8,294 points, K = 50,000 (room):    44,100 + 8,650 -> 178 + 200
//   FP32, 36,000 points, K = 50,000 (room):    3,472 +   982 -> 797 + 310
#include "vbgs_internal.cuh"
#include "vbgs_pair.cuh"
#include <algorithm>
#include <cmath>

namespace vbgs {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxPoints = 1 << 22;   // pass 2's group masks stay within 16 KB of shared memory
constexpr int kP2Warps = 8;
constexpr float kLog2e = 1.4426950408889634f;

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
    int N, Np, G, S;
    float *xf;             // 6 x Np: the points in FP32
    float *gbox, *gx2;     // 12 x G boxes (lo, hi), G largest |x|^2
    float *sbox, *sx2;     // 12 x S, S: the same over 32 groups
    float *thr, *gthr;     // Np, G: lse - t (log2 units), its minimum over a group
    int *sthr;             // S: its minimum over a super group (ordered integer)
    float *lse2f;          // Np: lse in log2 units (FP32 form)
    int K, Kp, Kg;
    float *cb;             // 11 x Kp: m (6), c + slack, lp, lc, la, slack per |x|^2
    float *cg;             // 17 x Kg: lo (6), hi (6), then max, min, min, min, max of the last five
    const double *rec;
    const float *rec32;
    float t2;              // t in log2 units
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

// A record row (28 of 32 floats), the same address in every lane.
__device__ __forceinline__ void load_rec(const float *__restrict__ rec32, int k, float r[28])
{
    const float4 *p = reinterpret_cast<const float4 *>(rec32 + (size_t)k * VBGS_REC);
#pragma unroll
    for (int i = 0; i < 7; i++) {
        const float4 v = p[i];
        r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
    }
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

// Bound terms of every component and of every 32 (a warp each); also resets
// the super groups' threshold minima for the pass that follows.
__global__ void __launch_bounds__(128) k_sp_comps(SpView V)
{
    pdl_wait();
    const int lane = threadIdx.x & 31, q = blockIdx.x * 4 + (threadIdx.x >> 5);
    for (int s = blockIdx.x * 128 + threadIdx.x; s < V.S; s += gridDim.x * 128) V.sthr[s] = 0x7fffffff;
    if (q >= V.Kg) return;
    const int k = q * 32 + lane;
    const bool valid = k < V.K;
    const float *r = V.rec32 + (size_t)min(k, V.K - 1) * VBGS_REC;
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

// Pass 1: lse_n.  A block per 32 points (one per lane of every warp); its
// warps share the components.
//   seed: every warp takes the component group with the largest bound among
//     its own and scores its 32 components; the best of them over the block is
//     a point's seed, whose logit gives the point's threshold lse - t.
//   FP64: each warp walks its groups (interleaved over the warps); a pair
//     whose FP32 bound reaches the threshold goes to the warp's queue, and 32
//     queued pairs are evaluated at once: sum_k exp(l_k - ref) with ref the
//     seed's FP64 logit.  A term above e^64 (a poor seed) first moves the
//     reference.  Terms of one point are added in queue order.
//   FP32: each warp walks whole K splits of the dense pass (kps components),
//     lanes keep their online (max, sum); the partials are merged in FP64.
struct P1Args {
    int kps, nsplit;       // FP32
    double2 *part;         // FP32: nsplit x N
    double *lse, *lse_part, *sum_out;
    unsigned int *done;
    unsigned long long *pairs;
};

template <typename T>
__global__ void __launch_bounds__(512) k_sp_pass1(SpView V, P1Args A)
{
    pdl_wait();
    constexpr bool kF64 = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double sx[32 * 6];
    __shared__ bool last;
    const int W = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = blockIdx.x;
    double *sref = reinterpret_cast<double *>(smem_raw), *ssum = sref + W * 32;
    float *sm = reinterpret_cast<float *>(ssum + W * 32);
    int *sk = reinterpret_cast<int *>(sm + W * 32);
    int *qk = sk + W * 32 + w * 128, *qp = qk + 64;
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
    if (kF64 && threadIdx.x < 192)
        sx[threadIdx.x] = V.X[(size_t)min(g * 32 + (int)threadIdx.x / 6, V.N - 1) * VBGS_XS + threadIdx.x % 6];
    if (kF64 && blockDim.x < 192)
        for (int i = threadIdx.x + blockDim.x; i < 192; i += blockDim.x)
            sx[i] = V.X[(size_t)min(g * 32 + i / 6, V.N - 1) * VBGS_XS + i % 6];

    // ---- seed ----
    float ub = -INFINITY;
    int bg = 0x7fffffff;
    for (int q = lane * W + w; q < V.Kg; q += 32 * W) {
        const float u = group_bound(V, q, lo, hi, x2);
        if (u > ub || bg == 0x7fffffff) { ub = u; bg = q; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ou = __shfl_xor_sync(kFull, ub, o);
        const int og = __shfl_xor_sync(kFull, bg, o);
        if (og != 0x7fffffff && (bg == 0x7fffffff || ou > ub || (ou == ub && og < bg))) { ub = ou; bg = og; }
    }
    float mx = -INFINITY;
    int km = -1;
    if (bg != 0x7fffffff) {
        const int k1 = min(V.K, bg * 32 + 32);
        for (int k = bg * 32; k < k1; k++) {
            float r[28];
            load_rec(V.rec32, k, r);
            const float l = logit<float>(r, x);
            if (l > mx || km < 0) { mx = l; km = k; }
        }
    }
    sm[w * 32 + lane] = mx;
    sk[w * 32 + lane] = km;
    __syncthreads();
    for (int i = 0; i < W; i++) {
        const float v = sm[i * 32 + lane];
        const int k = sk[i * 32 + lane];
        if (k >= 0 && (km < 0 || v > mx || (v == mx && k < km))) { mx = v; km = k; }
    }
    float thr;
    if (kF64) {
        if (w == 0) {
            double x6[6];
#pragma unroll
            for (int i = 0; i < 6; i++) x6[i] = sx[lane * 6 + i];
            const double l = logit<double>(V.rec + (size_t)km * VBGS_REC, x6);
            for (int i = 0; i < W; i++) { sref[i * 32 + lane] = l; ssum[i * 32 + lane] = 0.0; }
        }
        __syncthreads();
        const float l2 = (float)(sref[w * 32 + lane] * 1.4426950408889634);
        thr = l2 - fabsf(l2) * 2.5e-7f - V.t2;
    } else {
        thr = mx - V.t2;
    }
    if (!valid) thr = INFINITY;
    float bthr = warp_min(thr);
    unsigned npair = 0;

    // The pair tests of component k against the lanes' points; true in the
    // lanes whose pair reaches its threshold (r holds the record after it).
    auto screen = [&](int k, float r[28], float &q) -> bool {
        load_rec(V.rec32, k, r);
        const float c = fmaf(V.cb[(size_t)10 * V.Kp + k], x2, V.cb[(size_t)6 * V.Kp + k]);
        q = quad_pos(r, x);
        if (!__any_sync(kFull, valid && !(c - kQuadLo * q < thr))) return false;
        q = quad_rest(r, x, q);
        return valid && !(c - kQuadLo * q < thr);
    };

    if constexpr (kF64) {
        double *ref = sref + w * 32, *sum = ssum + w * 32;
        int qn = 0;
        auto evaluate = [&](int cnt) {
            __syncwarp();
            const bool act = lane < cnt;
            const int k = qk[act ? lane : 0], p = qp[act ? lane : 0];
            double x6[6], r[28];
#pragma unroll
            for (int i = 0; i < 6; i++) x6[i] = sx[p * 6 + i];
            const double2 *rp = reinterpret_cast<const double2 *>(V.rec + (size_t)k * VBGS_REC);
#pragma unroll
            for (int i = 0; i < 14; i++) { const double2 v = rp[i]; r[2 * i] = v.x; r[2 * i + 1] = v.y; }
            const double l = logit<double>(r, x6);
            double rf = ref[p];
            if (__any_sync(kFull, act && l > rf + 64.0)) {
                for (int e = 0; e < cnt; e++) {
                    const double le = __shfl_sync(kFull, l, e);
                    const int pe = __shfl_sync(kFull, p, e);
                    const double re = ref[pe];
                    __syncwarp();
                    if (lane == 0 && le > re + 64.0) { sum[pe] *= exp(re - le); ref[pe] = le; }
                    __syncwarp();
                }
                rf = ref[p];
            }
            const double v = exp(l - rf);
            // add the terms point by point, in queue order
            const unsigned peers = __match_any_sync(kFull, act ? p : 32 + lane);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            const int ranks = __reduce_max_sync(kFull, act ? rank : 0);
            for (int i = 0; i <= ranks; i++) {
                if (act && rank == i) sum[p] += v;
                __syncwarp();
            }
            npair += cnt;
        };
        for (int q0 = 0; q0 < V.Kg; q0 += 32 * W) {
            const int q = q0 + lane * W + w;
            unsigned m1 = __ballot_sync(kFull, q < V.Kg && !(group_bound(V, min(q, V.Kg - 1), lo, hi, x2) < bthr));
            while (m1) {
                const int b = __ffs(m1) - 1;
                m1 &= m1 - 1;
                const int k0 = (q0 + b * W + w) * 32, k = k0 + lane;
                unsigned m2 = __ballot_sync(kFull, k < V.K && !(comp_bound(V, min(k, V.K - 1), lo, hi, x2) < bthr));
                while (m2) {
                    const int kk = k0 + __ffs(m2) - 1;
                    m2 &= m2 - 1;
                    float r[28], qd;
                    const bool surv = screen(kk, r, qd);
                    const unsigned ms = __ballot_sync(kFull, surv);
                    if (!ms) continue;
                    if (surv) {
                        const int at = qn + __popc(ms & ((1u << lane) - 1u));
                        qk[at] = kk;
                        qp[at] = lane;
                        // a certified lower bound of the pair's logit raises the point's threshold
                        const float sl = V.cb[(size_t)6 * V.Kp + kk] - r[27];
                        thr = fmaxf(thr, r[27] - sl - V.cb[(size_t)10 * V.Kp + kk] * x2 - kQuadHi * qd - V.t2);
                    }
                    qn += __popc(ms);
                    if (qn >= 32) {
                        evaluate(32);
                        qn -= 32;
                        const int tk = qk[32 + lane], tp = qp[32 + lane];
                        __syncwarp();
                        if (lane < qn) { qk[lane] = tk; qp[lane] = tp; }
                    }
                }
                bthr = warp_min(thr);
            }
        }
        if (qn) evaluate(qn);
    } else {
        for (int s = w; s < A.nsplit; s += W) {
            const int k0 = s * A.kps, k1 = min(V.K, k0 + A.kps);
            float m = -INFINITY, sum = 0.f;
            for (int q0 = k0 >> 5; q0 * 32 < k1; q0 += 32) {
                const int q = q0 + lane;
                unsigned m1 = __ballot_sync(kFull, q * 32 < k1 && !(group_bound(V, min(q, V.Kg - 1), lo, hi, x2) < bthr));
                while (m1) {
                    const int kb = (q0 + __ffs(m1) - 1) * 32, k = kb + lane;
                    m1 &= m1 - 1;
                    unsigned m2 = __ballot_sync(kFull, k >= k0 && k < k1 &&
                                                           !(comp_bound(V, min(k, V.K - 1), lo, hi, x2) < bthr));
                    while (m2) {
                        const int kk = kb + __ffs(m2) - 1;
                        m2 &= m2 - 1;
                        float r[28], qd;
                        if (!__any_sync(kFull, screen(kk, r, qd))) continue;
                        npair += 32;
                        const float l = fmaf(-0.5f, qd, r[27]);
                        if (l > m) {
                            sum = fmaf(sum, ex2_approx(m - l), 1.f);
                            m = l;
                        } else {
                            sum += ex2_approx(l - m);
                        }
                    }
                    if (valid) thr = fmaxf(thr, m - V.t2);
                    bthr = warp_min(thr);
                }
            }
            if (valid) {
                double2 o = make_double2(-INFINITY, 0.0);
                if (!(sum == 0.f)) o = make_double2((double)m / (double)Arith<float>::lse_scale(), (double)sum);
                A.part[(size_t)s * V.N + n] = o;
            }
        }
    }
    __syncthreads();

    // ---- merge ----
    if (w == 0) {
        double R = -INFINITY, s = 0.0, v = 0.0;
        if constexpr (kF64) {
            for (int i = 0; i < W; i++) R = fmax(R, sref[i * 32 + lane]);
            for (int i = 0; i < W; i++) {
                const double f = sref[i * 32 + lane], t = ssum[i * 32 + lane];
                s += f == R ? t : t * exp(f - R);
            }
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
    if (!A.sum_out) return;
    // the block sums, added in block order by the last block to finish
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(A.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t += __ldcg(A.lse_part + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(kFull, t, o);
    if (lane == 0) ssum[w] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int i = 0; i < W; i++) tot += ssum[i];
        *A.sum_out = tot;
        *A.done = 0u;
    }
}

// Pass 2: Delta S.  A block takes C neighbouring components (8, or 1 when
// there are few) and a slice of the points.
//   1. its warps find the point groups whose box bound reaches their threshold
//      (super groups first), as bit masks per component;
//   2. every warp walks its share of those groups (FP64: the set bits round
//      robin, so that a heavy component is spread over the block; FP32: whole
//      N splits of the dense pass, whose sums are FP32), queues the pairs that
//      survive the FP32 test, and evaluates 32 of them at once: r = exp(l - lse)
//      one pair per lane, then the statistics with one feature per lane, pair
//      after pair;
//   3. the warps' FP64 sums are added in warp order.
// The sums of a component never leave the block (slices: one partial each).
struct P2Args {
    int slices;
    int gper;              // FP64: groups per slice
    int nps, nsplit, spy;  // FP32: points per split, splits, splits per slice
    int nw;                // mask words per component
    const double *lse;
    const float *anchor;   // rec32 (FP32 form: moments about the record's mean), else null
    const int *kperm;
    double *dS, *part;     // slices > 1: part[(slice * K + p) * 28 + f]
    unsigned long long *pairs;
};

template <typename T, int C>
__global__ void __launch_bounds__(kP2Warps * 32) k_sp_pass2(SpView V, P2Args A)
{
    pdl_wait();
    constexpr bool kF64 = sizeof(T) == 8;
    constexpr int W = kP2Warps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double sacc[W * C * 28];
    __shared__ T srec[C * 28];
    __shared__ T sx[W][32 * 8], sw[W][32];
    __shared__ unsigned sq[W][64];
    __shared__ int stag[W][64];
    __shared__ unsigned used[W];     // bit c: warp w holds a sum of component c
    unsigned *mask = reinterpret_cast<unsigned *>(smem_raw);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, p0 = blockIdx.x * C, y = blockIdx.y;
    int n0 = 0, n1 = V.N, j0 = 0, j1 = 0, ga, gb;
    if (kF64) {
        ga = y * A.gper;
        gb = min(V.G, ga + A.gper);
    } else {
        j0 = y * A.spy;
        j1 = min(A.nsplit, j0 + A.spy);
        n0 = j0 * A.nps;
        n1 = min((long long)V.N, (long long)j1 * A.nps);
        ga = n0 >> 5;
        gb = (n1 + 31) >> 5;
    }
    const int sa = ga >> 5, sb = (gb + 31) >> 5;
    for (int i = threadIdx.x; i < C * A.nw; i += W * 32) mask[i] = 0u;
    for (int i = threadIdx.x; i < C * 28; i += W * 32) {
        const int p = min(p0 + i / 28, V.K - 1);
        srec[i] = kF64 ? (T)V.rec[(size_t)p * VBGS_REC + i % 28] : (T)V.rec32[(size_t)p * VBGS_REC + i % 28];
    }
    if (threadIdx.x < W) used[threadIdx.x] = 0u;
    __syncthreads();

    // ---- 1. point groups per component ----
    {
        const int c = C == 1 ? 0 : w, p = p0 + c;
        if (p < V.K) {
            float m[6];
#pragma unroll
            for (int i = 0; i < 6; i++) m[i] = V.cb[(size_t)i * V.Kp + p];
            const float chi = V.cb[(size_t)6 * V.Kp + p], lp = V.cb[(size_t)7 * V.Kp + p], lc = V.cb[(size_t)8 * V.Kp + p],
                        la = V.cb[(size_t)9 * V.Kp + p], B = V.cb[(size_t)10 * V.Kp + p];
            auto reaches = [&](const float *box, int stride, int at, float xx, float t) {
                float lo[6], hi[6];
#pragma unroll
                for (int i = 0; i < 6; i++) {
                    lo[i] = box[(size_t)i * stride + at];
                    hi[i] = box[(size_t)(6 + i) * stride + at];
                }
                return !(box_bound(lo, hi, m, m, fmaf(B, xx, chi), lp, lc, la) < t);
            };
            int turn = 0;
            for (int s0 = sa; s0 < sb; s0 += 32) {
                const int s = min(s0 + lane, V.S - 1);
                unsigned m1 = __ballot_sync(kFull, s0 + lane < sb && reaches(V.sbox, V.S, s, V.sx2[s], ord2f(V.sthr[s])));
                while (m1) {
                    const int sg = s0 + __ffs(m1) - 1;
                    m1 &= m1 - 1;
                    if (C == 1 && turn++ % W != w) continue;
                    const int g = sg * 32 + lane, gc = min(g, V.G - 1);
                    const unsigned b =
                        __ballot_sync(kFull, g >= ga && g < gb && reaches(V.gbox, V.G, gc, V.gx2[gc], V.gthr[gc]));
                    if (lane == 0) mask[c * A.nw + sg - sa] = b;
                }
            }
        }
    }
    __syncthreads();

    // ---- 2. pairs ----
    unsigned *q = sq[w];
    int *tag = stag[w];
    T *xs = sx[w], *ws = sw[w];
    int qn = 0, cur = -1, curc = 0;
    unsigned mine = 0, npair = 0;
    T acc = T(0);
    // lane f holds feature f: product of columns ia, ib of [1, x]
    int ia = 0, ib = 0;
    {
        int u = 7;
        if (lane >= 1 && lane < 7) ia = lane;
#pragma unroll
        for (int a = 0; a < 6; a++)
#pragma unroll
            for (int b = a; b < 6; b++, u++)
                if (lane == u) { ia = a + 1; ib = b + 1; }
    }
    auto flush = [&]() {
        if (cur >= 0 && lane < 28) {
            double *d = sacc + (w * C + curc) * 28 + lane;
            *d = (mine >> curc & 1u) ? *d + (double)acc : (double)acc;
        }
        if (cur >= 0) mine |= 1u << curc;
        acc = T(0);
    };
    auto evaluate = [&](int cnt) {
        __syncwarp();
        if (lane < cnt) {
            const unsigned e = q[lane];
            const int n = (int)(e & 0xffffffu);
            const T *r = srec + (e >> 24) * 28;
            T xv[6], ref;
            if (kF64) {
                const double2 *xp = reinterpret_cast<const double2 *>(V.X + (size_t)n * VBGS_XS);
#pragma unroll
                for (int i = 0; i < 3; i++) { const double2 v = xp[i]; xv[2 * i] = (T)v.x; xv[2 * i + 1] = (T)v.y; }
                ref = (T)A.lse[n];
            } else {
#pragma unroll
                for (int i = 0; i < 6; i++) xv[i] = (T)V.xf[(size_t)i * V.Np + n];
                ref = (T)V.lse2f[n];
            }
            ws[lane] = Arith<T>::expd(logit<T>(r, xv) - ref);
            xs[lane * 8] = T(1);
#pragma unroll
            for (int i = 0; i < 6; i++) xs[lane * 8 + 1 + i] = kF64 ? xv[i] : xv[i] - r[i];
        }
        __syncwarp();
        for (int e = 0; e < cnt; e++) {
            const int t = tag[e];
            if (t != cur) {
                flush();
                cur = t;
                curc = (int)(q[e] >> 24);
            }
            const T wv = ws[e], a = xs[e * 8 + ia], b = xs[e * 8 + ib];
            if (kF64) acc = fma(wv, a * b, acc);
            else      acc = fma(wv * a, b, acc);   // w d_a, then times d_b (1 for the lower orders: an exact sum)
        }
        npair += cnt;
        __syncwarp();
    };
    for (int cc = 0; cc < C; cc++) {
        const int c = (cc + w) % C;
        if (p0 + c >= V.K) continue;
        const unsigned *mk = mask + c * A.nw;
        float r[28], x2c = 0.f, chic = 0.f;
        bool loaded = false;
        auto visit = [&](int g, int na, int nb, int tg) {
            if (!loaded) {
                load_rec(V.rec32, p0 + c, r);
                x2c = V.cb[(size_t)10 * V.Kp + p0 + c];
                chic = V.cb[(size_t)6 * V.Kp + p0 + c];
                loaded = true;
            }
            const int n = g * 32 + lane;
            const bool in = n >= na && n < nb;
            const float ch = fmaf(x2c, V.gx2[g], chic);
            float x[6];
#pragma unroll
            for (int i = 0; i < 6; i++) x[i] = V.xf[(size_t)i * V.Np + n];
            const float t = V.thr[n];
            float qd = quad_pos(r, x);
            if (!__any_sync(kFull, in && !(ch - kQuadLo * qd < t))) return;
            qd = quad_rest(r, x, qd);
            const bool surv = in && !(ch - kQuadLo * qd < t);
            const unsigned ms = __ballot_sync(kFull, surv);
            if (!ms) return;
            if (surv) {
                const int at = qn + __popc(ms & ((1u << lane) - 1u));
                q[at] = ((unsigned)c << 24) | (unsigned)n;
                tag[at] = tg;
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
        };
        if (kF64) {
            int turn = c;   // the first group of component c goes to warp -c mod W: light components spread
            for (int s = sa; s < sb; s++) {
                unsigned b = mk[s - sa];
                while (b) {
                    const int g = s * 32 + __ffs(b) - 1;
                    b &= b - 1;
                    if ((turn++ + w) % W == 0) visit(g, 0, V.N, c);
                }
            }
        } else {
            for (int j = j0 + (w + c) % W; j < j1; j += W) {
                const int na = j * A.nps, nb = min((long long)V.N, (long long)(j + 1) * A.nps);
                const int g0 = na >> 5, g1 = (nb - 1) >> 5;
                for (int s = g0 >> 5; s <= g1 >> 5; s++) {
                    unsigned b = mk[s - sa];
                    if (s == g0 >> 5) b &= kFull << (g0 & 31);
                    if (s == g1 >> 5) b &= kFull >> (31 - (g1 & 31));
                    while (b) {
                        const int g = s * 32 + __ffs(b) - 1;
                        b &= b - 1;
                        visit(g, na, nb, c * A.nsplit + j);
                    }
                }
            }
        }
    }
    if (qn) evaluate(qn);
    flush();
    if (lane == 0) used[w] = mine;
    if (A.pairs && lane == 0 && npair) atomicAdd(A.pairs, (unsigned long long)npair);
    __syncthreads();

    // ---- 3. sums of the warps; raw moments ----
    for (int c = w; c < C; c += W) {
        const int p = p0 + c;
        if (p >= V.K) continue;
        double s = 0.0;
        bool any = false;
        for (int i = 0; i < W; i++)
            if (used[i] >> c & 1u) {
                const double v = lane < 28 ? sacc[(i * C + c) * 28 + lane] : 0.0;
                s = any ? s + v : v;
                any = true;
            }
        if (A.slices > 1) {
            if (lane < 28) A.part[((size_t)y * V.K + p) * 28 + lane] = s;
            continue;
        }
        if (A.anchor && any) {
            // S1 = S1' + N a,  S2 = S2' + a S1'^T + S1' a^T + N a a^T
            const double nn = __shfl_sync(kFull, s, 0);
            const double sa1 = __shfl_sync(kFull, s, ia), sb1 = __shfl_sync(kFull, s, ib);
            const double aa = ia ? (double)A.anchor[(size_t)p * VBGS_REC + ia - 1] : 0.0;
            const double ab = ib ? (double)A.anchor[(size_t)p * VBGS_REC + ib - 1] : 0.0;
            if (ib) s += aa * sb1 + sa1 * ab + nn * aa * ab;
            else if (ia) s += nn * aa;
        }
        if (lane < 28) A.dS[(size_t)(A.kperm ? A.kperm[p] : p) * 28 + lane] = s;
    }
}

__host__ __device__ inline size_t even(size_t v) { return (v + 3) & ~size_t(3); }

} // namespace

size_t sparse_scratch_floats(int64_t N, int K)
{
    const size_t Np = (size_t)((N + 31) / 32) * 32, G = Np / 32, S = (G + 31) / 32;
    const size_t Kp = (size_t)((K + 31) / 32) * 32, Kg = Kp / 32;
    return even(8 * Np) + even(14 * G) + even(14 * S) + even(11 * Kp) + even(17 * Kg);
}

bool sparse_fits(int64_t N) { return N > 0 && N <= kMaxPoints; }

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
    f += even((size_t)8 * V.Np);
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
    }
    // warps per block: about 16 a sub-partition over the grid, and no more
    // than there are component groups to share
    int W = 4;
    while (W < 16 && (int64_t)V.G * W < 8 * (int64_t)num_sms * 4 && W < V.Kg) W *= 2;
    const size_t sh1 = (size_t)W * (32 * (8 + 8 + 4 + 4) + 128 * 4);
    P1Args a1{kps, p1_splits, reinterpret_cast<double2 *>(B.part), B.lse, B.lse_part, B.lse_part ? B.scal + SC_SUM_LSE : nullptr,
              done, pf->on ? pf->d_pairs + 1 : nullptr};
    pf->begin(VBGS_PROF_PASS1, st);
    if (f64) launch_pdl(k_sp_pass1<double>, V.G, W * 32, sh1, st, V, a1);
    else     launch_pdl(k_sp_pass1<float>, V.G, W * 32, sh1, st, V, a1);
    pf->end(st);
    if (!want_stats) return cudaGetLastError() == cudaSuccess ? launches - 1 : -1;

    // Components per block: eight while that still gives two blocks an SM;
    // fewer components are taken one by one, with the points cut into slices
    // until the grid fills the SMs (four resident blocks each).
    P2Args a2{};
    const bool many = (V.K + 7) / 8 >= 2 * num_sms;
    int slices = 1;
    if (!many) {
        const int unit = f64 ? (V.G + 15) / 16 : p2_splits;   // at least 512 points (one split) a slice
        slices = std::max(1, std::min(std::min(unit, (4 * num_sms + V.K - 1) / V.K), 1024));
        slices = (int)std::min<size_t>((size_t)slices, std::max<size_t>(1, B.part_cap / ((size_t)V.K * 28)));
    }
    a2.gper = (V.G + slices - 1) / slices;
    a2.spy = (p2_splits + slices - 1) / slices;
    slices = f64 ? (V.G + a2.gper - 1) / a2.gper : (p2_splits + a2.spy - 1) / a2.spy;
    a2.slices = slices;
    a2.nps = (int)nps;
    a2.nsplit = p2_splits;
    a2.nw = (f64 ? a2.gper : (int)(((int64_t)a2.spy * nps + 31) / 32)) / 32 + 2;
    a2.lse = B.lse;
    a2.anchor = f64 ? nullptr : B.rec32;
    a2.kperm = B.kperm;
    a2.dS = B.dS;
    a2.part = B.part;
    a2.pairs = pf->on ? pf->d_pairs : nullptr;
    const bool wide = many && (size_t)a2.nw * 32 <= 8192;   // eight masks of the slice fit
    const size_t sh2 = (size_t)a2.nw * 4 * (wide ? 8 : 1);
    const dim3 g2(wide ? (V.K + 7) / 8 : V.K, slices);
    pf->begin(VBGS_PROF_PASS2, st);
    if (f64) {
        if (wide) launch_pdl(k_sp_pass2<double, 8>, g2, kP2Warps * 32, sh2, st, V, a2);
        else      launch_pdl(k_sp_pass2<double, 1>, g2, kP2Warps * 32, sh2, st, V, a2);
    } else {
        if (wide) launch_pdl(k_sp_pass2<float, 8>, g2, kP2Warps * 32, sh2, st, V, a2);
        else      launch_pdl(k_sp_pass2<float, 1>, g2, kP2Warps * 32, sh2, st, V, a2);
    }
    pf->end(st);
    if (slices > 1) {
        pf->begin(VBGS_PROF_REDUCE, st);
        launch_reduce_splits(B.part, slices, V.K, a2.anchor, B.kperm, B.dS, st);
        pf->end(st);
        launches++;
    }
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

} // namespace vbgs

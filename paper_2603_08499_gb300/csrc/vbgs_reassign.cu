// vbgs_reassign.cu -- the reassign step of Alg. 1 (run before fit in every
// frame; Sec. 2.1.2): n points sampled toward low per-point ELBO, the n
// least-used components, and the prior means of those components set to the
// sampled points.
//
//   points      key_n = g_n - lse_n / tau in caller order; the n largest keys
//               are a sample of n distinct points with probability
//               proportional to exp(-lse_n / tau) (Gumbel-top-k; g_n are
//               standard Gumbel variates the caller draws); ties go to the
//               lower index.
//   components  ascending count N_k of S_past, ties by the caller's key v_k
//               (when given), then by the lower index.
//   apply       m0[comp_i] = x[point_i], i < n.
//
// Both orders are of 64-bit keys that order as the doubles they encode (sign
// bit set for non-negative values, every bit flipped for negative ones; -0 is
// first mapped to +0, so equal values tie).
//   n <= kSelectMax (a call moves 1% of the components): k_select finds the n
//     smallest (key, tie key, index) of the points and of the components side
//     by side, a cluster of blocks each: digits of 11 bits from the top narrow the
//     candidates down until little more than n remain, each of which then
//     counts the smaller ones.  It reads the keys three to six times from the
//     L2 (36,000 points and 50,000 components: 52 us), where three full radix
//     sorts of eight passes each took 220 us.
//   above: CUB's stable radix sort; sorting in caller order makes its
//     stability the tie rule.
#include "vbgs_internal.cuh"
#include <algorithm>
#include <cooperative_groups.h>
#include <cub/device/device_radix_sort.cuh>

namespace cg = cooperative_groups;

namespace vbgs {
namespace {

__device__ __forceinline__ unsigned long long ord64(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(__dadd_rn(v, 0.0));   // -0 -> +0
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Point keys, complemented so that an ascending order puts the largest key
// first.  lse: per-point lse in caller order without the shared
// -psi(sum alpha) term, psi at *psi; the key is g - (lse - psi) / tau with
// each operation rounded once.  bad: bit 0 for a non-finite variate, bit 1 for
// a non-finite component key.
__global__ void k_point_keys(const double *__restrict__ lse, int64_t N, const double *__restrict__ psi,
                             const double *__restrict__ g, double inv_tau, unsigned long long *__restrict__ keys,
                             int *__restrict__ idx, int *__restrict__ bad)
{
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const double l = __dsub_rn(lse[n], *psi), gn = g[n];
    keys[n] = ~ord64(__dsub_rn(gn, __dmul_rn(l, inv_tau)));
    if (idx) idx[n] = (int)n;
    if (!isfinite(gn)) atomicOr(bad, 1);
}

// First component pass (only with a caller key): order by v_k.
__global__ void k_comp_tie_keys(const double *__restrict__ v, int K, unsigned long long *__restrict__ keys,
                                int *__restrict__ idx, int *__restrict__ bad)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double vk = v[k];
    keys[k] = ord64(vk);
    if (idx) idx[k] = k;
    if (!isfinite(vk)) atomicOr(bad, 2);
}

// Second (or only) component pass: the counts N_k = S[k][0] of the sequence
// `order` (NULL: identity), sorted stably so that ties keep that sequence.
__global__ void k_comp_count_keys(const double *__restrict__ S, const int *__restrict__ order, int K,
                                  unsigned long long *__restrict__ keys, int *__restrict__ idx)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= K) return;
    const int k = order ? order[i] : i;
    keys[i] = ord64(S[(size_t)k * VBGS_F]);
    if (idx) idx[i] = k;
}

// The n smallest (key, tie, index) of M, in order.  Cluster 0 takes the points,
// cluster 1 the components (tie nullable); their blocks share the elements,
// add up their digit counts over distributed shared memory and so agree on
// every step; each collects its candidates and copies the others'.  (One block alone, 49
// elements a thread and pass, and a bitonic sort: 114 us.)
constexpr int kSelectMax = 1024, kSelectCap = 2048, kBins = 2048, kSelectThreads = 1024, kSelectCluster = 8;
struct SelectArgs {
    const unsigned long long *key, *tie;
    int M;
    int *out;
};

__global__ void __launch_bounds__(kSelectThreads) k_select(SelectArgs a0, SelectArgs a1, int n)
{
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long *sk = reinterpret_cast<unsigned long long *>(smem_raw), *st = sk + kSelectCap;
    unsigned long long *fk = st + kSelectCap, *ft = fk + kSelectCap;   // this block's candidates; all of them: sk, st, si
    int *si = reinterpret_cast<int *>(ft + kSelectCap), *fi = si + kSelectCap, *hist = fi + kSelectCap;
    __shared__ unsigned long long s_and, s_or;
    __shared__ int s_warp[32], s_bin, s_below, s_count, s_cnt;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const bool comps = blockIdx.x >= kSelectCluster;
    SelectArgs A;
    A.key = comps ? a1.key : a0.key;
    A.tie = comps ? a1.tie : a0.tie;
    A.M = comps ? a1.M : a0.M;
    A.out = comps ? a1.out : a0.out;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, g0 = rank * kSelectThreads + t;
    constexpr int kStep = kSelectCluster * kSelectThreads;
    // What is known of the n-th smallest: its levels before `level` exactly,
    // and the bits mask of val at that level (0: key, 1: tie, 2: index).  below
    // elements are smaller than everything that agrees, count agree.
    unsigned long long known0 = 0, known1 = 0, val = 0, mask = 0;
    int level = 0, below = 0, count = A.M;
    constexpr int kUnroll = 8;   // elements a thread has in flight: a pass is bound by the L2's latency
    int shift = 53;   // of the next digit of 11 bits (the last one has 9: shift 0)
    // (narrowed well below the capacity: the places cost the square of the number)
    const int enough = n + max(64, n >> 3);
    while (below + count > enough) {
        for (int b = t; b < kBins; b += kSelectThreads) hist[b] = 0;
        if (t == 0) { s_and = ~0ull; s_or = 0ull; }
        __syncthreads();
        unsigned long long va = ~0ull, vo = 0ull;
        for (int i0 = 0; i0 < A.M; i0 += kUnroll * kStep) {   // block-uniform: whole warps take part in the ballots
            unsigned long long k[kUnroll], x[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; u++) {
                const int i = i0 + u * kStep + g0;
                k[u] = i < A.M ? A.key[i] : 0ull;
                x[u] = i < A.M && level > 0 && A.tie ? A.tie[i] : 0ull;
            }
#pragma unroll
            for (int u = 0; u < kUnroll; u++) {
                const int i = i0 + u * kStep + g0;
                const unsigned long long v = level == 0 ? k[u] : level == 1 ? x[u] : (unsigned long long)i;
                int d = -1;
                if (i < A.M && (v & mask) == val && (level < 1 || k[u] == known0) && (level < 2 || !A.tie || x[u] == known1)) {
                    d = (int)(v >> shift) & (kBins - 1);
                    if (shift == 0) d &= 511;
                    va &= v;
                    vo |= v;
                }
                // digits are few at the top (exponents, equal counts): one add
                // for each of the warp's first three, the rest one by one
                unsigned left = __ballot_sync(0xffffffffu, d >= 0);
#pragma unroll
                for (int p = 0; p < 3 && left; p++) {
                    const int src = __ffs(left) - 1, dl = __shfl_sync(0xffffffffu, d, src);
                    const unsigned peers = __ballot_sync(0xffffffffu, d == dl) & left;
                    if (lane == src) atomicAdd(&hist[dl], __popc(peers));
                    left &= ~peers;
                }
                if (left >> lane & 1u) atomicAdd(&hist[d], 1);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            va &= __shfl_xor_sync(0xffffffffu, va, o);
            vo |= __shfl_xor_sync(0xffffffffu, vo, o);
        }
        if (lane == 0) { atomicAnd(&s_and, va); atomicOr(&s_or, vo); }
        cluster.sync();
        unsigned long long all_and = ~0ull, all_or = 0ull;
        for (int b = 0; b < kSelectCluster; b++) {
            all_and &= *cluster.map_shared_rank(&s_and, b);
            all_or |= *cluster.map_shared_rank(&s_or, b);
        }
        const bool equal = level < 2 && all_and == all_or;
        if (!equal) {
            // the bin that holds rank n - 1 - below
            int h0 = 0, h1 = 0;
#pragma unroll
            for (int b = 0; b < kSelectCluster; b++) {
                const int2 h = reinterpret_cast<const int2 *>(cluster.map_shared_rank(hist, b))[t];
                h0 += h.x;
                h1 += h.y;
            }
            int incl = h0 + h1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            if (lane == 31) s_warp[w] = incl;
            __syncthreads();
            int base = 0;
            for (int i = 0; i < w; i++) base += s_warp[i];
            const int e0 = base + incl - h0 - h1, e1 = e0 + h0, r = n - 1 - below;
            if (r >= e0 && r < e1) { s_bin = 2 * t; s_below = e0; s_count = h0; }
            if (r >= e1 && r < e1 + h1) { s_bin = 2 * t + 1; s_below = e1; s_count = h1; }
            __syncthreads();
            below += s_below;
            count = s_count;
            val |= (unsigned long long)s_bin << shift;
            mask |= (shift == 0 ? 511ull : (unsigned long long)(kBins - 1)) << shift;
        }
        if (level == 2) {            // (indices differ: at most one agrees after the last digit)
            shift = shift > 9 ? shift - 11 : 0;
        } else if (equal || shift == 0) {   // this level is known: the next one decides
            if (level == 0) known0 = equal ? all_and : val;
            else known1 = equal ? all_and : val;
            level = level == 0 && A.tie ? 1 : 2;
            val = mask = 0;
            shift = level == 2 ? 20 : 53;   // indices: 31 bits, three digits
        } else {
            shift = shift > 9 ? shift - 11 : 0;
        }
        cluster.sync();   // the counts are read before the next digit's
    }
    // candidates: smaller than what is known, or agreeing with it
    if (t == 0) s_cnt = 0;
    __syncthreads();
    for (int i0 = g0; i0 < A.M; i0 += kUnroll * kStep) {
        unsigned long long ku[kUnroll], xu[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; u++) {
            const int i = i0 + u * kStep;
            ku[u] = i < A.M ? A.key[i] : 0ull;
            xu[u] = i < A.M && A.tie ? A.tie[i] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kUnroll; u++) {
            const int i = i0 + u * kStep;
            if (i >= A.M) break;
            const unsigned long long k = ku[u], x = xu[u];
            bool take;
            if (level == 0) take = (k & mask) <= val;
            else if (k != known0) take = k < known0;
            else if (level == 1) take = (x & mask) <= val;
            else if (A.tie && x != known1) take = x < known1;
            else take = ((unsigned long long)i & mask) <= val;
            if (take) {
                const int at = atomicAdd(&s_cnt, 1);
                if (at < kSelectCap) { fk[at] = k; ft[at] = x; fi[at] = i; }
            }
        }
    }
    cluster.sync();
    // Every candidate's place is the number of smaller ones.  The blocks take
    // an eighth of the candidates each against a copy of all of them: lanes
    // hold 32 candidates, a warp compares them with a slice of the others.
    int *place = hist;   // of this block's share of the candidates
    int cnt = 0;
    for (int r = 0; r < kSelectCluster; r++) {
        const int c = min(*cluster.map_shared_rank(&s_cnt, r), kSelectCap - cnt);
        const unsigned long long *rk = cluster.map_shared_rank(fk, r), *rt = cluster.map_shared_rank(ft, r);
        const int *ri = cluster.map_shared_rank(fi, r);
        for (int i = t; i < c; i += kSelectThreads) { sk[cnt + i] = rk[i]; st[cnt + i] = rt[i]; si[cnt + i] = ri[i]; }
        cnt += c;
    }
    for (int i = t; i < kBins; i += kSelectThreads) place[i] = 0;
    cluster.sync();      // copied: a block may leave
    const int per = (cnt + kSelectCluster - 1) / kSelectCluster, e0 = rank * per, e1 = min(cnt, e0 + per);
    const int groups = (per + 31) / 32, slices = max(1, 32 / groups), len = (cnt + slices - 1) / slices;
    for (int job = w; job < groups * slices; job += 32) {
        const int e = e0 + job / slices * 32 + lane, ec = min(e, cnt - 1), j0 = job % slices * len, j1 = min(cnt, j0 + len);
        const unsigned long long k = sk[ec], x = st[ec];
        const int id = si[ec];
        int smaller = 0;
        for (int j = j0; j < j1; j++) {
            const unsigned long long kj = sk[j];
            smaller += kj < k || (kj == k && (st[j] < x || (st[j] == x && si[j] < id)));
        }
        if (e < e1) atomicAdd(&place[e - e0], smaller);
    }
    __syncthreads();
    for (int e = e0 + t; e < e1; e += kSelectThreads)
        if (place[e - e0] < n) A.out[place[e - e0]] = si[e];
}

// m0[comp_i] = x[point_i] (X: staged points, caller order, N x 8), unless the
// E-step or a caller's value was bad; rows and picks (points, then components)
// for the host.
__global__ void k_reassign_apply(const int *__restrict__ pts, const int *__restrict__ comps, int n,
                                 const double *__restrict__ X, double *__restrict__ m0, double *__restrict__ rows,
                                 int *__restrict__ picks, const int *__restrict__ flags, const int *__restrict__ bad)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * 6) return;
    const int i = t / 6, d = t - 6 * i;
    const double x = X[(size_t)pts[i] * VBGS_XS + d];
    const bool good = *bad == 0 && flags[FL_BAD_POINT] == 0 && flags[FL_NONPD] == 0 && flags[FL_TIMEOUT] == 0;
    if (good) m0[(size_t)comps[i] * 6 + d] = x;
    rows[t] = x;
    if (d == 0) {
        picks[i] = pts[i];
        picks[n + i] = comps[i];
    }
}

} // namespace

size_t reassign_temp_bytes(int64_t n)
{
    size_t bytes = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, bytes, (unsigned long long *)nullptr, (unsigned long long *)nullptr,
                                    (int *)nullptr, (int *)nullptr, (int)std::max<int64_t>(n, 1));
    return bytes;
}

int launch_reassign(const ReassignArgs &a, ReassignBuffers &rb, cudaStream_t st)
{
    const int64_t N = a.N;
    const int K = a.K, n = a.n;
    if (n <= 0 || n > N || n > K || N > rb.cap || K > rb.cap) return -1;
    int *picks = reinterpret_cast<int *>(rb.rows + (size_t)n * 6), *bad = picks + (size_t)n * 2;
    if (cudaMemsetAsync(bad, 0, 2 * sizeof(int), st) != cudaSuccess) return -1;   // and the M-step's flag
    const unsigned gn = (unsigned)((N + 255) / 256), gk = (unsigned)((K + 255) / 256);
    int launches = 0;
    if (n <= kSelectMax) {
        const int smem = kSelectCap * 40 + kBins * 4;
        static const bool ok =
            cudaFuncSetAttribute(k_select, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
        if (!ok) return -1;
        k_point_keys<<<gn, 256, 0, st>>>(a.lse, N, a.psi, rb.g, a.inv_tau, rb.k_in, nullptr, bad);
        if (a.have_v) k_comp_tie_keys<<<gk, 256, 0, st>>>(rb.v, K, rb.k_tie, nullptr, bad);
        k_comp_count_keys<<<gk, 256, 0, st>>>(a.S, nullptr, K, rb.k_out, nullptr);
        launch_pdl_cluster(k_select, 2 * kSelectCluster, kSelectThreads, kSelectCluster, smem, st,
                           SelectArgs{rb.k_in, nullptr, (int)N, rb.pts},
                           SelectArgs{rb.k_out, a.have_v ? rb.k_tie : nullptr, K, rb.comps}, n);
        launches = a.have_v ? 4 : 3;
    } else {
        size_t bytes;
        // points: keys in caller order, stable ascending sort of the complemented keys
        k_point_keys<<<gn, 256, 0, st>>>(a.lse, N, a.psi, rb.g, a.inv_tau, rb.k_in, rb.i_in, bad);
        bytes = rb.temp_bytes;
        if (cub::DeviceRadixSort::SortPairs(rb.temp, bytes, rb.k_in, rb.k_out, rb.i_in, rb.pts, (int)N, 0, 64, st) !=
            cudaSuccess)
            return -1;
        // components: by the caller's key first (when given), then stably by N_k
        const int *order = nullptr;
        launches = 4;
        if (a.have_v) {
            k_comp_tie_keys<<<gk, 256, 0, st>>>(rb.v, K, rb.k_in, rb.i_in, bad);
            bytes = rb.temp_bytes;
            if (cub::DeviceRadixSort::SortPairs(rb.temp, bytes, rb.k_in, rb.k_out, rb.i_in, rb.i_out, K, 0, 64, st) !=
                cudaSuccess)
                return -1;
            order = rb.i_out;
            launches += 2;
        }
        k_comp_count_keys<<<gk, 256, 0, st>>>(a.S, order, K, rb.k_in, rb.i_in);
        bytes = rb.temp_bytes;
        if (cub::DeviceRadixSort::SortPairs(rb.temp, bytes, rb.k_in, rb.k_out, rb.i_in, rb.comps, K, 0, 64, st) !=
            cudaSuccess)
            return -1;
    }
    k_reassign_apply<<<(n * 6 + 255) / 256, 256, 0, st>>>(rb.pts, rb.comps, n, a.X, a.m0, rb.rows, picks, a.flags, bad);
    launches++;
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

} // namespace vbgs

// residuals.cu -- eq. (1) residuals, objective and infeasibility certificate
// of the stored flows, all accumulated in FP64 whatever the working
// precision of the flows.
//
//  vertex pass  Delta_ik (eq. (3), (3h)) and h_ik = Delta_ik / delta_i
//               (eq. (2)) in FP64 (FP32 flows summed error-free in FP32
//               pairs first); per block: sum delta h^2, max |Delta|,
//               max |Delta| / d_k.  With FP32 flows it overwrites the sweeps'
//               heights with those of the stored flows.
//  edge pass    sum_k f_e,k, psi_e (eq. (41)), the certificate length
//               l_e = max(0, max_k (h_ik - h_jk)) and min_k f_e,k; per block:
//               sum psi^2, max psi, max psi/scale, sum u_e l_e, min f.
//  final pass   one block: gain = sum_k d_k (h_{s_k,k} - h_{t_k,k}), the
//               reduction of every partial in a fixed order, and
//               margin = gain - sum_e u_e l_e.
//
// Certificate (Theorems 1 and 2, made explicit by Farkas' lemma): with
// potentials pi = h and lengths l >= 0 with pi_ik - pi_jk <= l_e on every
// edge, any feasible flow satisfies
//   sum_k d_k (pi_{s_k,k} - pi_{t_k,k}) = sum_{e,k} f_e,k (pi_ik - pi_jk)
//                                      <= sum_e l_e sum_k f_e,k <= sum_e u_e l_e,
// so margin > 0 proves that eq. (1) has no solution.
//
// The kernels take one instance, or a table of them (a batch: blockIdx.y, in
// the final pass blockIdx.x, is the instance), so that a batch's pass is three
// launches and not three per instance.  One instance's arguments come from
// the constant bank: through the table's pointer the edge pass took 931 us
// against 681 us at m = 39,600, K = 10,000.
#include "widen.cuh"

#include <math.h>

namespace pdr {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kVParts = 3;  // per vertex block: zsum, cons_abs, cons_rel
constexpr int kEParts = 5;  // per edge block: psi2, cost, cap_abs, cap_rel, fmin

__device__ __forceinline__ double wsum(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}
// Of two values, each in every lane: half the additions, in the same tree.
__device__ __forceinline__ void wsum2(double& a, double& b)
{
    const bool upper = (threadIdx.x & 16) != 0;
    double x = (upper ? b : a) + __shfl_xor_sync(kFull, upper ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    a = __shfl_sync(kFull, x, 0);
    b = __shfl_sync(kFull, x, 16);
}
// The larger of a value that is not negative and another (NaN loses), compared
// by their bit patterns: comparisons of doubles run on the FP64 pipe.
__device__ __forceinline__ double max_nn(double x, double y)
{
    const long long b = __double_as_longlong(y);
    return b > __double_as_longlong(x) && b <= 0x7ff0000000000000ll ? y : x;
}
__device__ __forceinline__ double wmax(double x)  // 0 at least
{
    x = max_nn(0.0, x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = max_nn(x, __shfl_xor_sync(kFull, x, o));
    return x;
}
__device__ __forceinline__ double wmin(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmin(x, __shfl_xor_sync(kFull, x, o));
    return x;
}

// The first NS of NV values are summed, the next NX maximised (none is
// negative), the rest minimised, over a warp.
template <int NV, int NS, int NX>
__device__ __forceinline__ void warp_reduce(double* v)
{
#pragma unroll
    for (int q = 0; q + 1 < NS; q += 2) wsum2(v[q], v[q + 1]);
    if constexpr (NS & 1) v[NS - 1] = wsum(v[NS - 1]);
#pragma unroll
    for (int q = NS; q < NV; ++q) v[q] = q < NS + NX ? wmax(v[q]) : wmin(v[q]);
}
// The same over a block; the results are valid in thread 0.  Bound by the FP64
// pipe (every warp's additions, two per clock and SM): sums in pairs and maxima
// by bit patterns take 10 of its instructions per warp for five values, not 25.
template <int NV, int NS, int NX>
__device__ void block_reduce(double* v, double (*smem)[32])
{
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    warp_reduce<NV, NS, NX>(v);
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (l == 0) smem[q][w] = v[q];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = l < nw ? smem[q][l] : q < NS + NX ? 0.0 : INFINITY;
        warp_reduce<NV, NS, NX>(v);
    }
    __syncthreads();
}

// Exact error of one addition (Knuth's TwoSum): a + b = s + e exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Running sum of FP32 terms kept as an unevaluated pair (hi + lo): every
// addition is error-free (TwoSum) and only the small error terms are added
// in FP32, so hi + lo is the exact sum to about 2^-45 of the largest partial
// sum, well inside FP64 rounding of the quantities formed from it.
struct PairSum {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        float e;
        two_sum(hi, x, hi, e);
        lo = __fadd_rn(lo, e);
    }
};

// Four consecutive elements of a padded row as doubles.
__device__ __forceinline__ void load4(const double* p, double* x)
{
    const double2 a = __ldg(reinterpret_cast<const double2*>(p));
    const double2 b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    x[0] = a.x, x[1] = a.y, x[2] = b.x, x[3] = b.y;
}

// The largest |Delta_ik| and |Delta_ik| / d_k are found in FP64 without an
// FP64 division per element: an element goes through the exact FP64 path
// only when its FP32 estimate (relative error below 2^-21) comes within
// 2^-18 of the FP32 estimate of the best exact value so far, so no element
// that could be the maximum is skipped.
constexpr float kSlack = 0.99999619f;  // 1 - 2^-18

// The certificate length max_k (h_ik - h_jk) likewise: with FP32 heights a
// and b (each within 3 x 2^-24 of the FP64 ones) the FP64 difference lies
// within kHeightSlack (|a| + |b|) of a - b.  Only elements whose upper bound
// reaches the row's largest lower bound can be the maximum.
constexpr float kHeightSlack = 4.76837158e-7f;  // 2^-21

// h_i - h_j from Delta and 1/delta, each height rounded before the difference:
// the certificate's potentials are then one fixed vector, whose differences
// along a path telescope.  (A product fused into the subtraction would enter
// unrounded, and a path just as long as the demand's drop could seem shorter.)
__device__ __forceinline__ double height_drop(double di, double wi, double dj, double wj)
{
    return __dsub_rn(__dmul_rn(di, wi), __dmul_rn(dj, wj));
}

// Vertex pass, FP32 flows: one thread per (vertex, four commodities).
// Delta_ik = sum over in-edges (ascending id) - sum over out-edges
// (ascending) + the source/sink term (eq. (3), (3h)), the flows summed
// error-free (PairSum).  Stored: Delta in FP64, from which the later passes
// form h = Delta / delta_i (eq. (2)), and h rounded to FP32.
//
// GB300 issues two FP64 operations per clock and SM, conversions included,
// and that rate bounded the first form of this pass (83 % of the FP64 pipe,
// 19 % of HBM: 384 us at n = 10,000, m = 39,600, K = 2,500).  Here FP64 takes
// one addition and one multiply-add per element: the pair is widened on the
// integer pipe (widen), h is left to the few elements that need it in FP64,
// and 1/delta_i is applied once per four squares.  The three kernels of a
// residual pass at n = 10,000, m = 39,600, K = 10,000: 5.0 ms before, 2.04 ms
// now (vertex 1.31 ms, edge 0.68 ms).
template <bool TABLE>
__global__ void __launch_bounds__(256)
    resid_vertex_pair_kernel(const ResidTask<float>* __restrict__ tasks, const __grid_constant__ ResidTask<float> one)
{
    const ResidTask<float>& task = TABLE ? tasks[blockIdx.y] : one;
    const int nblocks = task.grid_v;
    if ((int)blockIdx.x >= nblocks) return;
    const SweepArgs<float>& a = task.a;
    const ResidIn r = task.r;
    float* const h32 = a.h;
    double* const delta = task.h64;
    double* const part = task.part;
    __shared__ double smem[5][32];
    const int K = a.K;
    const int64_t Kp = a.Kp;
    const float* const f = a.f;
    const int64_t* const inc_ptr = a.inc_ptr;
    const int32_t* const inc = a.inc;
    const uint32_t nvec = (uint32_t)(Kp / 4);
    const uint64_t total = (uint64_t)a.n * nvec;
    double zsum = 0.0, cabs = 0.0, crel = 0.0;
    float cabs32 = 0.f, crel32 = 0.f;  // FP32 estimates of the elements behind cabs, crel
    for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (uint64_t)nblocks * blockDim.x) {
        const uint32_t i = total <= 0xffffffffull ? (uint32_t)idx / nvec : (uint32_t)(idx / nvec);
        const uint32_t v = (uint32_t)(idx - (uint64_t)i * nvec);
        const int k0 = 4 * (int)v;
        PairSum acc[4];
        const int64_t q0 = inc_ptr[i], q1 = inc_ptr[i + 1];
        auto add = [&](int32_t ev, const float4& x) {
            const float sg = ev >= 0 ? 1.f : -1.f;  // in-edges e, then out-edges ~e
            acc[0].add(sg * x.x), acc[1].add(sg * x.y), acc[2].add(sg * x.z), acc[3].add(sg * x.w);
        };
        auto row = [&](int32_t ev) {
            const int64_t e = ev >= 0 ? ev : ~ev;
            return __ldg(reinterpret_cast<const float4*>(f + e * Kp) + v);
        };
        int64_t q = q0;
        for (; q + 4 <= q1; q += 4) {  // four rows in flight
            int32_t ev[4];
            float4 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) ev[u] = inc[q + u];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = row(ev[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) add(ev[u], x[u]);
        }
        for (; q < q1; ++q) {
            const int32_t ev = inc[q];
            add(ev, row(ev));
        }
        const int4 sv = __ldg(reinterpret_cast<const int4*>(a.s + k0));
        const int4 tv = __ldg(reinterpret_cast<const int4*>(a.t + k0));
        const float4 iv = __ldg(reinterpret_cast<const float4*>(r.inv_dem_f + k0));
        const int ss[4] = {sv.x, sv.y, sv.z, sv.w}, tt[4] = {tv.x, tv.y, tv.z, tv.w};
        const float idm[4] = {iv.x, iv.y, iv.z, iv.w};
        const float idg = a.inv_deg[i];
        double D[4], sq = 0.0;
        float hf[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = k0 + j;
            D[j] = widen(acc[j].hi) + widen(acc[j].lo);
            float D32 = __fadd_rn(acc[j].hi, acc[j].lo);
            if (k >= K) D[j] = 0.0, D32 = 0.f;  // the padding carries no commodity
            if (ss[j] == (int)i || tt[j] == (int)i) {  // padding has s = t = -1
                D[j] += ss[j] == (int)i ? r.dem_d[k] : -r.dem_d[k];
                D32 = (float)D[j];
            }
            hf[j] = D32 * idg;
            sq = fma(D[j], D[j], sq);
            const float ad = fabsf(D32);
            if (ad > 0.f) {
                if (ad >= cabs32 * kSlack) {
                    cabs = fmax(cabs, fabs(D[j]));
                    cabs32 = fmaxf(cabs32, ad);
                }
                const float rel = ad * idm[j];
                if (rel >= crel32 * kSlack) {
                    crel = fmax(crel, fabs(D[j]) / r.dem_d[k]);
                    crel32 = fmaxf(crel32, rel);
                }
            }
        }
        zsum = fma(sq, r.inv_deg_d[i], zsum);  // delta_i h^2 = Delta^2 / delta_i
        double2* dp = reinterpret_cast<double2*>(delta + (int64_t)i * Kp + k0);
        dp[0] = make_double2(D[0], D[1]);
        dp[1] = make_double2(D[2], D[3]);
        *reinterpret_cast<float4*>(h32 + (int64_t)i * Kp + k0) = make_float4(hf[0], hf[1], hf[2], hf[3]);
    }
    double v[3] = {zsum, cabs, crel};
    block_reduce<3, 1, 2>(v, smem);
    if (threadIdx.x == 0)
        for (int q = 0; q < kVParts; ++q) part[(int64_t)blockIdx.x * kVParts + q] = v[q];
}

// Vertex pass, FP64 flows: one warp per vertex, each lane four commodities at
// a time; h = Delta / delta_i stored in FP64.
template <bool TABLE>
__global__ void __launch_bounds__(256)
    resid_vertex_kernel(const ResidTask<double>* __restrict__ tasks, const __grid_constant__ ResidTask<double> one)
{
    const ResidTask<double>& task = TABLE ? tasks[blockIdx.y] : one;
    const int nblocks = task.grid_v;
    if ((int)blockIdx.x >= nblocks) return;
    const SweepArgs<double>& a = task.a;
    const ResidIn r = task.r;
    double* const h64 = task.h64;
    double* const part = task.part;
    __shared__ double smem[5][32];
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)nblocks * blockDim.x) >> 5;
    const int nvec = a.Kp / 4;
    double zsum = 0.0, cabs = 0.0, crel = 0.0;
    float cabs32 = 0.f, crel32 = 0.f;  // FP32 estimates of the elements behind cabs, crel
    for (int64_t i = warp; i < a.n; i += nwarps) {
        const int64_t i0 = a.in_ptr[i], i1 = a.in_ptr[i + 1], o0 = a.row_ptr[i], o1 = a.row_ptr[i + 1];
        const double invdeg = r.inv_deg_d[i];
        for (int v = lane; v < nvec; v += 32) {
            const int k0 = 4 * v;
            double D[4] = {0.0, 0.0, 0.0, 0.0};
            float D32[4];
            double x[4];
            for (int64_t q = i0; q < i1; ++q) {
                load4(a.f + (int64_t)a.in_eid[q] * a.Kp + k0, x);
#pragma unroll
                for (int j = 0; j < 4; ++j) D[j] += x[j];
            }
            for (int64_t e = o0; e < o1; ++e) {
                load4(a.f + e * a.Kp + k0, x);
#pragma unroll
                for (int j = 0; j < 4; ++j) D[j] -= x[j];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) D32[j] = (float)D[j];
            const int4 sv = __ldg(reinterpret_cast<const int4*>(a.s + k0));
            const int4 tv = __ldg(reinterpret_cast<const int4*>(a.t + k0));
            const int ss[4] = {sv.x, sv.y, sv.z, sv.w}, tt[4] = {tv.x, tv.y, tv.z, tv.w};
            double h[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = k0 + j;
                if (k >= a.K) D[j] = 0.0;  // the padding carries no commodity
                if (ss[j] == (int)i || tt[j] == (int)i) {  // padding has s = t = -1
                    D[j] += ss[j] == (int)i ? r.dem_d[k] : -r.dem_d[k];
                    D32[j] = (float)D[j];
                }
                h[j] = D[j] * invdeg;
                zsum = fma(D[j], h[j], zsum);  // delta_i h^2 = Delta h
                if (D[j] != 0.0) {
                    const float ad = fabsf(D32[j]);
                    if (ad >= cabs32 * kSlack) {
                        cabs = fmax(cabs, fabs(D[j]));
                        cabs32 = fmaxf(cabs32, ad);
                    }
                    const float rel = ad * r.inv_dem_f[k];
                    if (rel >= crel32 * kSlack) {
                        crel = fmax(crel, fabs(D[j]) / r.dem_d[k]);
                        crel32 = fmaxf(crel32, rel);
                    }
                }
            }
            double2* hp = reinterpret_cast<double2*>(h64 + i * a.Kp + k0);
            hp[0] = make_double2(h[0], h[1]);
            hp[1] = make_double2(h[2], h[3]);
        }
    }
    double v[3] = {zsum, cabs, crel};
    block_reduce<3, 1, 2>(v, smem);
    if (threadIdx.x == 0)
        for (int q = 0; q < kVParts; ++q) part[(int64_t)blockIdx.x * kVParts + q] = v[q];
}

// Edge pass: one warp per edge, each lane four commodities at a time:
// sum_k f_e,k (error-free pairs for FP32 flows), psi_e (eq. (41)), min_k f_e,k
// and the certificate length l_e = max(0, max_k (h_ik - h_jk)) in FP64 (only
// where u_e > 0: an edge without capacity adds nothing to sum_e u_e l_e).
// FP32 flows: h64 holds Delta, and the FP32 heights h32 decide which
// elements need their FP64 difference, so a row costs 12 bytes per element
// and FP64 only at its few candidates (both height rows in FP64 made the
// FP64 pipe the bound: 559 us at m = 39,600, K = 2,500).
template <typename T, bool TABLE>
__global__ void __launch_bounds__(256)
    resid_edge_kernel(const ResidTask<T>* __restrict__ tasks, const __grid_constant__ ResidTask<T> one)
{
    const ResidTask<T>& task = TABLE ? tasks[blockIdx.y] : one;
    const int nblocks = task.grid_e;
    if ((int)blockIdx.x >= nblocks) return;
    const SweepArgs<T>& a = task.a;
    const ResidIn r = task.r;
    const float* const h32 = sizeof(T) == 4 ? reinterpret_cast<const float*>(a.h) : nullptr;
    const double* const h64 = task.h64;
    double* const part = task.part + (int64_t)task.grid_v * kVParts;
    __shared__ double smem[5][32];
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)nblocks * blockDim.x) >> 5;
    const int K = a.K;
    const int64_t Kp = a.Kp, m = a.m;
    const T* const f = a.f;
    const int32_t* const src = a.src;
    const int32_t* const col = a.col;
    const int nvec = a.Kp / 4;
    double psi2 = 0.0, capa = 0.0, capr = 0.0, cost = 0.0, fmn = INFINITY;
    for (int64_t e = warp; e < m; e += nwarps) {
        const double ue = r.u_d[e];
        const bool need_l = ue > 0.0;
        const int64_t ro = (int64_t)src[e] * Kp, co = (int64_t)col[e] * Kp;
        double tot = 0.0, l = 0.0, mn = INFINITY;
        if constexpr (sizeof(T) == 4) {
            PairSum acc;
            // the largest lower bound, and the element with the largest
            // difference: its index and upper bound, and the largest upper
            // bound of the lane's other elements
            float mn32 = INFINITY, lb = 0.f, best = 0.f, up = 0.f, up2 = 0.f;
            int at = -1;
            const float4* fr = reinterpret_cast<const float4*>(f + e * Kp);
            const float4* hi = reinterpret_cast<const float4*>(h32 + ro);
            const float4* hj = reinterpret_cast<const float4*>(h32 + co);
            double wi = 0.0, wj = 0.0;
            if (need_l) {
                wi = r.inv_deg_d[src[e]];
                wj = r.inv_deg_d[col[e]];
            }
#pragma unroll 4
            for (int v = lane; v < nvec; v += 32) {
                const int k0 = 4 * v;
                const float4 x = __ldg(fr + v);
                const float xs[4] = {x.x, x.y, x.z, x.w};
                float p[4] = {}, q[4] = {};
                if (need_l) {
                    const float4 y = __ldg(hi + v), z = __ldg(hj + v);
                    p[0] = y.x, p[1] = y.y, p[2] = y.z, p[3] = y.w;
                    q[0] = z.x, q[1] = z.y, q[2] = z.z, q[3] = z.w;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (k0 + j >= K) continue;  // the padding carries no commodity
                    acc.add(xs[j]);
                    mn32 = fminf(mn32, xs[j]);
                    const float x0 = p[j] - q[j], sl = kHeightSlack * (fabsf(p[j]) + fabsf(q[j]));
                    lb = fmaxf(lb, x0 - sl);
                    const bool more = x0 > best;
                    up2 = fmaxf(up2, more ? up : x0 + sl);
                    up = more ? x0 + sl : up;
                    at = more ? k0 + j : at;
                    best = more ? x0 : best;
                }
            }
            tot = (double)acc.hi + (double)acc.lo;
            mn = (double)mn32;
            if (need_l) {
                const float low = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(lb)));  // lb >= 0
                if (at >= 0 && up >= low) l = fmax(l, height_drop(h64[ro + at], wi, h64[co + at], wj));
                if (__any_sync(0xffffffffu, up2 > 0.f && up2 >= low)) {  // a lane holds several such elements
                    const float* si = h32 + ro;
                    const float* sj = h32 + co;
                    for (int k = lane; k < K; k += 32) {
                        const float x0 = si[k] - sj[k], sl = kHeightSlack * (fabsf(si[k]) + fabsf(sj[k]));
                        if (x0 + sl > 0.f && x0 + sl >= low) l = fmax(l, height_drop(h64[ro + k], wi, h64[co + k], wj));
                    }
                }
            }
        } else {
            for (int v = lane; v < nvec; v += 32) {
                const int k0 = 4 * v;
                double x[4];
                load4(reinterpret_cast<const double*>(f) + e * Kp + k0, x);
                const int nk = K - k0 < 4 ? K - k0 : 4;  // the padding carries no commodity
                for (int j = 0; j < nk; ++j) {
                    tot += x[j];
                    mn = fmin(mn, x[j]);
                }
                if (need_l) {
                    double p[4], q[4];
                    load4(h64 + ro + k0, p);
                    load4(h64 + co + k0, q);
                    for (int j = 0; j < nk; ++j) l = fmax(l, p[j] - q[j]);
                }
            }
        }
        tot = wsum(tot);
        l = wmax(l);
        mn = wmin(mn);
        if (lane == 0) {
            const double over = tot - ue;
            const double psi = over > 0.0 ? over : 0.0;
            psi2 += psi * psi;
            capa = fmax(capa, psi);
            capr = fmax(capr, psi * a.inv_scale[e]);
            cost += ue * l;
            fmn = fmin(fmn, mn);
        }
    }
    double v[5] = {psi2, cost, capa, capr, fmn};
    block_reduce<5, 2, 2>(v, smem);
    if (threadIdx.x == 0)
        for (int q = 0; q < kEParts; ++q) part[(int64_t)blockIdx.x * kEParts + q] = v[q];
}

// One block; its time is the latency of the K gathers and of the partials, so
// every thread keeps several of them in flight.  FP32 flows: h64 holds Delta.
template <typename T, bool TABLE>
__global__ void __launch_bounds__(1024)
    resid_final_kernel(const ResidTask<T>* __restrict__ tasks, const __grid_constant__ ResidTask<T> one)
{
    const ResidTask<T>& task = TABLE ? tasks[blockIdx.x] : one;
    const SweepArgs<T>& a = task.a;
    const ResidIn r = task.r;
    const double* const h64 = task.h64;
    const double* const part = task.part;
    const int grid_v = task.grid_v, grid_e = task.grid_e;
    ResidOut* const out = task.out;
    __shared__ double smem[5][32];
    const double* dem_d = r.dem_d;
    double gain = 0.0, gabs = 0.0;
#pragma unroll 4
    for (int k = threadIdx.x; k < a.K; k += blockDim.x) {
        const int32_t i = a.s[k], j = a.t[k];
        const double wi = sizeof(T) == 4 ? r.inv_deg_d[i] : 1.0, wj = sizeof(T) == 4 ? r.inv_deg_d[j] : 1.0;
        const double diff = height_drop(h64[(int64_t)i * a.Kp + k], wi, h64[(int64_t)j * a.Kp + k], wj);
        gain += dem_d[k] * diff;
        gabs += dem_d[k] * fabs(diff);
    }
    double zv = 0.0, cabs = 0.0, crel = 0.0;
    for (int b = threadIdx.x; b < grid_v; b += blockDim.x) {
        zv += part[(int64_t)b * kVParts + 0];
        cabs = max_nn(cabs, part[(int64_t)b * kVParts + 1]);
        crel = max_nn(crel, part[(int64_t)b * kVParts + 2]);
    }
    const double* pe = part + (int64_t)grid_v * kVParts;
    double psi2 = 0.0, capa = 0.0, capr = 0.0, cost = 0.0, fmn = INFINITY;
    for (int b = threadIdx.x; b < grid_e; b += blockDim.x) {
        psi2 += pe[(int64_t)b * kEParts + 0];
        cost += pe[(int64_t)b * kEParts + 1];
        capa = max_nn(capa, pe[(int64_t)b * kEParts + 2]);
        capr = max_nn(capr, pe[(int64_t)b * kEParts + 3]);
        fmn = fmin(fmn, pe[(int64_t)b * kEParts + 4]);
    }
    double v1[5] = {gain, gabs, zv, cabs, crel};
    block_reduce<5, 3, 2>(v1, smem);
    double v2[5] = {psi2, cost, capa, capr, fmn};
    block_reduce<5, 2, 2>(v2, smem);
    if (threadIdx.x == 0) {
        out->z = 0.5 * (v2[0] + v1[2]);
        out->cap_abs = v2[2];
        out->cap_rel = v2[3];
        out->cons_abs = v1[3];
        out->cons_rel = v1[4];
        out->f_min = a.m > 0 ? v2[4] : 0.0;
        out->margin = v1[0] - v2[1];
        out->margin_scale = v1[1] + v2[1];
    }
}

}  // namespace

int resid_part_count(int32_t grid_v, int32_t grid_e) { return grid_v * kVParts + grid_e * kEParts; }

constexpr int kMaxGridY = 65535;

template <typename T, bool TABLE>
void launch_passes(const ResidTask<T>* tasks, const ResidTask<T>& one, int count, int gv, int ge, int longest, cudaStream_t stream)
{
    if constexpr (sizeof(T) == 4) resid_vertex_pair_kernel<TABLE><<<dim3(gv, count), 256, 0, stream>>>(tasks, one);
    else resid_vertex_kernel<TABLE><<<dim3(gv, count), 256, 0, stream>>>(tasks, one);
    resid_edge_kernel<T, TABLE><<<dim3(ge, count), 256, 0, stream>>>(tasks, one);
    resid_final_kernel<T, TABLE><<<count, longest > 2048 ? 1024 : longest > 256 ? 512 : 256, 0, stream>>>(tasks, one);
}

template <typename T>
cudaError_t launch_residuals(const ResidTask<T>* tasks, const ResidTask<T>* host, int count, cudaStream_t stream)
{
    int gv = 1, ge = 1, longest = 1;
    for (int i = 0; i < count; ++i) {
        gv = host[i].grid_v > gv ? host[i].grid_v : gv;
        ge = host[i].grid_e > ge ? host[i].grid_e : ge;
        longest = host[i].a.K > longest ? host[i].a.K : longest;
    }
    longest = gv > longest ? gv : longest;
    longest = ge > longest ? ge : longest;
    if (!tasks) launch_passes<T, false>(tasks, *host, 1, gv, ge, longest, stream);
    // the instance is the grid's y index, which ends at 65,535
    for (int at = 0; tasks && at < count; at += kMaxGridY)
        launch_passes<T, true>(tasks + at, *host, count - at < kMaxGridY ? count - at : kMaxGridY, gv, ge, longest, stream);
    return cudaGetLastError();
}

template cudaError_t launch_residuals<float>(const ResidTask<float>*, const ResidTask<float>*, int, cudaStream_t);
template cudaError_t launch_residuals<double>(const ResidTask<double>*, const ResidTask<double>*, int, cudaStream_t);

}  // namespace pdr

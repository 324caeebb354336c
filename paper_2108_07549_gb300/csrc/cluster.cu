// cluster.cu -- the cluster engine: the whole solve of a small instance inside
// the shared memory of one thread-block cluster.
//
// A sweep of a small instance is a chain of dependent steps, not a stream of
// bytes, so what counts is the latency of each step.  The csize blocks of a
// cluster split the vertices into contiguous ranges; a block owns its
// vertices' heights and the rows of their out-edges (contiguous in CSR order)
// and keeps them in its shared memory for all sweeps of the launch.  The rows
// of in-edges and the heights at edge heads that another block owns are read
// through distributed shared memory.  Whatever does not change in a sweep is
// worked out once per launch: the addresses of every vertex's incident rows
// (in fours, padded with a row of zeros), the source and sink terms, the
// addresses of the heights at both ends of an edge.  A sweep is two phases,
// each ended by one cluster barrier:
//
//   A  excess pass: h of the block's vertices, and each thread's part of z
//   B  edge QPs of the block's out-edges into the other flow buffer
//
// The stop decision is off this chain.  The block's last kDecWarps warps do
// no sweep work: during phase B they add the threads' parts and send the
// block's sum to every block of the cluster, during the next phase A the
// first of them adds the blocks' sums and applies the stop rules.  The
// decision on z^(t) is therefore known one phase after f^(t+1) was written,
// and the flows are double-buffered, so f^(t) is still there to return; a
// stopped solve has run one update too many, in place of a wait in every
// sweep.  Every block takes the decision from the same numbers in the same
// order, so all agree.
//
// Measured against the graph engine's two launches per sweep (us per sweep, FP32,
// 2000 sweeps; n, m, K): 25, 80, 10: 1.5 against 8.8 (one block); 100, 360, 30:
// 2.1 against 8.6; 200, 600, 50: 3.5 against 9.7; 300, 1200, 56: 5.4 against
// 10.2 (8 blocks); 400, 1600, 90: 9.1 against 10.3 (the graph's gathers have become
// faster since: 6.5 in the first, 7.8 in the third).  In the large ones the reads
// from the other blocks' shared memory bound it (a block's half of the rows
// comes in at roughly 14 bytes per clock), in the small ones the chain of phase
// B: one pass of the search and its decisions, about 1500 cycles.
//
// Per element the arithmetic and its order are those of the standalone
// kernels with the same lane-group variant (excess_body, edge_group_body), so
// the flows, the roots and the residuals equal theirs bit for bit (a padding
// row adds or takes away +0); the parts of z are grouped otherwise (z agrees
// to rounding).
#include "edge_root.cuh"
#include "widen.cuh"

namespace pdr {
namespace {

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_index()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
// Address of `local` (a shared-memory address of this block) in block `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
// All threads of the cluster; orders the shared-memory writes of one phase,
// remote ones included, before the reads of the next.
template <bool CL>
__device__ __forceinline__ void sync_phase()
{
    if constexpr (CL)
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
}
template <bool CL>
__device__ __forceinline__ float4 ld_shared(uint32_t addr)
{
    float4 v;
    if constexpr (CL)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(addr));
    else
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(addr));
    return v;
}

constexpr int kDecWarps = 4;

// Shared-memory layout, the same offsets in every block of a cluster (sized
// for its largest share), each part 16-byte aligned.
struct ClusterLayout {
    int f, fstep;  // flow rows of buffer 0, then one row of zeros; buffer 1 lies fstep bytes further
    int h, d;      // heights; source (+d) and sink (-d) terms
    int th, wm, rstep;  // roots and warm starts of buffer 0; of buffer 1 rstep bytes further
    int u, isc, head, tail, chunk, off, dgt, ideg, idem, sum, mx, dpart, slot, vs, bytes;
};
__host__ __device__ inline ClusterLayout cluster_layout(int n, int m, int chunks, int Kp, int csize)
{
    ClusterLayout L{};
    int o = 0;
    auto take = [&o](int64_t bytes) {
        const int at = o;
        o += (int)((bytes + 15) & ~int64_t(15));
        return at;
    };
    L.f = take((int64_t)(m + 1) * Kp * 4);
    L.fstep = take((int64_t)(m + 1) * Kp * 4) - L.f;
    L.h = take((int64_t)n * Kp * 4);
    L.d = take((int64_t)n * Kp * 4);
    L.th = take((int64_t)m * 4);
    L.wm = take((int64_t)m * 4);
    L.rstep = take((int64_t)m * 4) - L.th;
    take((int64_t)m * 4);
    L.u = take((int64_t)m * 4);
    L.isc = take((int64_t)m * 4);
    L.head = take((int64_t)m * 4);
    L.tail = take((int64_t)m * 4);
    L.chunk = take((int64_t)chunks * 16);
    L.off = take((int64_t)(2 * n + 1) * 4);
    L.dgt = take((int64_t)n * 4);
    L.ideg = take((int64_t)n * 4);
    L.idem = take((int64_t)Kp * 4);
    L.sum = take(1024 * 8);
    L.mx = take(32 * 8);
    L.dpart = take(kDecWarps * 8);
    L.slot = take((int64_t)csize * 16);
    L.vs = take((int64_t)2 * (csize + 1) * 4);
    L.bytes = o;
    return L;
}

// *dst = *src by the whole block, a word per thread.
template <typename X>
__device__ __forceinline__ void copy_words(X* dst, const X* src, int tid)
{
    static_assert(sizeof(X) % 4 == 0, "whole words");
    for (int w = tid; w < (int)(sizeof(X) / 4); w += blockDim.x)
        reinterpret_cast<uint32_t*>(dst)[w] = reinterpret_cast<const uint32_t*>(src)[w];
}

__device__ __forceinline__ float warp_max_pos(float x)  // of values >= 0
{
    return __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(x)));
}

// The sum over lanes whose numbers differ in the bits `from`, from / 2, .. 1.
__device__ __forceinline__ Acc<float>::V xor_sum(Acc<float>::V z, int from)
{
#pragma unroll
    for (int o = from; o > 0; o >>= 1) z = Acc<float>::add(z, Acc<float>::shfl(z, o));
    return z;
}

// The full decision, on the state in shared memory, after `lag` sweeps that
// passed the rules without it: the last of them had 2 z = zl and the maxima
// lcons and lcap, the sweep before it 2 z = zb, and rmin is the smallest
// max(cons, cap) among them.  By one lane; decide = 0 only settles.
__device__ __noinline__ void full_decision(DevState* st, double* trace, int lag, double zl, double zb, float lcons, float lcap,
                                           float rmin, int decide, double z, float cons, float cap, int* stop_now)
{
    if (lag > 0) {
        st->t += lag;
        st->evals += lag;
        st->z = st->z_prev = 0.5 * zl;
        if (lag > 1) st->dz = st->z - 0.5 * zb;
        st->cons_rel = (double)lcons;
        st->cap_rel = (double)lcap;
        if (st->plat_window > 0 && (double)rmin < st->plat_cur) st->plat_cur = (double)rmin;
    }
    if (decide && apply_stop_rules(*st, MODE_SOLVE, trace, 0.5 * z, (double)cons, (double)cap))
        *stop_now = 1;
}

// One cluster per instance: instance table[ids[c]] for cluster c, or `one`.
// The variant's lane groups of G lanes run on P = G / R lanes (edge_root.cuh).
template <int G, int R, int V, bool CL>
__global__ void __launch_bounds__(1024, 1)
    cluster_solve_kernel(const ClusterArgs* __restrict__ table, const int* __restrict__ ids,
                         const __grid_constant__ ClusterArgs one)
{
    using A = Acc<float>;
    constexpr int N = 4, P = G / R, GPW = 32 / P;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ ClusterArgs ca;
    __shared__ ClusterLayout L;
    __shared__ DevState st;
    __shared__ int stop_now;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int workers = (int)blockDim.x - 32 * kDecWarps;
    const int nww = workers >> 5;
    {
        const ClusterArgs* from = table ? table + ids[CL ? cluster_index() : blockIdx.x] : &one;
        copy_words(&ca, from, tid);
        __syncthreads();
        copy_words(&st, ca.a.st, tid);
        if (tid == 0) {
            L = cluster_layout(ca.max_n, ca.max_m, ca.max_chunks, ca.a.Kp, CL ? ca.csize : 1);
            stop_now = 0;
        }
    }
    __syncthreads();
    if (st.stop) return;  // the same in every block: none has written it back before the first barrier
    const int csize = CL ? ca.csize : 1;
    const uint32_t rank = CL ? cluster_rank() : 0u;
    const int Kp = ca.a.Kp, vpr = Kp / N;
    const uint32_t row = 16u * (uint32_t)vpr;  // bytes
    const int v0 = ca.v_start[rank], nr = ca.v_start[rank + 1] - v0;
    const int64_t e0 = ca.a.row_ptr[v0];
    const int mr = (int)(ca.a.row_ptr[v0 + nr] - e0);
    auto fl = [&](int off) { return reinterpret_cast<float*>(sm + off); };
    auto in = [&](int off) { return reinterpret_cast<int32_t*>(sm + off); };
    auto un = [&](int off) { return reinterpret_cast<uint32_t*>(sm + off); };
    const uint32_t base = smem_u32(sm);

    // ---- the block's share into shared memory
    {
        int32_t* const vs = in(L.vs);  // first vertex of every block, then its first edge
        int32_t* const es = vs + csize + 1;
        for (int r = tid; r <= csize; r += blockDim.x) {
            vs[r] = ca.v_start[r];
            es[r] = (int32_t)ca.a.row_ptr[ca.v_start[r]];
        }
        if (tid == 0) {  // chunk offsets of every vertex's in-edges and out-edges
            int c = 0;
            for (int i = 0; i < nr; ++i) {
                in(L.off)[2 * i] = c;
                c += (int)(ca.a.in_ptr[v0 + i + 1] - ca.a.in_ptr[v0 + i] + 3) / 4;
                in(L.off)[2 * i + 1] = c;
                c += (int)(ca.a.row_ptr[v0 + i + 1] - ca.a.row_ptr[v0 + i] + 3) / 4;
            }
            in(L.off)[2 * nr] = c;
        }
        const float4* src = reinterpret_cast<const float4*>(ca.a.f + e0 * Kp);
        float4* dst = reinterpret_cast<float4*>(sm + L.f);
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = tid; q < mr * vpr; q += blockDim.x) dst[q] = src[q];
        const uint32_t zero_row = base + L.f + (uint32_t)ca.max_m * row;
        for (int q = tid; q < 2 * vpr; q += blockDim.x)
            reinterpret_cast<float4*>(sm + L.f + ca.max_m * (int)row + (q >= vpr ? L.fstep : 0))[q >= vpr ? q - vpr : q] = z4;
        for (int q = tid; q < nr * vpr; q += blockDim.x) reinterpret_cast<float4*>(sm + L.d)[q] = z4;
        __syncthreads();
        for (int e = tid; e < mr; e += blockDim.x) {
            fl(L.th)[e] = ca.a.theta_in[e0 + e];
            fl(L.wm)[e] = ca.a.theta_in[ca.a.m + e0 + e];
            fl(L.u)[e] = ca.a.u[e0 + e];
            fl(L.isc)[e] = ca.a.inv_scale_t[e0 + e];
            un(L.tail)[e] = base + L.h + (uint32_t)(ca.a.src[e0 + e] - v0) * row;
            const int j = ca.a.col[e0 + e];
            int r = 0;
            while (j >= vs[r + 1]) ++r;
            const uint32_t at = base + L.h + (uint32_t)(j - vs[r]) * row;
            un(L.head)[e] = CL ? map_rank(at, r) : at;
        }
        for (int i = tid; i < nr; i += blockDim.x) {
            const int64_t i0 = ca.a.in_ptr[v0 + i], i1 = ca.a.in_ptr[v0 + i + 1];
            const int o0 = (int)(ca.a.row_ptr[v0 + i] - e0), o1 = (int)(ca.a.row_ptr[v0 + i + 1] - e0);
            fl(L.ideg)[i] = ca.a.inv_deg[v0 + i];
            fl(L.dgt)[i] = (float)((int)(i1 - i0) + o1 - o0);
            uint32_t* at = un(L.chunk) + 4 * in(L.off)[2 * i];
            for (int64_t q = i0; q < i1; ++q) {
                const int e = ca.a.in_eid[q];
                int r = 0;
                while (e >= es[r + 1]) ++r;
                const uint32_t x = base + L.f + (uint32_t)(e - es[r]) * row;
                *at++ = CL ? map_rank(x, r) : x;
            }
            for (const uint32_t* end = un(L.chunk) + 4 * in(L.off)[2 * i + 1]; at < end; ++at)
                *at = CL ? map_rank(zero_row, rank) : zero_row;
            for (int e = o0; e < o1; ++e) *at++ = base + L.f + (uint32_t)e * row;
            for (const uint32_t* end = un(L.chunk) + 4 * in(L.off)[2 * i + 2]; at < end; ++at) *at = zero_row;
        }
        for (int k = tid; k < Kp; k += blockDim.x) {
            fl(L.idem)[k] = ca.a.inv_dem[k];
            const int s = ca.a.s[k] - v0, t = ca.a.t[k] - v0;  // the padding's -1 stays negative
            if (s >= 0 && s < nr) fl(L.d)[s * Kp + k] = ca.a.dem[k];
            if (t >= 0 && t < nr) fl(L.d)[t * Kp + k] = -ca.a.dem[k];
        }
    }
    __syncthreads();
    const int den = ca.a.ck ? 0 : 2;
    const int sweeps = ca.sweeps;
    int applied = 0;  // sweeps of this launch whose flows stand

    if (warp < nww) {
        // ================================================= sweep work
        const int gl = lane & (P - 1), gw = lane / P;
        const uint32_t F = base + L.f, fstep = (uint32_t)L.fstep;
        float* const th = fl(L.th);
        const int rstep = L.rstep / 4, wmo = (L.wm - L.th) / 4;
        const float* const uu = fl(L.u);
        const float* const isc = fl(L.isc);
        const uint32_t* const head = un(L.head);
        const uint32_t* const tail = un(L.tail);
        const int32_t* const off = in(L.off);
        const uint4* const chunk = reinterpret_cast<const uint4*>(sm + L.chunk);
        // ---- congestion of the starting flows: their row sums in a solve's first
        // launch, the roots of the sweep that made them (psi = den theta) in a later one
        A::V zacc = A::zero();
        float capmax = 0.f;
        for (int b0 = warp * GPW; b0 < mr; b0 += nww * GPW) {
            const int e = b0 + gw;
            const bool valid = e < mr;
            float psi;
            if (ca.first) {
                float rs[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    rs[r] = 0.f;
#pragma unroll
                    for (int q = 0; q < V; ++q) {
                        const int v = gl + r * P + q * G;
                        if (valid && v < vpr) {
                            float x[N];
                            unpack(reinterpret_cast<const float4*>(sm + L.f)[e * vpr + v], x);
#pragma unroll
                            for (int j = 0; j < N; ++j) rs[r] += x[j];
                        }
                    }
                }
                const float sum = share_sum<float, P, R>(rs), ue = valid ? uu[e] : 0.f;
                psi = sum - ue > 0.f ? sum - ue : 0.f;
            } else {
                psi = valid ? (float)den * th[e] : 0.f;
            }
            if (valid && gl == 0) {
                zacc = A::add(zacc, psi * psi);
                const float c = psi * isc[e];
                capmax = c > capmax ? c : capmax;
            }
        }
        // this thread's first (vertex, vector) item and the step to its next
        const int items = nr * vpr;
        const int i0 = tid / vpr, x0 = tid - i0 * vpr, di = workers / vpr, dx = workers - di * vpr;
        sync_phase<CL>();
        for (int q = 0;; ++q) {
            const int b = q & 1;
            if (q == sweeps) {  // the launch's last decision
                __syncthreads();
                applied = stop_now ? q - 1 : q;
                break;
            }
            // ---- phase A
            float cons = 0.f;
            for (int idx = tid, i = i0, v = x0; idx < items; idx += workers) {
                const uint32_t at0 = (b ? fstep : 0u) + 16u * (uint32_t)v;
                const int c0 = off[2 * i], c1 = off[2 * i + 1], c2 = off[2 * i + 2];
                float acc[N] = {0.f, 0.f, 0.f, 0.f};
                for (int c = c0; c < c1; ++c) {
                    const uint4 at = chunk[c];
                    const float4 x = ld_shared<CL>(at.x + at0), y = ld_shared<CL>(at.y + at0);
                    const float4 z = ld_shared<CL>(at.z + at0), w = ld_shared<CL>(at.w + at0);
                    acc[0] += x.x, acc[1] += x.y, acc[2] += x.z, acc[3] += x.w;
                    acc[0] += y.x, acc[1] += y.y, acc[2] += y.z, acc[3] += y.w;
                    acc[0] += z.x, acc[1] += z.y, acc[2] += z.z, acc[3] += z.w;
                    acc[0] += w.x, acc[1] += w.y, acc[2] += w.z, acc[3] += w.w;
                }
                for (int c = c1; c < c2; ++c) {
                    const uint4 at = chunk[c];
                    const float4 x = ld_shared<false>(at.x + at0), y = ld_shared<false>(at.y + at0);
                    const float4 z = ld_shared<false>(at.z + at0), w = ld_shared<false>(at.w + at0);
                    acc[0] -= x.x, acc[1] -= x.y, acc[2] -= x.z, acc[3] -= x.w;
                    acc[0] -= y.x, acc[1] -= y.y, acc[2] -= y.z, acc[3] -= y.w;
                    acc[0] -= z.x, acc[1] -= z.y, acc[2] -= z.z, acc[3] -= z.w;
                    acc[0] -= w.x, acc[1] -= w.y, acc[2] -= w.z, acc[3] -= w.w;
                }
                float dk[N], id[N], hv[N], zt = 0.f;
                unpack(reinterpret_cast<const float4*>(sm + L.d)[idx], dk);
                unpack(reinterpret_cast<const float4*>(sm + L.idem)[v], id);
                const float dgt = fl(L.dgt)[i], idg = fl(L.ideg)[i];
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    acc[j] += dk[j];
                    hv[j] = acc[j] * idg;
                }
                reinterpret_cast<float4*>(sm + L.h)[idx] = pack4(hv);
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    zt += dgt * hv[j] * hv[j];
                    const float r = fabsf(acc[j]) * id[j];
                    cons = r > cons ? r : cons;
                }
                zacc = A::add(zacc, zt);
                i += di;
                v += dx;
                if (v >= vpr) {
                    v -= vpr;
                    ++i;
                }
            }
            reinterpret_cast<float2*>(sm + L.sum)[tid] = make_float2(zacc.hi, zacc.lo);
            cons = warp_max_pos(cons);
            capmax = warp_max_pos(capmax);
            if (lane == 0) reinterpret_cast<float2*>(sm + L.mx)[warp] = make_float2(cons, capmax);
            zacc = A::zero();
            capmax = 0.f;
            sync_phase<CL>();
            if (stop_now) {  // the previous sweep stopped: its f is in the other buffer
                applied = q - 1;
                break;
            }
            // ---- phase B
            const uint32_t fin = F + (b ? fstep : 0u), fout = F + (b ? 0u : fstep);
            float* const th_in = th + b * rstep;
            float* const th_out = th + (b ^ 1) * rstep;
            for (int b0 = warp * GPW; b0 < mr; b0 += nww * GPW) {
                const int e = b0 + gw;
                const bool valid = e < mr;
                const float ue = valid ? uu[e] : 0.f, w = valid ? th_in[wmo + e] : 0.f;
                const uint32_t hj = valid ? head[e] : 0u, hi = valid ? tail[e] : 0u, fr = fin + (uint32_t)e * row;
                float c[R][V][N];
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int q2 = 0; q2 < V; ++q2) {
                        const int v = gl + r * P + q2 * G;
                        if (valid && v < vpr) {
                            float fx[N], ax[N], bx[N];
                            unpack(ld_shared<CL>(hj + 16u * (uint32_t)v), bx);
                            unpack(ld_shared<false>(fr + 16u * (uint32_t)v), fx);
                            unpack(ld_shared<false>(hi + 16u * (uint32_t)v), ax);
#pragma unroll
                            for (int j = 0; j < N; ++j) c[r][q2][j] = fmaf(0.5f, ax[j] - bx[j], fx[j]);
                        } else {
#pragma unroll
                            for (int j = 0; j < N; ++j) c[r][q2][j] = 0.f;
                        }
                    }
                const float theta = qp_root_group<float, P, R, V, N>(c, ue, w, valid, Kp, den);
                unsigned char* const orow = sm + (fout - base) + (uint32_t)e * row;
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int q2 = 0; q2 < V; ++q2) {
                        const int v = gl + r * P + q2 * G;
                        float o[N];
#pragma unroll
                        for (int j = 0; j < N; ++j) {
                            const float x = c[r][q2][j] - theta;
                            o[j] = x > 0.f ? x : 0.f;
                        }
                        if (valid && v < vpr) reinterpret_cast<float4*>(orow)[v] = pack4(o);
                    }
                if (valid && gl == 0) {
                    th_out[wmo + e] = next_warm_start(theta, th_in[e]);
                    th_out[e] = theta;
                    const float psi = (float)den * theta;
                    zacc = A::add(zacc, psi * psi);
                    const float cc = psi * isc[e];
                    capmax = cc > capmax ? cc : capmax;
                }
            }
            sync_phase<CL>();
        }
    } else {
        // ================================================= sums and decisions
        const int dw = warp - nww, dt = tid - workers;
        double* const trace = rank == 0 ? ca.a.trace : nullptr;
        const bool trace_on = ca.a.trace != nullptr && st.trace_len > 0;  // (in every block: all decide alike)
        int4* const slot = reinterpret_cast<int4*>(sm + L.slot);
        float2* const dpart = reinterpret_cast<float2*>(sm + L.dpart);
        // z is summed as the standalone kernels sum it: FP32 pairs within a block,
        // the blocks' sums in FP64, and its change dz is formed in FP64.  An ordinary
        // sweep then passes the rules in FP32 on registers: whatever is not clear of
        // its threshold by more than the rounding of that (1 % is far more), and every
        // sweep that is traced, takes the full decision in FP64, which costs more than
        // a whole phase of a tiny instance.  eps <= 0 never fires; a tolerance rounded
        // down to a float decides floats as it would in FP64.
        const float eps = st.eps_obj > 0.0 ? 2.02f * __double2float_ru(st.eps_obj) : -1.f;
        const float epr = st.eps_rel > 0.0 ? 1.01f * __double2float_ru(st.eps_rel) : -1.f;
        const float tol = st.resid_tol > 0.0 ? __double2float_rd(st.resid_tol) : -1.f;
        const bool fall = st.stop_on_rise != 0;
        double zl = 0.0, zb = 0.0;  // 2 z of the last two sweeps (lag of them unsettled)
        float lcons = 0.f, lcap = 0.f, rmin = 0.f;
        int lag = 0, left = 0;  // left: sweeps before the sweep cap or the end of a plateau window
        auto decide = [&]() {
            int4 p = make_int4(0, 0, 0, 0);
            if (lane < csize) p = slot[lane];
            double z = widen(__int_as_float(p.x)) + widen(__int_as_float(p.y));
            const float cons = warp_max_pos(__int_as_float(p.z)), cap = warp_max_pos(__int_as_float(p.w));
            if constexpr (CL) {
                for (int o = csize >> 1; o > 0; o >>= 1) z += __shfl_xor_sync(kFull, z, o);
            }
            z = __shfl_sync(kFull, z, 0);
            const float dz = (float)(z - zl), zf = (float)z, slack = 1e-13f * zf, least = fmaxf(eps, epr * zf);
            if (left > 0 && fabsf(zf) < 1e38f && (least < 0.f || fabsf(dz) > least + slack) &&
                !(cap <= tol && cons <= tol) && !(fall && dz > -slack)) {
                zb = zl;
                zl = z;
                lcons = cons;
                lcap = cap;
                const float r = cons > cap ? cons : cap;
                rmin = lag > 0 && rmin < r ? rmin : r;
                ++lag;
                --left;
                return;
            }
            if (lane == 0) full_decision(&st, trace, lag, zl, zb, lcons, lcap, rmin, 1, z, cons, cap, &stop_now);
            __syncwarp();
            lag = 0;
            zl = z;
            long long room = st.max_sweeps - st.t;
            if (st.plat_window > 0 && st.plat_t0 + st.plat_window - 1 - st.t < room)
                room = st.plat_t0 + st.plat_window - 1 - st.t;
            left = trace_on ? 0 : room < 0x7fffffff ? (int)room : 0x7fffffff;
        };
        sync_phase<CL>();
        for (int q = 0;; ++q) {
            if (q == sweeps) {
                if (dw == 0) decide();
                __syncthreads();
                applied = stop_now ? q - 1 : q;
                break;
            }
            if (dw == 0 && q > 0) decide();
            sync_phase<CL>();
            if (stop_now) {
                applied = q - 1;
                break;
            }
            // the threads' parts, then the block's sum to every block
            constexpr int kParts = 1024 / (32 * kDecWarps);
            A::V part[kParts];
#pragma unroll
            for (int l = 0; l < kParts; ++l) {
                const int at = dt + l * 32 * kDecWarps;
                const float2 x = at < workers ? reinterpret_cast<const float2*>(sm + L.sum)[at] : make_float2(0.f, 0.f);
                part[l] = A::V{x.x, x.y};
            }
#pragma unroll
            for (int w = kParts / 2; w > 0; w >>= 1)
#pragma unroll
                for (int l = 0; l < w; ++l) part[l] = A::add(part[l], part[l + w]);
            const A::V z = xor_sum(part[0], 16);
            if (lane == 0) dpart[dw] = A::store(z);
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kDecWarps) : "memory");
            if (dw == 0) {
                float2 mx = make_float2(0.f, 0.f);
                if (lane < nww) mx = reinterpret_cast<const float2*>(sm + L.mx)[lane];
                const float2 p = dpart[lane & (kDecWarps - 1)];
                const A::V zz = xor_sum(A::V{p.x, p.y}, kDecWarps / 2);
                const float cons = warp_max_pos(mx.x), cap = warp_max_pos(mx.y);
                if (lane < csize) {
                    if constexpr (CL)
                        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                         map_rank(smem_u32(slot) + 16u * rank, lane)),
                                     "r"(__float_as_int(zz.hi)), "r"(__float_as_int(zz.lo)), "r"(__float_as_int(cons)),
                                     "r"(__float_as_int(cap))
                                     : "memory");
                    else
                        *slot = make_int4(__float_as_int(zz.hi), __float_as_int(zz.lo), __float_as_int(cons),
                                          __float_as_int(cap));
                }
            }
            sync_phase<CL>();
        }
        if (rank == 0 && dt == 0) {
            full_decision(&st, trace, lag, zl, zb, lcons, lcap, rmin, 0, zl, 0.f, 0.f, &stop_now);
            *ca.a.st = st;
        }
    }

    // ---- the current flows, roots and warm starts back to their global buffers
    {
        const int b = applied & 1;
        float* gf = b ? ca.a.f_out : ca.a.f;
        float* gth = b ? ca.a.theta : const_cast<float*>(ca.a.theta_in);
        float4* dst = reinterpret_cast<float4*>(gf + e0 * Kp);
        const float4* src = reinterpret_cast<const float4*>(sm + L.f + b * L.fstep);
        for (int q = tid; q < mr * vpr; q += blockDim.x) dst[q] = src[q];
        for (int e = tid; e < mr; e += blockDim.x) {
            gth[e0 + e] = fl(L.th + b * L.rstep)[e];
            gth[ca.a.m + e0 + e] = fl(L.wm + b * L.rstep)[e];
        }
    }
}

template <int G, int R, int V, bool CL>
cudaError_t launch_gv(const ClusterArgs* table, const int* ids, const ClusterArgs& one, int count, int csize, int threads,
                      int bytes, cudaStream_t stream)
{
    auto* kernel = cluster_solve_kernel<G, R, V, CL>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterSmemMax);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(count * csize));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)csize;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = CL ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, table, ids, one);
}

}  // namespace

int cluster_bytes(int max_n, int max_m, int max_chunks, int Kp, int csize)
{
    // (64-bit first: an instance far beyond shared memory must not wrap)
    const int64_t rows = 8 * (int64_t)max_m * Kp + 8 * (int64_t)max_n * Kp;
    if (rows > kClusterSmemMax || (int64_t)max_chunks + max_m + max_n > kClusterSmemMax) return kClusterSmemMax + 1;
    return cluster_layout(max_n, max_m, max_chunks, Kp, csize).bytes;
}

int cluster_workers(int threads) { return threads - 32 * kDecWarps; }

int cluster_shares(int cfg, int want)  // the largest share count built for the variant, up to `want`
{
    return edge_plain_config(cfg) == 5 ? (want >= 2 ? 2 : 1) : want >= 4 ? 4 : want >= 2 ? 2 : 1;
}

cudaError_t launch_cluster(int cfg, int shares, const ClusterArgs* table, const int* ids, const ClusterArgs& one, int count,
                           int csize, int threads, int bytes, cudaStream_t stream)
{
    if (count <= 0) return cudaSuccess;
    if (csize < 1 || csize > kClusterMax || (csize & (csize - 1)) || threads <= 32 * kDecWarps || threads > 1024 ||
        threads % 32 || bytes < 0 || bytes > kClusterSmemMax)
        return cudaErrorInvalidValue;
#define PDR_CLUSTER_R(G, R, V)                                                                            \
    return csize > 1 ? launch_gv<G, R, V, true>(table, ids, one, count, csize, threads, bytes, stream)    \
                     : launch_gv<G, R, V, false>(table, ids, one, count, csize, threads, bytes, stream)
#define PDR_CLUSTER(G, V)                       \
    if (shares == 4) PDR_CLUSTER_R(G, 4, V);    \
    if (shares == 2) PDR_CLUSTER_R(G, 2, V);    \
    PDR_CLUSTER_R(G, 1, V)
    switch (edge_plain_config(cfg)) {
    case 0: PDR_CLUSTER(4, 1);
    case 1: PDR_CLUSTER(8, 1);
    case 2: PDR_CLUSTER(16, 1);
    case 3: PDR_CLUSTER(32, 1);
    case 4: PDR_CLUSTER(32, 2);
    case 5:
        if (shares == 2) PDR_CLUSTER_R(32, 2, 4);
        PDR_CLUSTER_R(32, 1, 4);
    default: return cudaErrorInvalidValue;
    }
#undef PDR_CLUSTER
#undef PDR_CLUSTER_R
}

}  // namespace pdr

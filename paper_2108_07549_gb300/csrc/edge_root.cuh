// edge_root.cuh -- the root search of Alg. 2 over one lane group, shared by the
// edge kernels (sweep.cu) and the cluster engine (cluster.cu).
#pragma once

#include "sweep_common.cuh"

namespace pdr {
namespace {

// ------------------------------------------------------------------ the root search of Alg. 2
//
// Every pass over a row returns three group-wide values for a threshold w:
// S(w) = sum of the c_k > w, n(w) = their number and m(w) = the smallest of
// them.  theta = (S(w) - u)/(2 + n(w)) is the root of the active set
// A = {c > w}; if m(w) > theta, no element of A falls at or below theta, so A
// is the active set of its own root and the search ends without another
// pass.  Otherwise the elements c <= theta leave (Michelot's step) and the
// next pass starts at theta.  In a converged solve the warm start w lies just
// below the root with no element in between, so one pass decides the edge.

// A lane group of G lanes may run on P = G / R of them: physical lane p then
// holds the rows of lanes p, p + P, ... p + (R - 1) P (its R shares, c[r]),
// and the sums follow the tree of G lanes (the offsets G/2 .. P inside a lane,
// the rest by shuffle), so the results are those of G lanes bit for bit.  The
// fixed cost of an edge (shuffles, decisions, the division) is per physical
// warp, so R = 4 needs about a third of the instructions per edge where the
// rows are short.

// Sum over the group of one value per share.
template <typename T, int P, int R>
__device__ __forceinline__ T share_sum(T (&x)[R])
{
#pragma unroll
    for (int s = R / 2; s > 0; s >>= 1)
#pragma unroll
        for (int r = 0; r < s; ++r) x[r] += x[r + s];
    return group_sum<P>(x[0]);
}

template <typename T, int P, int R, int V, int N>
__device__ __forceinline__ void above(const T (&c)[R][V][N], T w, T& S, int& n, T& mn)
{
    T sl[R], ml = T(INFINITY);
    int nl = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        sl[r] = T(0);
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const T x = c[r][q][j];
                if (exceeds(x, w)) {
                    sl[r] += x;
                    ++nl;
                    ml = min_pos(x, ml);
                }
            }
    }
    S = share_sum<T, P, R>(sl);
    if constexpr (P == 32 && sizeof(T) == 4) {
        // whole-warp groups: one redux each for the count and the minimum
        // (every counted x exceeds w >= 0, so ml is positive or +inf and its
        // bit pattern orders as an unsigned integer)
        n = (int)__reduce_add_sync(kFull, (unsigned)nl);
        mn = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(ml)));
    } else {
        n = group_sum<P>(nl);
#pragma unroll
        for (int o = P / 2; o > 0; o >>= 1) ml = min_pos(__shfl_xor_sync(kFull, ml, o), ml);
        mn = ml;
    }
}

// The search for the root of one edge, one step per pass over its row: feed it
// the sums above threshold w and it sets the next threshold, or done.
//
// While no threshold at or below the root is known, w is a guess: the warm
// start, certified by g(w) = sum max(0, c - w) - u - den w >= 0.  A guess that
// fails lies above the root; since g is convex and decreasing, the tangent at
// w meets 0 at (S(w) - u)/(den + n(w)) <= root, which is the next guess (and
// the root itself if no element lies between the two).  Only if rounding spoils
// that too does the search start from w = 0, where Case 1 of Alg. 2 is
// decided.  From a certified threshold on, Michelot's steps raise theta to the
// root.  The root is (S_A - u)/(den + |A|) of its active set however it is
// reached.  (A failed guess used to start again from 0, two to four passes
// away.  Passes per search, of the slowest edge of a warp, are now 1.02 to 1.3.)
// den = 2 for Alg. 2 (the congestion term of eq. (10) gives theta = (S_A - u)/
// (2 + |A|)); den = 0 with the capacity kept (Program (6): sum_A (c - theta) = u).
template <typename T>
struct RootSearch {
    T w, theta = T(0);
    int nA = 0;            // size of the active set behind theta, or of the last failed guess
    bool certified = false, guessed = false, done;
    __device__ __forceinline__ RootSearch(T w0, bool valid) : w(w0 > T(0) ? w0 : T(0)), done(!valid) {}
    __device__ __forceinline__ void step(T S, int n, T mn, T ue, int den)
    {
        if (done) return;
        if (certified) {
            if (n >= nA || n == 0) {  // no element left: keep theta
                done = true;
                return;
            }
        } else if (w <= T(0)) {
            if (S <= ue) {  // Case 1 of Alg. 2: nothing to shed
                done = true;
                return;
            }
            certified = true;  // Case 2 (S > u >= 0, so n >= 1)
        } else if (n > 0 && ((guessed && n == nA) || S - T(n) * w - ue - T(den) * w >= T(0))) {
            certified = true;  // w <= root, Case 2
        }
        const T t = n > 0 ? (S - ue) / T(den + n) : T(0);
        nA = n;
        if (certified) {
            w = theta = t;
            done = mn > theta;  // no element of the set at or below its root
        } else {
            w = !guessed && t > T(0) && t < w ? t : T(0);
            guessed = true;
        }
    }
    // A Case 2 root below 0 can only come from rounding in sums that put
    // s = sum max(0, c) within rounding of u: that edge is in Case 1 (root 0).
    // Without the clamp, f' = max(0, c - theta) would lift every c <= 0 --
    // the zero padding included -- to -theta.
    __device__ __forceinline__ T root() const { return theta > T(0) ? theta : T(0); }
};

// theta = psi'/2 for the row c (all lanes of the warp call it; `valid` is
// uniform over the lane group).  w0 is the warm start (>= 0).
template <typename T, int P, int R, int V, int N>
__device__ __forceinline__ T qp_root_group(const T (&c)[R][V][N], T ue, T w0, bool valid, int Kp, int den)
{
    RootSearch<T> rs(w0, valid);
    for (int it = 0; it <= Kp + 4; ++it) {  // the limit is never reached: nA drops every certified step
        T S, mn;
        int n;
        above<T, P, R, V, N>(c, rs.w, S, n, mn);
        rs.step(S, n, mn, ue, den);
        if (!__any_sync(kFull, !rs.done)) break;
    }
    return rs.root();
}

// One lane per lane of the group (R = 1).
template <typename T, int G, int V, int N>
__device__ __forceinline__ T qp_root_group(const T (&c)[V][N], T ue, T w0, bool valid, int Kp, int den)
{
    return qp_root_group<T, G, 1, V, N>(reinterpret_cast<const T(&)[1][V][N]>(c), ue, w0, valid, Kp, den);
}

// Warm start of the next sweep's root search from this sweep's root theta
// and the previous one, prev.  A root that rose is expected to stay at or
// above theta; one that fell is expected to fall by about as much again.
// Starting the search at the previous root itself leaves out the many
// entries whose flows have decayed to zero, which sit just above it (c_k =
// theta + f'_k): one pass decides almost every edge.  A start above the
// new root is detected by its certificate g(w) < 0 and costs a cold pass.
template <typename T>
__device__ __forceinline__ T next_warm_start(T theta, T prev)
{
    if (theta > prev) return theta;
    const T w = T(0.999) * theta + T(2) * (theta - prev);
    return w > T(0) ? w : T(0);
}

}  // namespace
}  // namespace pdr

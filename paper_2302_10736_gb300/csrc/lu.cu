// lu.cu - sparse LU solve of the reduced Newton system J_r dx = F on the GPU
// (the paper hands the Jacobian to a sparse direct solver, KLU, and does not
// study the solve; this is this library's own).
//
// Analysis (host, once per set of bus types):
//   * J_r is structurally symmetric when equation P_i is paired with unknown
//     theta_i and Q_i with v_i, so its pattern is that of a graph on the
//     buses; the buses are ordered by minimum degree (each elimination joins
//     the eliminated bus's neighbours into a clique; ties to the lowest bus),
//     which keeps the factor close to the matrix on power grids (about 1.5
//     times its entries on the synthetic grids), and a bus's unknowns stay
//     adjacent (theta, then v).
//   * The elimination tree of the buses and its columns' patterns; chains of
//     the tree whose patterns nest are merged into fronts (supernodes), also
//     where that adds a bounded share of zeros (merge_fronts), and the unknowns
//     renumbered so that a front's pivots are consecutive and follow its
//     subtree's (postorder).
//
// Numeric phase (GPU), multifrontal LU without pivoting (Duff & Reid 1983): a
// front of p pivots and r border unknowns is a dense (p + r) x (p + r + 1)
// matrix (the last column the right-hand side) that sums the entries of A whose
// first unknown it owns and its children's updates; eliminating its pivots
// leaves the pivot rows of U and y and an r x (r + 1) update for its parent:
//     l_i = m_ik / m_kk,   m_ij -= l_i m_kj     (k < p; i, j > k, y with it)
// Backward, x_p = U_pp^-1 (y - U_pr x_r) from the root down.
//
// What bounds it.  The arithmetic is small (5.5 M FMAs at 25,000 buses, 10 us of
// the GPU's FP64 rate); the solve is the latency of the tree's longest path, so it
// is built around few, cheap dependent steps:
//   * Fronts instead of columns: 105 levels of buses are 22 of fronts at 10,000
//     buses, and a front's only global round trips are its children's updates in
//     and its own out.
//   * No schedule and no polling on the way up: a warp, CTA or cluster that
//     finishes a front counts itself at the parent, and the last child to arrive
//     goes on with the parent.
//   * A sub-partition's FP64 unit takes a warp instruction in 64 cycles, whatever
//     its active lanes and however independent the next one (measured: 64.1
//     cycles per FMA for 1 to 64 threads of an SM, dependent or 8 chains; 76 with
//     all four sub-partitions busy).  So a row of a front lies across a whole
//     warp, rows go round the sub-partitions and, for large fronts, the SMs of a
//     cluster, and nothing uniform is computed more than once: pivot rows are
//     scaled by the reciprocal (unit-diagonal U), so that multipliers and the
//     backward solve need no FP64 operation of their own.
// The kernels, by the size of a front (plan_classes): k_mf_small, a warp per front
// in shared memory; k_mf_mid, a CTA, and k_mf_wide, a cluster of 8 CTAs, with the
// front in registers; k_mf_huge, a cluster in global memory.  k_mf_back_big,
// k_mf_back_small: the backward solve; a CTA or warp follows one heavy path of the
// tree down and waits (bounded) only at its head.
//
// One solve (CUDA-profiled kernels, us): 2,000 buses 378 -> 155, 10,000 962 -> 293,
// 25,000 1,752 -> 490, 70,000 3,111 -> 857, against a left-looking factorization
// by columns whose every level cost a chain of L2 round trips, with the top of the
// tree as one dense block of a cluster and an FP64 reciprocal in each of its warps.
// Of the 293 us at 10,000 buses, small 19, mid 101 (4 us a level of the tree, of
// which the update's way to the parent through L2, by atomic and back, is half),
// wide 105, backward 64.
//
// Every sum has a fixed order (children in order of their pivots, lane-strided
// partial sums joined by a fixed shuffle tree): the results are bitwise
// repeatable.  A zero or non-finite pivot sets the grid's error word (no trap);
// a wait that runs out (2 s) sets it to a time-out and ends the warp or CTA.
#include <algorithm>
#include <set>
#include <vector>

#include "fastmath.cuh"
#include "pf_internal.h"
#include "ptx.cuh"

namespace pf {

namespace {

constexpr uint64_t kLuWaitNs = 2000000000ull;   // bounded waits (2 s)
// classes of fronts, by who eliminates them (kMfClasses): a warp, a CTA, a
// cluster of CTAs, and, beyond those, a cluster with the front in global memory
constexpr int kMfSmall = 12, kMfMid = 63, kMfWide = 255;   // most unknowns of a front of the first three
constexpr int kMfNone = (int)0x80000000;   // no source
constexpr int kMfSmallLd = 13;        // row stride of a small front (odd: no bank conflicts down a column)
constexpr int kMfSmallWarps = 16;     // warps per CTA of k_mf_small and k_mf_back_small
constexpr int kMfMidWarps = 8;        // warps per CTA of the second class
constexpr int kMfWideWarps = 8, kMfWideCtas = 8;           // of the third
constexpr int kMfBackSmall = kMfSmall * kMfSmall + kMfSmall;   // doubles of a small front's pivot rows and y
constexpr int kMfHugeThreads = 512, kMfHugeCtas = 8;       // of the last
constexpr int kMfBackThreads = 512;
constexpr int kMfMidRows = kMfMid;    // pivot rows kept in shared memory at a time: all of a front of the second class
constexpr size_t kMfWideRowBytes = 200u * 1024u;           // ... and what fits, of the third
constexpr size_t kMfMaxSmem = 220u * 1024u;

struct MfArgs {
    int n, nf, nnzA;
    int backmax;            // unknowns of the largest front but the small ones
    int backp, backw;       // its pivots in whole warps; doubles of the backward solve's copies of U
    int nleaf[kMfClasses];  // fronts without children of their class
    int npath[2];           // backward paths of the small fronts, of the others
    const MfFront *fr;
    const int *leaf[kMfClasses];   // longest remaining path first
    const int *path[2];            // heads, top down
    const int2 *el;         // per element of a front: {its first source (mf_source; kMfNone), its further ones in ext (-1: none)}
    const int4 *ext;        // {how many, the first three}, then the others
    const int *bidx;        // per border unknown: its number
    const int *rel;         // ... and its place in the parent (pivots, border)
    const int *perm;        // unknown -> reduced index
    const double *A, *F;
    double *U, *cb, *x, *dx, *mat;   // pivot rows and y; updates; solution; fronts beyond shared memory
    int *cnt;               // [nf] children arrived; [nf] x written; item counters
    int *err;
};

// The kernels of a solve are programmatic dependents of one another: the next
// one's CTAs start as this one runs out of work, and wait here until it is done
// (a Newton step at 25,000 buses 520 -> 511 us, four in a power flow at 10,000
// buses 1,358 -> 1,320; 513 and 1,333 with every slot waited for, mf_drain).
__device__ __forceinline__ void mf_begin()
{
    pdl_launch_dependents();
    pdl_wait();
}

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// wait until *p != 0, at most kLuWaitNs; false (and the grid's error word set
// to a time-out) if it stays 0
__device__ __forceinline__ bool mf_wait(const MfArgs &a, const int *p)
{
    if (ld_acquire(p)) return true;
    const uint64_t t0 = global_timer_ns();
    for (;;) {
        __nanosleep(20);
        if (ld_acquire(p)) return true;
        if (global_timer_ns() - t0 > kLuWaitNs) {
            atomicExch(a.err, DEV_TIMEOUT);
            return false;
        }
    }
}

// wait for a pivot row's slot (phase 0 of its mbarrier), bounded in the same way;
// no sleep between the polls: the slot's arrival is on the critical path
__device__ __forceinline__ bool mf_wait_slot(const MfArgs &a, uint64_t *bar)
{
    uint64_t t0 = 0;
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, 0)) return true;
        if (i % 1024 == 0) {
            const uint64_t t = global_timer_ns();
            if (t0 == 0) t0 = t;
            if (t - t0 > kLuWaitNs) {
                atomicExch(a.err, DEV_TIMEOUT);
                return false;
            }
        }
    }
}

__device__ __forceinline__ void pivot_check(const MfArgs &a, double d)
{
    if (!(fabs(d) > 0.0) || !isfinite(d)) atomicExch(a.err, DEV_SINGULAR);
}

// t / w for 0 <= t < w^2 and 1 <= w <= 2^10 (rw = 1 / w): t + 1/2 is exact and
// at least 1/2 from every multiple of w, and the quotient, below 2^10, is off by
// less than 2^-22 of itself, below 1 / (2 w)
__device__ __forceinline__ int fast_div(int t, float rw) { return (int)(((float)t + 0.5f) * rw); }

// ------------------------------------------------------- factorization ----

// a front's source: an element of an update, or (negative) an entry of A or F
__device__ __forceinline__ double mf_source(const MfArgs &a, int k)
{
    if (k >= 0) return __ldcg(a.cb + k);
    k = ~k;
    return k < a.nnzA ? a.A[k] : a.F[k - a.nnzA];
}

// N elements from their sources, in order (A's entry, then the children's): the
// first sources and the lists of the further ones are in flight together, then
// three further ones of each.  The (few) elements with more are left marked in
// `rest` for mf_gather_rest, so that no loop keeps the next elements' loads back.
template <int N>
__device__ __forceinline__ void mf_gather(const MfArgs &a, const int2 (&e)[N], double (&x)[N], uint32_t &rest)
{
    int4 q[N];
#pragma unroll
    for (int u = 0; u < N; ++u) q[u] = e[u].y >= 0 ? a.ext[e[u].y] : make_int4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < N; ++u) x[u] = e[u].x != kMfNone ? mf_source(a, e[u].x) : 0.0;
    double v[N][3];
#pragma unroll
    for (int u = 0; u < N; ++u) {
        v[u][0] = q[u].x > 0 ? mf_source(a, q[u].y) : 0.0;
        v[u][1] = q[u].x > 1 ? mf_source(a, q[u].z) : 0.0;
        v[u][2] = q[u].x > 2 ? mf_source(a, q[u].w) : 0.0;
    }
    rest = 0;
#pragma unroll
    for (int u = 0; u < N; ++u) {
        if (q[u].x > 0) x[u] += v[u][0];
        if (q[u].x > 1) x[u] += v[u][1];
        if (q[u].x > 2) x[u] += v[u][2];
        if (q[u].x > 3) rest |= 1u << u;
    }
}

// an element with more than four sources: the fifth on
__device__ __forceinline__ double mf_gather_rest(const MfArgs &a, int list, double x)
{
    for (int n = a.ext[list].x - 3, t = list + 1; n > 0; n -= 8, t += 2) {
        int4 r[2];
        double v[8];
        r[0] = a.ext[t];
        r[1] = n > 4 ? a.ext[t + 1] : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            v[4 * h] = n > 4 * h ? mf_source(a, r[h].x) : 0.0;
            v[4 * h + 1] = n > 4 * h + 1 ? mf_source(a, r[h].y) : 0.0;
            v[4 * h + 2] = n > 4 * h + 2 ? mf_source(a, r[h].z) : 0.0;
            v[4 * h + 3] = n > 4 * h + 3 ? mf_source(a, r[h].w) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (n > u) x += v[u];
    }
    return x;
}

// a small front's elements, a lane's share
constexpr int kMfSmallEl = (kMfSmall * (kMfSmall + 1) + 31) / 32;
__device__ __forceinline__ void mf_small_el(const MfArgs &a, const MfFront &fr, int2 (&e)[kMfSmallEl], int lane)
{
    const int n = fr.f * (fr.f + 1);
#pragma unroll
    for (int u = 0; u < kMfSmallEl; ++u)
        e[u] = lane + 32 * u < n ? a.el[fr.s0 + lane + 32 * u] : make_int2(kMfNone, -1);
}

// One small front by one warp, in its shared memory S
__device__ __forceinline__ void mf_small_front(const MfArgs &a, const MfFront &fr, const int2 (&e)[kMfSmallEl], double *S,
                                               int lane)
{
    const int p = fr.p, f = fr.f, ld = (f + 1) | 1, r = f - p;
    {
        double x[kMfSmallEl];
        uint32_t rest;
        mf_gather(a, e, x, rest);
#pragma unroll
        for (int u = 0; u < kMfSmallEl; ++u)
            if (rest >> u & 1) x[u] = mf_gather_rest(a, e[u].y, x[u]);
        const float rw = 1.0f / (float)(f + 1);
#pragma unroll
        for (int u = 0; u < kMfSmallEl; ++u) {
            const int t = lane + 32 * u, i = fast_div(t, rw);
            if (i < f) S[i * ld + (t - i * (f + 1))] = x[u];
        }
    }
    __syncwarp();
    for (int k = 0; k < p; ++k) {
        const double dk = S[k * ld + k], inv = fast_rcp(dk);
        if (k + 1 + lane <= f) S[k * ld + k + 1 + lane] *= inv;
        if (lane == 31) pivot_check(a, dk);
        __syncwarp();
        const int w = f - k, m = f - k - 1;   // columns k + 1 .. f, rows k + 1 .. f - 1
        const float rw = 1.0f / (float)w;
        const double *Sk = S + k * ld + k + 1;
        double *Sb = S + (k + 1) * ld + k;
        for (int t = lane; t < m * w; t += 32) {
            const int i = fast_div(t, rw), j = t - i * w;
            Sb[i * ld + 1 + j] = fma(-Sb[i * ld], Sk[j], Sb[i * ld + 1 + j]);
        }
        __syncwarp();
    }
    // the pivot rows and y, then the update
    double *U = a.U + fr.u0;
    {
        const float rf = 1.0f / (float)f;
        for (int t = lane; t < p * f; t += 32) {
            const int i = fast_div(t, rf), j = t - i * f;
            U[t] = S[i * ld + j];
        }
    }
    if (lane < p) U[p * f + lane] = S[lane * ld + f];
    {
        const float rr = 1.0f / (float)(r + 1);
        for (int t = lane; t < r * (r + 1); t += 32) {
            const int i = fast_div(t, rr), j = t - i * (r + 1);
            a.cb[fr.c0 + t] = S[(p + i) * ld + p + j];
        }
    }
    __syncwarp();   // S is read before the next front overwrites it
}

__global__ void __launch_bounds__(32 * kMfSmallWarps) k_mf_small(MfArgs a)
{
    mf_begin();
    extern __shared__ __align__(16) double msm[];
    const int lane = threadIdx.x & 31;
    double *S = msm + (size_t)(threadIdx.x >> 5) * (kMfSmall * kMfSmallLd);
    int *next = a.cnt + 2 * a.nf;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(next, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= a.nleaf[0]) break;
        MfFront fr = a.fr[a.leaf[0][t]];
        int2 e[kMfSmallEl];
        mf_small_el(a, fr, e, lane);
        for (;;) {
            // the parent's plan is in flight while this front is eliminated, in
            // case this warp is the last child to arrive and goes on with it
            const bool up = fr.parent_need > 0;   // 0: a root, or the parent is of another class
            const MfFront nx = a.fr[up ? fr.parent : 0];
            mf_small_front(a, fr, e, S, lane);
            if (!up) break;
            mf_small_el(a, nx, e, lane);
            int arrived = 0;
            if (lane == 0) {
                __threadfence();
                arrived = atomicAdd(a.cnt + fr.parent, 1);
                __threadfence();
            }
            arrived = __shfl_sync(0xffffffffu, arrived, 0);
            if (arrived + 1 != fr.parent_need) break;
            __syncwarp();   // lane 0's fence before every lane's reads of the other children's updates
            fr = nx;
        }
    }
}

// ---- fronts in registers ----
//
// A CTA's (NC = 1) or cluster's warps hold the front in registers: a warp holds a
// row, a column per lane and 32-column block, and the rows go round the warps
// (warp gw has rows gw, gw + NW, ...).  The warp that
// owns row k scales it by its pivot's reciprocal (so that U has a unit diagonal
// and the multipliers are the plain column: no other FP64 instruction is
// uniform) and puts it into slot k of every CTA's shared memory, where an
// mbarrier per slot announces it; every warp then takes row k out of its rows.
// No barrier joins the warps: the owner of row k + 1 updates that row first and
// sends it on while the others still work on row k, so a step costs the chain
// wait - multiply-add - reciprocal - scale - send or the FP64 time of the rows,
// whichever is longer.  Slots are not reused within a batch of rows; a batch
// ends with a barrier of all warps, writes its rows to U and starts afresh.
template <int NC>
struct MfGroup {
    uint64_t *bar;      // [rows] mbarriers
    double *row;        // [rows][32 C2] pivot rows
    int rank;           // this CTA in the cluster
    int gw;             // this warp among the group's
    bool dead;          // a wait ran out: no further waits
    bool lost;          // ... for a slot to be read out (this thread's)
    uint32_t rrow[NC], rbar[NC];   // row and bar in every CTA of a cluster

    __device__ __forceinline__ MfGroup(uint64_t *bar_, double *row_, int rank_, int gw_)
        : bar(bar_), row(row_), rank(rank_), gw(gw_), dead(false), lost(false)
    {
        if (NC > 1)
            for (int q = 0; q < NC; ++q) {
                const int to = (rank + 1 + q) % NC;   // the CTA that owns the next row first
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rrow[q]) : "r"(smem_addr(row)), "r"(to));
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar[q]) : "r"(smem_addr(bar)), "r"(to));
            }
    }

    __device__ __forceinline__ void sync() const
    {
        if (NC == 1) {
            __syncthreads();
        } else {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        }
    }
};

// the slots of rows k0 .. k1 - 1 ready to receive (every thread; ends with a
// barrier of the group)
template <int NC, int C2>
__device__ __forceinline__ void mf_slots(const MfGroup<NC> &g, int k0, int k1)
{
    for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) mbar_init(g.bar + (k - k0), 1);
    mbar_fence_init();
    if (NC > 1) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x)
            mbar_arrive_expect_tx(g.bar + (k - k0), 256u * (uint32_t)(C2 - k / 32));
    }
    g.sync();
}

// a column of a pivot row into slot `slot` of every CTA
template <int NC, int C2>
__device__ __forceinline__ void mf_send(const MfGroup<NC> &g, int slot, int col, double u)
{
    const uint32_t at = (uint32_t)slot * (32 * C2) + (uint32_t)col;
    if (NC == 1) {
        g.row[at] = u;
    } else {
#pragma unroll
        for (int q = 0; q < NC; ++q)
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(
                             g.rrow[q] + 8 * at),
                         "d"(u), "r"(g.rbar[q] + 8 * (uint32_t)slot)
                         : "memory");
    }
}

// Every slot of rows k0 .. k1 - 1 complete in every CTA, before mf_rows_out (every
// thread; ends with a barrier of the group).  Across a cluster only a slot's own
// mbarrier tells that its row has arrived: the group's barrier does not order the
// asynchronous stores, and a warp without later rows has not waited for the slot in
// the elimination (a root's last row is waited for by none).  So the threads of each
// CTA look at a slot each; all but the last few have long arrived.
template <int NC>
__device__ __forceinline__ void mf_drain(const MfArgs &a, MfGroup<NC> &g, int k0, int k1)
{
    if (NC > 1)
        for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x)
            if (!g.lost) g.lost = !mf_wait_slot(a, g.bar + (k - k0));
    g.sync();
}

// rows k0 .. k1 - 1 of the batch from their slots (drained) to U and y (the CTAs of a
// group in turn, a warp per row), and the end of their mbarriers
template <int NC, int C2>
__device__ __forceinline__ void mf_rows_out(const MfArgs &a, const MfFront &fr, const MfGroup<NC> &g, int k0, int k1)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, f = fr.f;
    double *U = a.U + fr.u0;
    for (int k = k0 + wid * NC + g.rank; k < k1; k += nw * NC) {
        const double *rw = g.row + (size_t)(k - k0) * (32 * C2);
        for (int j = k + 1 + lane; j < f; j += 32) U[(size_t)k * f + j] = rw[j];
        if (lane == 0) U[(size_t)fr.p * f + k] = rw[f];
    }
    for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) mbar_inval(g.bar + (k - k0));   // as initialised
}

// a word of shared memory of every CTA of the group (one thread)
template <int NC>
__device__ __forceinline__ void mf_tell(int *word, int value)
{
    if (NC == 1) {
        *(volatile int *)word = value;
    } else {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            uint32_t d;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(smem_addr(word)), "r"(q));
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(d), "r"(value) : "memory");
        }
    }
}

// row k (in mr; block C0, already free of rows 0 .. k - 1) scaled and sent by its warp
template <int NC, int C2, int C0>
__device__ __forceinline__ void mf_publish(const MfArgs &a, const MfGroup<NC> &g, const double (&mr)[C2], int k, int slot)
{
    const int lane = threadIdx.x & 31;
    const double d = __shfl_sync(0xffffffffu, mr[C0], k & 31);
    const double inv = fast_rcp(d);
#pragma unroll
    for (int c = C0; c < C2; ++c) mf_send<NC, C2>(g, slot, 32 * c + lane, mr[c] * inv);
    if (NC == 1) {
        __syncwarp();
        if (lane == 0) mbar_arrive(g.bar + slot);
    }
    if (lane == 0) pivot_check(a, d);
}

// row k (its columns from block C0 on in u) out of a row
template <int C2, int C0>
__device__ __forceinline__ void mf_take(double (&mr)[C2], const double (&u)[C2], int k)
{
    const double x = -__shfl_sync(0xffffffffu, mr[C0], k & 31);
#pragma unroll
    for (int c = C0; c < C2; ++c) mr[c] = fma(x, u[c], mr[c]);
}

// the pivots from K0 on: of one column block (the blocks before it are done, their
// registers are not touched any more) and of one row per warp, so that the
// registers of a pivot row are known when this is compiled
template <int NC, int NW, int R, int C2, int K0>
__device__ __forceinline__ void mf_pivots(const MfArgs &a, const MfFront &fr, MfGroup<NC> &g, int rows, int &kb,
                                          double (&m)[R][C2])
{
    constexpr int N = NW < 32 ? NW : 32, C0 = K0 / 32, Q = K0 / NW;
    constexpr bool same = (K0 + N) % 32 != 0;   // the next pivots are of the same block
    const int p = fr.p, gw = g.gw, lane = threadIdx.x & 31;
    const int last = gw < fr.f ? gw + (fr.f - 1 - gw) / NW * NW : -1;   // this warp's last row
    const int k1 = min(p, K0 + N);
    for (int k = K0; k < k1; ++k) {
        if (k == kb + rows) {   // the batch's slots are used up
            mf_drain(a, g, kb, k);
            mf_rows_out<NC, C2>(a, fr, g, kb, k);
            g.sync();
            kb = k;
            mf_slots<NC, C2>(g, kb, min(p, kb + rows));
        }
        const int slot = k - kb;
        // a row that its owner could not send ahead: the first of a batch or block
        if ((slot == 0 || k == 32 * C0) && k % NW == gw) mf_publish<NC, C2, C0>(a, g, m[Q], k, slot);
        if (last <= k) continue;   // no rows left
        if (!g.dead) g.dead = !__all_sync(0xffffffffu, mf_wait_slot(a, g.bar + slot));
        double u[C2];
        const double *rw = g.row + (size_t)slot * (32 * C2) + lane;
#pragma unroll
        for (int c = C0; c < C2; ++c) u[c] = rw[32 * c];
        // the next pivot row first, and on its way at once
        const int kn = k + 1;
        const bool mine = kn < p && kn < kb + rows && kn % NW == gw;
        const bool here = mine && kn < K0 + N, next = mine && same && kn == K0 + N;
        if (here) {
            mf_take<C2, C0>(m[Q], u, k);
            mf_publish<NC, C2, C0>(a, g, m[Q], kn, slot + 1);
        }
        if constexpr (Q + 1 < R)
            if (next) {
                mf_take<C2, C0>(m[Q + 1], u, k);
                mf_publish<NC, C2, C0>(a, g, m[Q + 1], kn, slot + 1);
            }
#pragma unroll
        for (int q = Q; q < R; ++q) {
            const int i = gw + NW * q;
            if (!(q == Q && here) && !(q == Q + 1 && next) && i <= last && i > k) mf_take<C2, C0>(m[q], u, k);
        }
    }
    if constexpr ((K0 + N) / 32 < C2 && (K0 + N) / NW < R)
        if (p > K0 + N) mf_pivots<NC, NW, R, C2, K0 + N>(a, fr, g, rows, kb, m);
}

// the plan of the thread's elements of a front
template <int NW, int R, int C2>
__device__ __forceinline__ void mf_plan(const MfArgs &a, const MfFront &fr, int gw, int2 *e)
{
    const int f = fr.f, w = f + 1, lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
        for (int c = 0; c < C2; ++c) {
            const int i = gw + NW * q, j = 32 * c + lane;
            e[q * C2 + c] = i < f && j < w ? a.el[fr.s0 + i * w + j] : make_int2(kMfNone, -1);
        }
}

// a front from its plan e to its update and pivot rows; `nx`, with which the group
// may go on, is loaded on the way
template <int NC, int NW, int R, int C2>
__device__ __forceinline__ void mf_tile_front(const MfArgs &a, const MfFront &fr, MfGroup<NC> &g, int rows,
                                              const int2 *e, MfFront &nx)
{
    const int p = fr.p, f = fr.f, r = f - p;
    const int lane = threadIdx.x & 31, gw = g.gw;
    // ---- the front's elements: their sources, a few at a time, while the slots
    // are made ready ----
    mf_slots<NC, C2>(g, 0, min(p, rows));
    double m[R][C2];
    constexpr int G = R * C2 % 4 == 0 ? 4 : R * C2 % 3 == 0 ? 3 : 2;   // elements at a time
    static_assert(R * C2 % G == 0);
    uint32_t rest = 0;
#pragma unroll
    for (int t = 0; t < R * C2; t += G) {
        int2 es[G];
        double x[G];
        uint32_t more;
#pragma unroll
        for (int u = 0; u < G; ++u) es[u] = e[t + u];
        mf_gather(a, es, x, more);
        rest |= more << t;
#pragma unroll
        for (int u = 0; u < G; ++u) m[(t + u) / C2][(t + u) % C2] = x[u];
    }
    if (rest)
#pragma unroll
        for (int t = 0; t < R * C2; ++t)
            if (rest >> t & 1) m[t / C2][t % C2] = mf_gather_rest(a, e[t].y, m[t / C2][t % C2]);
    int kb = 0;   // first row of the batch
    mf_pivots<NC, NW, R, C2, 0>(a, fr, g, rows, kb, m);
    if (fr.parent_need > 0) nx = a.fr[fr.parent];
    // ---- the update ----
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int i = gw + NW * q;
        if (i >= p && i < f) {
            double *cb = a.cb + fr.c0 + (size_t)(i - p) * (r + 1) - p;
#pragma unroll
            for (int c = 0; c < C2; ++c) {
                const int j = 32 * c + lane;
                if (j >= p && j <= f) cb[j] = m[q][c];
            }
        }
    }
    mf_drain(a, g, kb, p);
    mf_rows_out<NC, C2>(a, fr, g, kb, p);
}

// after a group's front: whether it goes on with the parent (its last child to
// arrive does).  Every thread; contains barriers of the group.
template <int NC>
__device__ __forceinline__ bool mf_climb(const MfArgs &a, const MfFront &fr, const MfGroup<NC> &g, int *s_next)
{
    g.sync();   // the group's writes, before its arrival
    if (g.rank == 0 && threadIdx.x == 0) {
        __threadfence();
        const int go = atomicAdd(a.cnt + fr.parent, 1) + 1 == fr.parent_need;
        __threadfence();
        mf_tell<NC>(s_next, go);
    }
    g.sync();
    return *(volatile int *)s_next != 0;
}

// the next front of the group's class without children there (-1: none left)
template <int NC>
__device__ __forceinline__ int mf_next(const MfArgs &a, int cls, const MfGroup<NC> &g, int *s_next)
{
    g.sync();
    if (g.rank == 0 && threadIdx.x == 0) mf_tell<NC>(s_next, atomicAdd(a.cnt + 2 * a.nf + cls, 1));
    g.sync();
    const int t = *(volatile int *)s_next;
    return t < a.nleaf[cls] ? a.leaf[cls][t] : -1;
}

__global__ void __launch_bounds__(32 * kMfMidWarps, 2) k_mf_mid(MfArgs a)
{
    mf_begin();
    __shared__ __align__(16) double row[kMfMidRows * 64];
    __shared__ uint64_t bar[kMfMidRows];
    __shared__ int s_next;
    MfGroup<1> g(bar, row, 0, (int)threadIdx.x >> 5);
    for (int s; (s = mf_next(a, 1, g, &s_next)) >= 0;) {
        MfFront fr = a.fr[s], nx = fr;
        // a front's plan; the parent's is in flight while this CTA counts itself there
        // (k_mf_mid 90 -> 85 us at 2,000 buses, 108 -> 101 at 10,000)
        int2 e[16];
        auto plan = [&](const MfFront &x) {
            if (x.f < 32)
                mf_plan<kMfMidWarps, 4, 1>(a, x, g.gw, e);
            else
                mf_plan<kMfMidWarps, 8, 2>(a, x, g.gw, e);
        };
        plan(fr);
        for (;;) {
            if (fr.f < 32)
                mf_tile_front<1, kMfMidWarps, 4, 1>(a, fr, g, kMfMidRows, e, nx);
            else
                mf_tile_front<1, kMfMidWarps, 8, 2>(a, fr, g, kMfMidRows, e, nx);
            if (fr.parent_need == 0) break;
            plan(nx);
            if (!mf_climb(a, fr, g, &s_next)) break;
            fr = nx;
        }
    }
}

template <int R, int C2>
__device__ __forceinline__ void mf_wide_front(const MfArgs &a, const MfFront &fr, MfGroup<kMfWideCtas> &g)
{
    constexpr int NW = kMfWideWarps * kMfWideCtas;
    int2 e[R * C2];
    MfFront nx;
    mf_plan<NW, R, C2>(a, fr, g.gw, e);
    mf_tile_front<kMfWideCtas, NW, R, C2>(a, fr, g, (int)(kMfWideRowBytes / (256 * C2)), e, nx);
}

__global__ void __cluster_dims__(kMfWideCtas, 1, 1) __launch_bounds__(32 * kMfWideWarps, 1) k_mf_wide(MfArgs a)
{
    mf_begin();
    extern __shared__ __align__(16) double msm[];
    __shared__ int s_next;
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    // consecutive rows on different SMs
    MfGroup<kMfWideCtas> g(reinterpret_cast<uint64_t *>(msm), msm + (kMfWide + 1), (int)rank,
                           ((int)threadIdx.x >> 5) * kMfWideCtas + (int)rank);
    for (int s; (s = mf_next(a, 2, g, &s_next)) >= 0;)
        for (;;) {
            const MfFront fr = a.fr[s];
            // the owner's chain takes and scales every column block it is compiled
            // for: with 4 blocks for all fronts below 128 unknowns this kernel took
            // 140 us at 10,000 buses and 316 at 25,000, with 2, 3 and 4 (and rows sent
            // to the next row's CTA first) 105 and 279
            if (fr.f < 64)
                mf_wide_front<1, 2>(a, fr, g);
            else if (fr.f < 96)
                mf_wide_front<2, 3>(a, fr, g);
            else if (fr.f < 128)
                mf_wide_front<2, 4>(a, fr, g);
            else if (fr.f < 192)
                mf_wide_front<3, 6>(a, fr, g);
            else
                mf_wide_front<4, 8>(a, fr, g);
            if (fr.parent_need == 0 || !mf_climb(a, fr, g, &s_next)) break;
            s = fr.parent;
        }
    g.sync();   // every CTA has drained its slots (mf_drain): none is sent to any more
}

// One front by a cluster in global memory M, in panels of kMfHugeB pivots:
//   * every CTA factors the panel's diagonal block for itself, in shared memory (no
//     barrier of the cluster),
//   * its pivot rows U and columns L beyond the block, a thread per column or row
//     of the front (each needs the block only), dealt out over the cluster,
//   * the rest less L U, in tiles dealt out over the cluster.
// Every element takes its terms in the order of the pivots, each by one FMA: the
// result does not depend on the panels.
// Bound by the cluster's FP64 pipes (at the 528 G multiply-adds a second of all
// SMs, 49 of the 51 ms of 1,598 unknowns) and, at a few hundred unknowns, by the panels' serial steps.
// One CTA a front, a pivot at a time over all of it, waited for L2 instead.  A solve,
// ms: complete graphs of 278 / 598 / 1,598 unknowns 4.9 / 47 / 845 -> 1.2 / 4.8 / 51,
// square meshes of 100 x 100 / 150 x 150 buses (fronts of 304 / 510 unknowns) 16 / 122
// -> 3.6 / 14.6 (a left-looking factorization by columns: 13 / 59).
constexpr int kMfHugeB = 32, kMfHugeT = 64;
constexpr int kMfHugeLd = kMfHugeB + 1;

struct MfHugeSmem {
    double D[kMfHugeB * kMfHugeLd];    // diagonal block: L, strict upper U
    double inv[kMfHugeB];              // reciprocals of its pivots
    double L[kMfHugeT * kMfHugeLd];    // a tile's L and U
    double U[kMfHugeB * kMfHugeT];
};

__device__ __forceinline__ void mf_huge_front(const MfArgs &a, const MfFront &fr, double *M,
                                              const MfGroup<kMfHugeCtas> &g, MfHugeSmem &sm)
{
    constexpr int TB = kMfHugeThreads, B = kMfHugeB, T = kMfHugeT, NW = TB / 32 * kMfHugeCtas;
    const int p = fr.p, f = fr.f, r = f - p;
    const size_t ld = (size_t)((f + 1) | 1);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, gt = g.rank * TB + tid;
    for (int t = gt; t < f * (f + 1); t += kMfHugeCtas * TB) {
        const int2 e[1] = {a.el[fr.s0 + t]};
        double x[1];
        uint32_t rest;
        mf_gather(a, e, x, rest);
        if (rest) x[0] = mf_gather_rest(a, e[0].y, x[0]);
        M[(size_t)(t / (f + 1)) * ld + t % (f + 1)] = x[0];
    }
    g.sync();
    double *U = a.U + fr.u0;
    for (int k0 = 0; k0 < p; k0 += B) {
        const int nb = min(B, p - k0), k1 = k0 + nb;
        // ---- the diagonal block (an identity where the last panel is short) ----
        for (int t = tid; t < B * B; t += TB) {
            const int i = t / B, j = t % B;
            sm.D[i * kMfHugeLd + j] =
                i < nb && j < nb ? __ldcg(M + (size_t)(k0 + i) * ld + k0 + j) : (i == j ? 1.0 : 0.0);
        }
        if (tid >= nb && tid < B) sm.inv[tid] = 1.0;
        __syncthreads();
        for (int k = 0; k < nb; ++k) {
            if (wid == 0) {
                const double d = sm.D[k * kMfHugeLd + k], inv = fast_rcp(d);
                if (lane > k) sm.D[k * kMfHugeLd + lane] *= inv;
                if (lane == 0) {
                    sm.inv[k] = inv;
                    if (g.rank == 0) pivot_check(a, d);
                }
            }
            __syncthreads();
            for (int i = k + 1 + wid; i < nb; i += TB / 32) {
                double *Di = sm.D + i * kMfHugeLd;
                if (lane > k) Di[lane] = fma(-Di[k], sm.D[k * kMfHugeLd + lane], Di[lane]);
            }
            __syncthreads();
        }
        if (g.rank == 0)
            for (int t = tid; t < B * B; t += TB) {
                const int i = t / B, j = t % B;
                if (i < j && j < nb) U[(size_t)(k0 + i) * f + k0 + j] = sm.D[i * kMfHugeLd + j];
            }
        // ---- columns k1 .. f of its rows, rows k1 .. f - 1 of its columns ----
        const int nc = f + 1 - k1, items = nc + f - k1;
        for (int t = gt; t < items; t += kMfHugeCtas * TB) {
            double x[B];
            if (t < nc) {
                const int j = k1 + t;
                double *Mj = M + (size_t)k0 * ld + j;
#pragma unroll
                for (int k = 0; k < B; ++k) x[k] = k < nb ? __ldcg(Mj + k * ld) : 0.0;
#pragma unroll
                for (int k = 0; k < B; ++k) {
#pragma unroll
                    for (int m = 0; m < k; ++m) x[k] = fma(-sm.D[k * kMfHugeLd + m], x[m], x[k]);
                    x[k] *= sm.inv[k];
                }
#pragma unroll
                for (int k = 0; k < B; ++k)
                    if (k < nb) {
                        Mj[k * ld] = x[k];
                        U[j < f ? (size_t)(k0 + k) * f + j : (size_t)p * f + k0 + k] = x[k];
                    }
            } else {
                double *Mi = M + (size_t)(k1 + t - nc) * ld + k0;
#pragma unroll
                for (int k = 0; k < B; ++k) x[k] = k < nb ? __ldcg(Mi + k) : 0.0;
#pragma unroll
                for (int k = 0; k < B; ++k)
#pragma unroll
                    for (int m = 0; m < k; ++m) x[k] = fma(-x[m], sm.D[m * kMfHugeLd + k], x[k]);
#pragma unroll
                for (int k = 0; k < B; ++k)
                    if (k < nb) Mi[k] = x[k];
            }
        }
        g.sync();
        // ---- the rest, a warp 4 rows of a tile, a lane 2 columns of it ----
        const int nr = f - k1, tr = (nr + T - 1) / T, tc = (nc + T - 1) / T;
        for (int t = g.rank; t < tr * tc; t += kMfHugeCtas) {
            const int i0 = k1 + t / tc * T, j0 = k1 + t % tc * T;
            double c[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int i = i0 + 4 * wid + u, j = j0 + lane + 32 * v;
                    c[u][v] = i < f && j <= f ? __ldcg(M + (size_t)i * ld + j) : 0.0;
                }
            for (int x = tid; x < T * B; x += TB) {
                const int i = i0 + x / B, j = j0 + x % T;
                sm.L[x / B * kMfHugeLd + x % B] = i < f && x % B < nb ? __ldcg(M + (size_t)i * ld + k0 + x % B) : 0.0;
                sm.U[x] = j <= f && x / T < nb ? __ldcg(M + (size_t)(k0 + x / T) * ld + j) : 0.0;
            }
            __syncthreads();
            for (int k = 0; k < nb; ++k)
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v)
                        c[u][v] = fma(-sm.L[(4 * wid + u) * kMfHugeLd + k], sm.U[k * T + lane + 32 * v], c[u][v]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int i = i0 + 4 * wid + u, j = j0 + lane + 32 * v;
                    if (i < f && j <= f) M[(size_t)i * ld + j] = c[u][v];
                }
            __syncthreads();
        }
        g.sync();
    }
    for (int i = wid * kMfHugeCtas + g.rank; i < r; i += NW)
        for (int j = lane; j <= r; j += 32)
            a.cb[fr.c0 + (size_t)i * (r + 1) + j] = __ldcg(M + (size_t)(p + i) * ld + p + j);
}

__global__ void __cluster_dims__(kMfHugeCtas, 1, 1) __launch_bounds__(kMfHugeThreads, 1) k_mf_huge(MfArgs a)
{
    mf_begin();
    __shared__ MfHugeSmem sm;
    __shared__ int s_next;
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const MfGroup<kMfHugeCtas> g(reinterpret_cast<uint64_t *>(sm.inv), sm.D, (int)rank, 0);   // its barrier alone is used
    for (int s; (s = mf_next(a, 3, g, &s_next)) >= 0;)
        for (;;) {
            const MfFront fr = a.fr[s];
            mf_huge_front(a, fr, a.mat + fr.m0, g, sm);
            if (fr.parent_need == 0 || !mf_climb(a, fr, g, &s_next)) break;
            s = fr.parent;
        }
}

// ------------------------------------------------------ backward solve ----

// The other fronts: x_p of the fronts of one path, from its head down, by one CTA.
// t = y - U_pr x_r (a thread per row and quarter of the border), then U_pp x_p = t
// (unit diagonal) from the bottom in blocks of 32 rows: a block's triangle by one
// warp (a lane per row), its terms out of the rows above by a thread per row.
// The chain from front to front is what counts: a front's x stays in shared memory,
// where the next front of the path finds its border (a child's border is among its
// parent's pivots and border), and that front's pivot rows are copied there while
// the triangle is solved, by the other warps (before the wait, for a path's head).
// The border's products by a warp per row, each with a shuffle tree of 5 additions
// (FP64 instructions like the products), and every load behind the front before
// took 65 us at 10,000 buses and 192 at 70,000; so 44 and 138 (the small fronts, by
// the same means, 24 -> 20 and 38 -> 32).
__global__ void __launch_bounds__(kMfBackThreads) k_mf_back_big(MfArgs a)
{
    mf_begin();
    extern __shared__ __align__(16) double msm[];
    __shared__ int s_next, s_ok;
    // x of the front (pivots, border) and of the one before; partial sums; pivot rows and y
    double *const sp = msm + 2 * a.backmax, *const Wm = sp + 4 * a.backp;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int TB = kMfBackThreads, nw = TB / 32;
    int *next = a.cnt + 2 * a.nf + kMfClasses + 1, *done = a.cnt + a.nf;
    auto room = [](const MfFront &f) { return f.p * (f.f | 1) + f.p; };   // doubles of its copy
    auto stage = [&](const MfFront &f, double *W, int w0, int w1) {   // by warps w0 .. w1 - 1
        const int ld = f.f | 1;
        const double *U = a.U + f.u0;
        for (int i = wid - w0; i < f.p; i += w1 - w0)
            for (int j = i + 1 + lane; j < f.f; j += 32) cp_async8(W + i * ld + j, U + (size_t)i * f.f + j);
        for (int i = tid - 32 * w0; i < f.p; i += 32 * (w1 - w0)) cp_async8(W + f.p * ld + i, U + (size_t)f.p * f.f + i);
    };
    for (;;) {
        if (tid == 0) s_next = atomicAdd(next, 1);
        __syncthreads();
        const int t = s_next;
        __syncthreads();
        if (t >= a.npath[1]) break;
        int s = a.path[1][t], cur = 0;
        MfFront fr = a.fr[s];
        bool head = true, staged = false;   // staged: its copy was begun with the front before
        double *W = Wm;
        int rl = 0;   // the place of the thread's first border unknown
        for (;;) {
            const int p = fr.p, f = fr.f, r = f - p, own = room(fr);
            const bool in = own <= a.backw;
            if (!staged) {
                W = Wm;
                if (in) stage(fr, W, 0, nw);
            }
            // the next front, of which nothing is used before this one's border products
            const MfFront nx = a.fr[fr.heavy >= 0 ? fr.heavy : s];
            double *X = msm + cur * a.backmax;
            const double *Xp = msm + (cur ^ 1) * a.backmax;
            if (head) {
                const int bj = tid < r ? a.bidx[fr.b0 + tid] : 0;
                if (fr.wait) {
                    if (tid == 0) s_ok = mf_wait(a, done + fr.parent);
                    __syncthreads();
                    if (!s_ok) {
                        cp_async_wait_all();
                        return;
                    }
                }
                for (int j = tid; j < r; j += TB) X[p + j] = __ldcg(a.x + (j == tid ? bj : a.bidx[fr.b0 + j]));
            } else {
                for (int j = tid; j < r; j += TB) X[p + j] = Xp[j == tid ? rl : a.rel[fr.b0 + j]];
            }
            cp_async_wait_all();
            __syncthreads();
            const double *T = in ? W : a.U + fr.u0;
            const int ld = in ? f | 1 : f;
            for (int u = wid; u < (p + 31) / 32 * 4; u += nw) {
                const int i = (u >> 2) * 32 + lane;
                double sum = 0.0;
                if (i < p)
#pragma unroll 4
                    for (int j = u & 3; j < r; j += 4) sum = fma(T[(size_t)i * ld + p + j], X[p + j], sum);
                sp[32 * u + lane] = sum;
            }
            __syncthreads();
            // the next front's copy at the other end of the room, if both fit
            const bool ahead = fr.heavy >= 0 && own + room(nx) <= a.backw;
            double *const Wn = W == Wm ? Wm + (a.backw - room(nx)) : Wm;
            if (ahead && wid > 0) stage(nx, Wn, 1, nw);
            rl = fr.heavy >= 0 && tid < nx.f - nx.p ? a.rel[nx.b0 + tid] : 0;
            for (int i = tid; i < p; i += TB) {
                const double *q = sp + 128 * (i >> 5) + (i & 31);
                X[i] = T[(size_t)p * ld + i] - ((q[0] + q[32]) + (q[64] + q[96]));
            }
            __syncthreads();
            for (int b1 = p; b1 > 0; b1 -= 32) {
                const int b0 = b1 > 32 ? b1 - 32 : 0, w = b1 - b0;
                if (wid == 0) {
                    const double *Ti = T + (size_t)(b0 + min(lane, w - 1)) * ld + b0;
                    double x = lane < w ? X[b0 + lane] : 0.0;
#pragma unroll 4
                    for (int k = w - 1; k > 0; --k) {
                        const double uk = lane < k ? Ti[k] : 0.0;
                        const double xk = __shfl_sync(0xffffffffu, x, k);
                        if (lane < k) x = fma(-uk, xk, x);
                    }
                    if (lane < w) {
                        X[b0 + lane] = x;
                        a.x[fr.e0 + b0 + lane] = x;
                        a.dx[a.perm[fr.e0 + b0 + lane]] = x;
                    }
                }
                __syncthreads();
                if (b0 == 0) break;
                for (int i = tid; i < b0; i += TB) {
                    const double *Ti = T + (size_t)i * ld + b0;
                    double y = X[i];
#pragma unroll 4
                    for (int k = 0; k < w; ++k) y = fma(-Ti[k], X[b0 + k], y);
                    X[i] = y;
                }
                __syncthreads();
            }
            if (tid == 0 && fr.light) {   // someone waits for this front
                __threadfence();
                atomicExch(done + s, 1);
            }
            if (fr.heavy < 0) break;
            s = fr.heavy;
            fr = nx;
            cur ^= 1;
            head = false;
            staged = ahead;
            if (ahead) W = Wn;
        }
    }
}

// Small fronts: the same by one warp; the lanes are (row, part) pairs that split
// the row's border terms, joined by a shuffle tree.  The path's next front is
// loaded while this one is solved, its border's x come from this one's lanes.
__global__ void __launch_bounds__(32 * kMfSmallWarps) k_mf_back_small(MfArgs a)
{
    mf_begin();
    extern __shared__ __align__(16) double msm[];
    const int lane = threadIdx.x & 31;
    double *const Wm = msm + (size_t)(threadIdx.x >> 5) * (2 * kMfBackSmall);   // pivot rows and y of two fronts
    int *next = a.cnt + 2 * a.nf + kMfClasses, *done = a.cnt + a.nf;
    auto stage = [&](const MfFront &f, double *W) {
        for (int q = lane; q < f.p * f.f + f.p; q += 32) cp_async8(W + q, a.U + f.u0 + q);
    };
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(next, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= a.npath[0]) break;
        int s = a.path[0][t];
        MfFront fr = a.fr[s];
        double *W = Wm;
        stage(fr, W);
        const int bj = lane < fr.f - fr.p ? a.bidx[fr.b0 + lane] : 0;
        int pm = lane < fr.p ? a.perm[fr.e0 + lane] : 0;
        // the head of a path waits for its parent unless an earlier launch wrote it
        if (fr.wait && !__all_sync(0xffffffffu, mf_wait(a, done + fr.parent))) {
            cp_async_wait_all();
            return;
        }
        __syncwarp();
        double xb = lane < fr.f - fr.p ? __ldcg(a.x + bj) : 0.0;
        for (;;) {
            const int p = fr.p, f = fr.f, r = f - p;
            const MfFront nx = a.fr[fr.heavy >= 0 ? fr.heavy : s];
            cp_async_wait_all();
            __syncwarp();
            // lane = row i + p2 * part g
            const int p2 = p <= 1 ? 1 : 1 << (32 - __clz(p - 1)), g = lane / p2, i = lane & (p2 - 1), ng = 32 / p2;
            double sum = 0.0;
            for (int j0 = 0; j0 < r; j0 += ng) {
                const int j = j0 + g;
                const double xj = __shfl_sync(0xffffffffu, xb, j & 31);
                if (j < r && i < p) sum = fma(W[i * f + p + j], xj, sum);
            }
            for (int off = p2; off < 32; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            double *const Wn = W == Wm ? Wm + kMfBackSmall : Wm;
            int rl = 0, pn = 0;
            if (fr.heavy >= 0) {
                stage(nx, Wn);
                rl = lane < nx.f - nx.p ? a.rel[nx.b0 + lane] : 0;
                pn = lane < nx.p ? a.perm[nx.e0 + lane] : 0;
            }
            double x = 0.0;
            if (i < p) x = W[p * f + i] - sum;
            for (int k = p - 1; k > 0; --k) {
                const double xk = __shfl_sync(0xffffffffu, x, k);
                if (i < k) x = fma(-W[i * f + k], xk, x);
            }
            if (lane < p) {
                a.x[fr.e0 + lane] = x;
                a.dx[pm] = x;
            }
            __syncwarp();
            if (lane == 0 && fr.light) {   // someone waits for this front
                __threadfence();
                atomicExch(done + s, 1);
            }
            if (fr.heavy < 0) break;
            // a border unknown of the next front is a pivot or border unknown of this one
            const double u = __shfl_sync(0xffffffffu, x, rl & 31), v = __shfl_sync(0xffffffffu, xb, (rl - p) & 31);
            xb = rl < p ? u : v;
            s = fr.heavy;
            fr = nx;
            pm = pn;
            W = Wn;
        }
    }
}

// ------------------------------------------------------------ analysis ----

// Minimum-degree order of an undirected graph (explicit elimination: the
// neighbours of each eliminated node become a clique; ties to the lowest node).
std::vector<int> min_degree_order(std::vector<std::vector<int>> adj)
{
    const int n = (int)adj.size();
    std::set<std::pair<int, int>> pq;
    for (int u = 0; u < n; ++u) pq.insert({(int)adj[u].size(), u});
    std::vector<char> gone(n, 0);
    std::vector<int> order;
    order.reserve(n);
    std::vector<int> merged;
    while (!pq.empty()) {
        const int u = pq.begin()->second;
        pq.erase(pq.begin());
        gone[u] = 1;
        order.push_back(u);
        const std::vector<int> nb = adj[u];   // sorted, live nodes only
        for (int v : nb) {
            pq.erase({(int)adj[v].size(), v});
            merged.clear();
            std::set_union(adj[v].begin(), adj[v].end(), nb.begin(), nb.end(), std::back_inserter(merged));
            adj[v].clear();
            for (int x : merged)
                if (x != v && x != u) adj[v].push_back(x);
            pq.insert({(int)adj[v].size(), v});
        }
        adj[u].clear();
        adj[u].shrink_to_fit();
    }
    return order;
}

// The fronts of an elimination tree on the buses: node j starts as a front of
// its own (pivots wt[j] unknowns, border bw[j] unknowns) and takes in a child
// k's front while that adds few zeros: none at all (the border of k is j and
// the border of j), or at most 40 % of the merged front's pivot rows and
// columns up to 16 unknowns (a level of the tree costs 2-3 us, more than the
// added arithmetic of a small front; 10,000 buses: 9,409 fronts on 29 levels ->
// 4,209 on 22), and 2 % above.
struct FrontTree {
    std::vector<int> top;                     // front -> its top node
    std::vector<std::vector<int>> members;    // front -> its nodes, ascending
    std::vector<int> parent;                  // front -> parent front (-1: a root)
};

FrontTree merge_fronts(const std::vector<int> &par, const std::vector<int> &wt, const std::vector<int> &bw)
{
    const int B = (int)par.size();
    std::vector<std::vector<int>> ch(B), mem(B);
    std::vector<int> p(wt), owner(B);
    std::vector<double> zeros(B, 0.0);
    for (int j = 0; j < B; ++j)
        if (par[j] >= 0) ch[par[j]].push_back(j);
    std::vector<char> gone(B, 0);
    for (int j = 0; j < B; ++j) {
        mem[j] = {j};
        for (;;) {
            int best = -1;
            double bz = 0.0;
            for (int k : ch[j]) {
                const double z = 2.0 * p[k] * (p[j] + bw[j] - bw[k]);
                if (best < 0 || z < bz) {
                    best = k;
                    bz = z;
                }
            }
            if (best < 0) break;
            const double fn = (double)p[best] + p[j] + bw[j], tot = fn * fn - (double)bw[j] * bw[j];
            const double z = bz + zeros[best] + zeros[j];
            if (bz > 0.0 && z > (fn <= 12.0 ? 0.4 : 0.02) * tot) break;
            zeros[j] = z;
            p[j] += p[best];
            gone[best] = 1;
            mem[j].insert(mem[j].end(), mem[best].begin(), mem[best].end());
            ch[j].erase(std::find(ch[j].begin(), ch[j].end(), best));
            ch[j].insert(ch[j].end(), ch[best].begin(), ch[best].end());
            std::vector<int>().swap(mem[best]);
            std::vector<int>().swap(ch[best]);
        }
    }
    // postorder of the fronts (children before parents, a subtree consecutive)
    FrontTree T;
    std::vector<int> id(B, -1), stack;
    std::vector<std::pair<int, size_t>> st;
    for (int j = 0; j < B; ++j) {
        if (gone[j] || par[j] >= 0) continue;   // a root's top node has no parent
        st.push_back({j, 0});
        while (!st.empty()) {
            auto &[u, c] = st.back();
            if (c < ch[u].size()) {
                const int v = ch[u][c++];
                st.push_back({v, 0});
                continue;
            }
            id[u] = (int)T.top.size();
            T.top.push_back(u);
            std::sort(mem[u].begin(), mem[u].end());
            T.members.push_back(std::move(mem[u]));
            st.pop_back();
        }
    }
    T.parent.assign(T.top.size(), -1);
    for (int u : T.top)
        for (int v : ch[u]) T.parent[id[v]] = id[u];
    return T;
}

// The class of every front: the smallest that its size allows, and its subtree's.
// The classes run one launch after the other, so a long chain of fronts that one
// class could take holds up the next class's other fronts: chains are cut where
// the model's time of all three launches is least (rough us of a front, fitted to
// timestamps of the kernels; 25,000 buses: the small fronts' launch ends after 27
// instead of 52 us and the next one's after 70 instead of 110).
void plan_classes(std::vector<MfFront> &fr)
{
    const int nf = (int)fr.size();
    std::vector<int> best(nf), cls(nf);
    std::vector<double> t[3], cost[3];
    for (auto &v : cost) v.resize(nf);
    for (int s = 0; s < nf; ++s) {
        const int p = fr[s].p, f = fr[s].f;
        cost[0][s] = 4.5 + 0.6 * p;
        cost[1][s] = f < 32 ? 3.2 + 0.4 * p : 7.0 + 0.8 * p;
        cost[2][s] = 6.0 + (f < 128 ? 0.7 : 1.0) * p;
    }
    double least = 1e300;
    for (double lim0 : {15.0, 25.0, 40.0, 1e9})
        for (double lim1 : {25.0, 40.0, 60.0, 90.0, 1e9}) {
            for (auto &v : t) v.assign(nf, 0.0);
            std::fill(cls.begin(), cls.end(), 0);
            double end[3] = {0.0, 0.0, 0.0}, work[3] = {0.0, 0.0, 0.0};
            for (int s = 0; s < nf; ++s) {   // t[c][s], cls[s]: so far from its children
                const int f = fr[s].f;
                int c = std::max(cls[s], f <= kMfSmall ? 0 : f <= kMfMid ? 1 : f <= kMfWide ? 2 : 3);
                if (c == 0 && t[0][s] + cost[0][s] > lim0) c = 1;
                if (c == 1 && t[1][s] + cost[1][s] > lim1) c = 2;
                cls[s] = c;
                const int k = std::min(c, 2);
                t[k][s] += cost[k][s];
                end[k] = std::max(end[k], t[k][s]);
                work[k] += cost[k][s];
                if (const int q = fr[s].parent; q >= 0) {
                    cls[q] = std::max(cls[q], c);
                    t[k][q] = std::max(t[k][q], t[k][s]);
                }
            }
            // at least the work over what runs at once (warps, CTAs, clusters), fitted with
            // the costs above to 148 SMs' worth and 18 clusters: with the part's 152 and 19 a
            // Newton step at 25,000 buses takes 534 us instead of 512
            const double total = std::max(end[0], work[0] / (148 * 16.0)) + std::max(end[1], work[1] / (148 * 2.0)) +
                                 std::max(end[2], work[2] / 18.0);
            if (total < least) {
                least = total;
                best = cls;
            }
        }
    for (int s = 0; s < nf; ++s) fr[s].cls = best[s];
}

}  // namespace

pf_status host_lu(int nb, int n, int npvpq, const std::vector<int> &colptr, const std::vector<int> &rowidx,
                  const std::vector<int> &fmap, HostLu &L)
{
    L = HostLu{};
    L.n = n;
    // bus graph of the unknowns' buses (every unknown's bus has a theta unknown)
    std::vector<int> node(nb, -1), bus_of;
    for (int k = 0; k < npvpq; ++k) {
        node[fmap[k]] = (int)bus_of.size();
        bus_of.push_back(fmap[k]);
    }
    const int B = (int)bus_of.size();
    std::vector<std::vector<int>> adj(B);
    for (int c = 0; c < n; ++c)
        for (int p = colptr[c]; p < colptr[c + 1]; ++p) {
            const int u = node[fmap[rowidx[p]]], v = node[fmap[c]];
            if (u < 0 || v < 0) return set_error(PF_EINVAL, "jac_reduced_solve: an unknown without a bus angle");
            if (u != v) {
                adj[u].push_back(v);
                adj[v].push_back(u);
            }
        }
    for (auto &a : adj) {
        std::sort(a.begin(), a.end());
        a.erase(std::unique(a.begin(), a.end()), a.end());
    }
    std::vector<int> tidx(nb, -1), vidx(nb, -1);
    for (int k = 0; k < npvpq; ++k) tidx[fmap[k]] = k;
    for (int k = npvpq; k < n; ++k) vidx[fmap[k]] = k;
    const std::vector<int> order = min_degree_order(adj);
    std::vector<int> pos(B);
    for (int i = 0; i < B; ++i) pos[order[i]] = i;
    // elimination tree of the ordered buses and the patterns of its columns, by
    // row subtrees (rows ascending: every column's come out ascending)
    std::vector<int> par(B, -1), flag(B, -1), wt(B), bw(B, 0);
    std::vector<std::vector<int>> col(B);
    for (int i = 0; i < B; ++i) {
        wt[i] = vidx[bus_of[order[i]]] >= 0 ? 2 : 1;
        flag[i] = i;
        for (int u : adj[order[i]]) {
            int k = pos[u];
            if (k > i) continue;
            while (k != -1 && flag[k] != i) {
                if (par[k] == -1) par[k] = i;
                col[k].push_back(i);
                flag[k] = i;
                k = par[k];
            }
        }
    }
    for (int i = 0; i < B; ++i)
        for (int x : col[i]) bw[i] += wt[x];
    FrontTree T = merge_fronts(par, wt, bw);
    const int nf = (int)T.top.size();
    // unknowns renumbered front by front
    L.perm.reserve(n);
    std::vector<int> first(B), front_of(B);   // a node's first unknown, its front
    L.fr.resize(nf);
    for (int s = 0; s < nf; ++s) {
        MfFront &f = L.fr[s];
        f.e0 = (int)L.perm.size();
        for (int i : T.members[s]) {
            first[i] = (int)L.perm.size();
            front_of[i] = s;
            const int b = bus_of[order[i]];
            L.perm.push_back(tidx[b]);
            if (vidx[b] >= 0) L.perm.push_back(vidx[b]);
        }
        f.p = (int)L.perm.size() - f.e0;
        f.parent = T.parent[s];
    }
    if ((int)L.perm.size() != n) return set_error(PF_EINVAL, "jac_reduced_solve: unknowns do not match buses");
    std::vector<int> iperm(n), sn(n);
    for (int i = 0; i < n; ++i) iperm[L.perm[i]] = i;
    // borders, update and pivot-row storage
    long long u0 = 0, c0 = 0, b0 = 0, s0 = 0;
    std::vector<int> tmp;
    for (int s = 0; s < nf; ++s) {
        MfFront &f = L.fr[s];
        for (int i = 0; i < f.p; ++i) sn[f.e0 + i] = s;
        tmp.clear();
        for (int x : col[T.top[s]])
            for (int w = 0; w < wt[x]; ++w) tmp.push_back(first[x] + w);
        std::sort(tmp.begin(), tmp.end());
        const int r = (int)tmp.size();
        f.f = f.p + r;
        f.b0 = (int)b0;
        f.u0 = (int)u0;
        f.c0 = (int)c0;
        f.s0 = (int)s0;
        L.bidx.insert(L.bidx.end(), tmp.begin(), tmp.end());
        b0 += r;
        u0 += (long long)f.p * f.f + f.p;
        c0 += (long long)r * (r + 1);
        s0 += (long long)f.f * (f.f + 1);
        if (u0 >= (1LL << 31) || c0 >= (1LL << 31) || s0 >= (1LL << 31) || f.f > 46000)
            return set_error(PF_EUNSUPPORTED, "jac_reduced_solve: factor too large");
    }
    L.nU = u0;
    L.nC = c0;
    // the place of unknown x in front s
    auto place = [&](int s, int x) {
        const MfFront &f = L.fr[s];
        if (x < f.e0 + f.p) return x - f.e0;
        const auto b = L.bidx.begin() + f.b0, e = b + (f.f - f.p);
        return f.p + (int)(std::lower_bound(b, e, x) - b);
    };
    // the place of every border unknown in the parent (both borders ascend)
    std::vector<int> &rel = L.rel;
    rel.assign(std::max<long long>(b0, 1), 0);
    std::vector<std::vector<int>> kids(nf);
    for (int s = 0; s < nf; ++s) {
        const MfFront &f = L.fr[s];
        if (f.parent < 0) continue;
        kids[f.parent].push_back(s);
        const MfFront &q = L.fr[f.parent];
        int at = 0;
        for (int j = 0; j < f.f - f.p; ++j) {
            const int x = L.bidx[f.b0 + j];
            if (x < q.e0 + q.p) {
                rel[f.b0 + j] = x - q.e0;
            } else {
                while (L.bidx[q.b0 + at] != x) ++at;
                rel[f.b0 + j] = q.p + at;
            }
        }
    }
    // the sources of every element, by counting: A's entries and F first, then
    // the children's updates in order
    const int nnzA = colptr[n];
    std::vector<int> aplace(nnzA);
    auto each = [&](auto &&take) {   // take(element, source)
        for (int p = 0; p < nnzA; ++p) take(aplace[p], ~p);
        for (int s = 0; s < nf; ++s) {
            const MfFront &f = L.fr[s];
            const int w = f.f + 1;
            for (int i = 0; i < f.p; ++i) take(f.s0 + i * w + f.f, ~(nnzA + L.perm[f.e0 + i]));
            for (int c : kids[s]) {
                const MfFront &q = L.fr[c];
                const int r = q.f - q.p, *rl = rel.data() + q.b0;
                for (int i = 0; i < r; ++i) {
                    const int row = f.s0 + rl[i] * w, cb = q.c0 + i * (r + 1);
                    for (int j = 0; j < r; ++j) take(row + rl[j], cb + j);
                    take(row + f.f, cb + r);
                }
            }
        }
    };
    for (int c = 0; c < n; ++c)
        for (int p = colptr[c]; p < colptr[c + 1]; ++p) {
            const int i = iperm[rowidx[p]], j = iperm[c], s = sn[std::min(i, j)];
            aplace[p] = L.fr[s].s0 + place(s, i) * (L.fr[s].f + 1) + place(s, j);
        }
    if (nnzA + n >= INT32_MAX / 2) return set_error(PF_EUNSUPPORTED, "jac_reduced_solve: system too large");
    L.el.assign(std::max<long long>(s0, 1), make_int2(kMfNone, -1));
    std::vector<int> more(std::max<long long>(s0, 1), -1);   // further sources of an element, then how many are placed
    each([&](int e, int) { more[e]++; });
    long long next = 0;
    for (long long e = 0; e < s0; ++e)
        if (more[e] > 0) {
            L.el[e].y = (int)next;
            next += 1 + more[e] / 4;
        }
    if (next >= INT32_MAX / 4) return set_error(PF_EUNSUPPORTED, "jac_reduced_solve: factor too large");
    L.ext.assign(std::max<long long>(next, 1), make_int4(0, 0, 0, 0));
    each([&](int e, int k) {
        if (L.el[e].x == kMfNone) {
            L.el[e].x = k;
            return;
        }
        int *rec = &L.ext[L.el[e].y].x;   // the count, then the sources
        rec[1 + rec[0]++] = k;
    });
    std::vector<int> need(nf, 0);
    std::vector<double> rem(nf, 0.0), down(nf, 0.0);
    plan_classes(L.fr);
    for (int s = 0; s < nf; ++s)
        for (int c : kids[s]) need[s] += L.fr[c].cls == L.fr[s].cls;
    // the longest remaining path to the root and down to a leaf, in rough us
    for (int s = nf - 1; s >= 0; --s) {
        const MfFront &f = L.fr[s];
        double fl = 0.0;
        for (int k = 0; k < f.p; ++k) fl += (double)(f.f - k) * (f.f - k);
        rem[s] = 3.0 + 0.2 * f.p + fl / 3500.0 + (f.parent >= 0 ? rem[f.parent] : 0.0);
    }
    for (int s = 0; s < nf; ++s) {
        down[s] += 1.0 + 0.05 * L.fr[s].p;
        if (L.fr[s].parent >= 0) down[L.fr[s].parent] = std::max(down[L.fr[s].parent], down[s]);
    }
    // backward paths: the small fronts with small subtrees a warp each, the others
    // a CTA each (a path goes on with the child that reaches furthest down among
    // those of its launch), and the order of the leaves and heads
    std::vector<char> cont(nf, 0), large(nf, 0);
    for (int s = 0; s < nf; ++s) {
        large[s] = L.fr[s].f > kMfSmall;
        for (int c : kids[s]) large[s] |= large[c];
    }
    for (int s = 0; s < nf; ++s) {
        MfFront &f = L.fr[s];
        f.parent_need = f.parent >= 0 && L.fr[f.parent].cls == f.cls ? need[f.parent] : 0;
        f.heavy = -1;
        for (int c : kids[s])
            if (large[c] == large[s] && (f.heavy < 0 || down[c] > down[f.heavy])) f.heavy = c;
        f.light = f.wait = 0;
        f.m0 = -1;
        if (f.heavy >= 0) cont[f.heavy] = 1;
        if (large[s]) L.bigp = std::max(L.bigp, f.p), L.backmax = std::max(L.backmax, f.f);
        if (need[s] == 0) L.leaf[f.cls].push_back(s);
    }
    for (int s = 0; s < nf; ++s) {
        MfFront &f = L.fr[s];
        if (cont[s]) continue;
        L.path[large[s]].push_back(s);
        if (f.parent >= 0 && large[f.parent] == large[s]) {
            f.wait = 1;
            L.fr[f.parent].light = 1;
        }
    }
    auto by = [](const std::vector<double> &key) {
        return [&key](int x, int y) { return key[x] > key[y]; };
    };
    for (auto &v : L.leaf) std::stable_sort(v.begin(), v.end(), by(rem));
    // (a parent reaches further down than its children: parents' paths come first)
    for (auto &v : L.path) std::stable_sort(v.begin(), v.end(), by(down));
    return PF_OK;
}

// doubles of the backward solve without its copies (k_mf_back_big): x of two fronts,
// four partial sums of every pivot row.  The limit on a front: about 4,690 unknowns,
// all of them pivots.
static long long back_fixed(const HostLu &L) { return 2LL * L.backmax + 4LL * ((L.bigp + 31) / 32 * 32); }

// doubles of the backward solve's copies: what a front and the next of its path
// take, as far as it fits
static int back_room(const HostLu &L)
{
    auto room = [](const MfFront &f) { return (long long)f.p * (f.f | 1) + f.p; };
    long long most = 0;
    for (int h : L.path[1])
        for (int s = h; s >= 0; s = L.fr[s].heavy)
            most = std::max(most, room(L.fr[s]) + (L.fr[s].heavy >= 0 ? room(L.fr[L.fr[s].heavy]) : 0));
    const long long left = (long long)(kMfMaxSmem / sizeof(double)) - back_fixed(L);
    return (int)std::max(0LL, std::min(most, left));
}

// Upload the plan of the grid's current bus types and size its workspace.
pf_status lu_prepare(Grid *g, cudaStream_t s)
{
    if (g->lu_ready) return PF_OK;
    HostLu L;
    if (pf_status st = host_lu(g->nb, g->red_n, g->red_npvpq, g->red_h_colptr, g->red_h_rowidx, g->red_h_fmap, L))
        return st;
    size_t nmat = 0;
    for (MfFront &f : L.fr)
        if (f.cls == 3) {
            f.m0 = (long long)nmat;
            nmat += (size_t)f.f * ((f.f + 1) | 1);
        }
    if (back_fixed(L) * (long long)sizeof(double) > (long long)kMfMaxSmem)
        return set_error(PF_EUNSUPPORTED, "jac_reduced_solve: a front of %d unknowns exceeds shared memory", L.backmax);
    const int nf = (int)L.fr.size();
    cudaError_t e = cudaSuccess;
    auto up = [&](auto **dst, const auto &v) -> cudaError_t {
        cudaError_t r = g->arena.alloc(dst, std::max<size_t>(v.size(), 1));
        if (r == cudaSuccess && !v.empty())
            r = cudaMemcpyAsync(*dst, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice, s);
        return r;
    };
    if ((e = up(&g->lu_fr, L.fr)) || (e = up(&g->lu_leaf[0], L.leaf[0])) || (e = up(&g->lu_leaf[1], L.leaf[1])) ||
        (e = up(&g->lu_leaf[2], L.leaf[2])) || (e = up(&g->lu_leaf[3], L.leaf[3])) || (e = up(&g->lu_path[0], L.path[0])) ||
        (e = up(&g->lu_path[1], L.path[1])) || (e = up(&g->lu_el, L.el)) || (e = up(&g->lu_ext, L.ext)) ||
        (e = up(&g->lu_bidx, L.bidx)) || (e = up(&g->lu_rel, L.rel)) || (e = up(&g->lu_perm, L.perm)) ||
        (e = g->arena.alloc(&g->lu_U, (size_t)std::max<long long>(L.nU, 1))) ||
        (e = g->arena.alloc(&g->lu_cb, (size_t)std::max<long long>(L.nC, 1))) ||
        (e = g->arena.alloc(&g->lu_x, (size_t)std::max(L.n, 1))) ||
        (e = g->arena.alloc(&g->lu_mat, std::max<size_t>(nmat, 1))) ||
        (e = g->arena.alloc(&g->lu_cnt, 2 * (size_t)nf + kMfClasses + 2)) || (e = cudaStreamSynchronize(s))) {
        lu_release(g);
        return cuda_error(e, "jac_reduced_solve: set-up");
    }
    g->lu_n = L.n;
    g->lu_nf = nf;
    for (int c = 0; c < kMfClasses; ++c) g->lu_nleaf[c] = (int)L.leaf[c].size();
    for (int c = 0; c < 2; ++c) g->lu_npath[c] = (int)L.path[c].size();
    g->lu_backmax = L.backmax;
    g->lu_backp = (L.bigp + 31) / 32 * 32;
    g->lu_backw = back_room(L);
    g->lu_ready = 1;
    return PF_OK;
}

void lu_release(Grid *g)
{
    for (void *p : {(void *)g->lu_fr, (void *)g->lu_leaf[0], (void *)g->lu_leaf[1], (void *)g->lu_leaf[2], (void *)g->lu_leaf[3],
                    (void *)g->lu_path[0], (void *)g->lu_path[1], (void *)g->lu_el, (void *)g->lu_ext,
                    (void *)g->lu_bidx, (void *)g->lu_rel, (void *)g->lu_perm, (void *)g->lu_U, (void *)g->lu_cb, (void *)g->lu_x,
                    (void *)g->lu_mat, (void *)g->lu_cnt})
        g->arena.release(p);
    g->lu_fr = nullptr;
    for (int *&p : g->lu_leaf) p = nullptr;
    for (int *&p : g->lu_path) p = nullptr;
    g->lu_el = nullptr;
    g->lu_ext = nullptr;
    g->lu_bidx = g->lu_rel = g->lu_perm = g->lu_cnt = nullptr;
    g->lu_U = g->lu_cb = g->lu_x = g->lu_mat = nullptr;
    g->lu_ready = 0;
}

cudaError_t launch_lu_solve(Grid *g, const double *Jr, const double *F, double *dx, cudaStream_t s)
{
    if (g->lu_n == 0) return cudaSuccess;
    MfArgs a{};
    a.n = g->lu_n;
    a.nf = g->lu_nf;
    a.nnzA = (int)g->red_nnz;
    a.backmax = g->lu_backmax;
    for (int c = 0; c < kMfClasses; ++c) {
        a.nleaf[c] = g->lu_nleaf[c];
        a.leaf[c] = g->lu_leaf[c];
    }
    for (int c = 0; c < 2; ++c) {
        a.npath[c] = g->lu_npath[c];
        a.path[c] = g->lu_path[c];
    }
    a.fr = g->lu_fr;
    a.el = g->lu_el;
    a.ext = g->lu_ext;
    a.bidx = g->lu_bidx;
    a.rel = g->lu_rel;
    a.backp = g->lu_backp;
    a.backw = g->lu_backw;
    a.perm = g->lu_perm;
    a.A = Jr;
    a.F = F;
    a.U = g->lu_U;
    a.cb = g->lu_cb;
    a.x = g->lu_x;
    a.dx = dx;
    a.mat = g->lu_mat;
    a.cnt = g->lu_cnt;
    a.err = g->err;
    cudaError_t e;
    if (g->nsm == 0) {
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&g->nsm, cudaDevAttrMultiProcessorCount, dev)))
            return e;
    }
    const size_t sm_small = sizeof(double) * kMfSmallWarps * kMfSmall * kMfSmallLd;
    const size_t sm_bsmall = sizeof(double) * kMfSmallWarps * 2 * kMfBackSmall;
    const size_t sm_wide = sizeof(double) * (kMfWide + 1) + kMfWideRowBytes;
    const size_t sm_bbig = sizeof(double) * (2 * (size_t)g->lu_backmax + 4 * (size_t)g->lu_backp + g->lu_backw);
    if ((e = ensure_dyn_smem(reinterpret_cast<const void *>(k_mf_wide), sm_wide)) ||
        (e = ensure_dyn_smem(reinterpret_cast<const void *>(k_mf_back_big), sm_bbig)))
        return e;
    // arrivals, written marks and item counters
    if ((e = cudaMemsetAsync(a.cnt, 0, (2 * (size_t)a.nf + kMfClasses + 2) * sizeof(int), s))) return e;
    auto ctas = [&](int items, int per_cta, int per_sm) {
        return std::max(1, std::min(per_sm * g->nsm, (items + per_cta - 1) / per_cta));
    };
    bool first = true;
    auto launch = [&](void (*kernel)(MfArgs), int grid, int block, size_t smem) {
        if (e == cudaSuccess) e = launch_k(kernel, grid, block, smem, s, !first, a);
        first = false;
    };
    if (a.nleaf[0] > 0) launch(k_mf_small, ctas(a.nleaf[0], kMfSmallWarps, 2), 32 * kMfSmallWarps, sm_small);
    if (a.nleaf[1] > 0) launch(k_mf_mid, ctas(a.nleaf[1], 1, 6), 32 * kMfMidWarps, 0);
    if (a.nleaf[2] > 0)
        launch(k_mf_wide, kMfWideCtas * std::min(a.nleaf[2], std::max(1, g->nsm / kMfWideCtas)), 32 * kMfWideWarps, sm_wide);
    if (a.nleaf[3] > 0)
        launch(k_mf_huge, kMfHugeCtas * std::min(a.nleaf[3], std::max(1, g->nsm / kMfHugeCtas)), kMfHugeThreads, 0);
    if (a.npath[1] > 0) launch(k_mf_back_big, ctas(a.npath[1], 1, 2), kMfBackThreads, sm_bbig);
    if (a.npath[0] > 0) launch(k_mf_back_small, ctas(a.npath[0], kMfSmallWarps, 2), 32 * kMfSmallWarps, sm_bsmall);
    return e;
}

}  // namespace pf

using namespace pf;

PF_API pf_status jac_reduced_solve(pf_grid *grid, const double *Jr, const double *F, double *dx, pf_stream stream)
{
    if (!grid) return set_error(PF_EINVAL, "jac_reduced_solve: grid is NULL");
    Grid *g = &grid->g;
    if (!g->red_set) return set_error(PF_EINVAL, "jac_reduced_solve: call grid_set_bus_types first");
    if (g->red_n == 0) return PF_OK;
    if (!Jr || !F || !dx) return set_error(PF_EINVAL, "jac_reduced_solve: NULL argument");
    cudaStream_t s = (cudaStream_t)stream;
    if (pf_status st = lu_prepare(g, s)) return st;
    TraceScope t(g, PF_K_LU, s);
    PF_CUDA(launch_lu_solve(g, Jr, F, dx, s));
    return PF_OK;
}

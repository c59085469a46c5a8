// k_elementwise.cu - element-wise method (Sec. II-B, IV-C) on the GPU: one
// CTA per window of consecutive buses, one launch per evaluation and no
// synchronisation between CTAs.
//
// Phasors.  The paper's element-wise loop evaluates the angle-difference terms
// inside its per-line loop; here each CTA first forms the phasors
// U = e^{j theta}, V = v U of every bus its terminals touch - its own buses
// and its ghost buses (the other ends outside the window, listed at setup) -
// into a window-local table in shared memory.  A bus is transformed once per
// window that touches it (about 1.6-1.8 times per bus on grids numbered with
// spatial locality) instead of once per terminal, and no CTA waits for
// another: the kernel is a plain launch of one CTA per window.
//
// Evaluation step (the per-element loop of Sec. IV-C, one terminal per
// thread).  Terminal t of a branch (owner bus o, other bus q) has precomputed
// constants Ys_t, Yc_t (k_setup.cu) such that its complex power (Eqs. 5-6) is
//     S_t = v_o^2 conj(Ys_t) + K_t,   K_t = conj(Yc_t) V_o conj(V_q),
// where V_o conj(V_q) = v_o v_q e^{j(theta_o - theta_q)} carries the sine and
// cosine of the angle difference.  Its 8 partials (16 per branch):
//     dS_t/dtheta_q = -j K_t            dS_t/dv_q = K_t / v_q = conj(Yc_t) V_o conj(U_q)
//     dS_t/dtheta_o = +j K_t            dS_t/dv_o = 2 v_o conj(Ys_t) + K_t / v_o
// The thread computes G = conj(Yc_t) V_o conj(U_q) (= dS_t/dv_q) in 64-bit
// fixed point on the integer pipe (fixrot.cuh: the phasor table holds U as
// 2^62-scaled integers and V_o in block floating point, the setup Yc_t), then
// K_t = v_q G: 2 FP64 instructions.  The injections alone take the same steps
// (K_t only).
//
// Reduction step (Eq. 7 and the copy-add of Fig. 2, without atomics).
// Terminals are stored sorted by (owner, other bus), so a CTA owns a window of
// consecutive buses together with all of their terminals: the off-diagonal
// slot (o, q) is written by the terminal's thread (the first of a run of
// parallel branches, which are adjacent in the sorted order, adds the others),
// and two threads per bus (the real and the imaginary parts; the window's buses
// taken by decreasing terminal count, so that a warp's lanes loop equally
// long) sum K in a fixed order, with a Jacobian along the bus's staged row, whose
// J11 and J21 entries are the K, else over its terminals:
//     S_o           = v_o^2 conj(Yd_o) + sum K
//     dS_o/dtheta_o = j sum K
//     dS_o/dv_o     = 2 v_o conj(Yd_o) + (sum K) / v_o
// with Yd_o = sum_t Ys_t + y_sh,o, a parameter-only per-bus constant formed at
// setup from the same terminal constants.
//
// Work balance.  The windows are cut at equal estimated FP64 cost into a
// whole number of waves of the CTAs that fit on the GPU (host_layout.cpp), so
// every SM gets the same work.
//
// GB300 data movement.  Every global load of a window (its voltages, the
// ghost voltages, the terminal constants of the first pass, the bus metadata)
// is issued before any arithmetic, in two levels of dependent loads (the
// fixed-stride window records, then what they index).  A window's Jacobian rows are one
// contiguous slice of each of the P and Q halves of J (canonical layout): it
// is assembled in shared memory and written back with TMA bulk stores,
// together with P and Q.
#include <algorithm>

#include "fastmath.cuh"
#include "fixrot.cuh"
#include "pf_internal.h"
#include "ptx.cuh"

namespace pf {

struct EwArgs {
    int nnz, nwin, max_nbus, max_nt, max_L, max_nph, aligned;
    const int4 *desc, *bmeta;
    const int *slotbus, *town, *rorder;
    const double2 *yd, *tcoup;
    const longlong2 *tcfx;
    const int *tce;
    const ITrig *trig;
    const int2 *tloc;
    const double *vm, *va;
    double *P, *Q, *J;
    // mapped outputs (k_ew_red): the destination of every canonical J position
    // in Jr (-1: not kept) and, for the reduced Newton system, the reduced index
    // of every bus's P and Q equation
    const int *jinv;
    const int2 *binv;
    const double *Ps, *Qs;
    double *F, *Jr;
};

#ifdef PF_PHASE_PROBE
// Phase probe (builds with -DPF_PHASE_PROBE only): thread 0 of every CTA of
// the single-evaluation kernel records, per window, the %globaltimer at its
// start and end, its SM, the clock64 cycles from its start to the end of each
// phase (loads, phasors, evaluation, reduction, stores), and the %globaltimer
// when its programmatic-dependent-launch wait returned.
constexpr int kProbeMaxWin = 8192, kProbeSlots = 9;
__device__ unsigned long long g_phase_probe[kProbeMaxWin * kProbeSlots];
__device__ __forceinline__ unsigned long long probe_gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
#define PF_PROBE_MARK(k)                                 \
    do {                                                 \
        if (probe && tid == 0) pt[k] = clock64() - pt0;  \
    } while (0)
#else
#define PF_PROBE_MARK(k) \
    do {                 \
    } while (0)
#endif

// Write x[b0 .. b1) from shared staging `s` (element b0 at s[b0 & 1]) to
// global memory: an unaligned head and tail element by plain stores, the
// 16-byte aligned middle by one bulk store (issued by the calling thread).
__device__ __forceinline__ void store_range(double *x, const double *s, int b0, int b1)
{
    const int par = b0 & 1;
    if (par) x[b0] = s[1];
    const int ge = b0 + par;
    const int cm = (b1 - ge) & ~1;
    if (cm > 0) bulk_s2g(x + ge, s + 2 * par, 8u * (uint32_t)cm);
    if ((b1 - ge) & 1) x[b1 - 1] = s[b1 - 1 - b0 + par];
}

// ---- the Ybus method on the same windows (YBUS) ----
// Its row sum I_i = sum_j Y_ij V_j enters S_i = V_i conj(I_i) and the diagonal
// of the Jacobian only through products with V_i, so each entry's term
// K_ij = V_i conj(Y_ij V_j) = v_j dS_i/dv_j, which the Jacobian needs anyway
// (Eqs. 3-4), is formed once and summed over the row:
//     S_i = v_i^2 conj(Y_ii) + sum K,   conj(I_i) U_i = S_i / v_i.
// An entry of a parallel run holds the run's sum (k_ybus_values writes the
// values in terminal order, zero for the run's later terminals).  Rows with a
// magnitude whose products or quotient might leave the range of normal
// doubles, or with a non-finite angle, are evaluated whole from their current in
// FP64 instead (ybus_row), after the others (calls among the evaluation's products
// and sums, with their spills: 10.1 against 9.4 us at 70,000 buses).  So is a row whose
// own magnitude is zero, since its conj(I_i) U_i is no quotient; zero entries (branches
// out of service) and zero magnitudes of other buses are ordinary factors.
// The rows of a window that go that way are listed first and taken a lane each:
// an FP64 instruction costs a warp the same for one lane as for 32.  70,000 buses, a
// Jacobian, us: 1 % of the branches out of service 8.3, as without; 1 % / 10 % of the
// buses dead 17.3 / 20.2 (34.3, and 33.5 / 50.2, with zeros among the extreme values,
// each row by the two threads of its bus and its phasors formed anew; row kernels with
// the sine and cosine per entry 21).
//
// Why windows: with W lanes per CSR row and the sine and cosine per entry
// (the earlier one-launch form) every bus was transformed 3.5 times and the
// row's results left as scattered 8-byte stores; on windows it is 1.7 times,
// and the results leave as bulk copies.  70,000 buses, Jacobian back to back:
// 21.2 -> 9.4 us a call (k_ew: 8.6); 410,000: 98.5 -> 45.2; 25,000, injections,
// on the device: 9.9 -> 4.8.
constexpr int kYbusSlowRow = (int)0x80000000;

// a biased exponent within 2^-300 .. 2^300
__device__ __forceinline__ bool ybus_mid(int e) { return (unsigned)(e - 723) <= 600u; }

// or zero: a product with it is exact
__device__ __forceinline__ bool ybus_mid_or_zero(double v)
{
    return ybus_mid(fix_vexp(v)) || (dbl_bits(v) << 1) == 0;
}

// Row o by its current I_o (Eqs. 1, 3, 4) in FP64, in the order of operations of
// a row kernel's lane (k_jac_ybus_b), from the window's phasors: its sorted terminals
// from p on, the row's own phasor slot b and diagonal position kd; its d entries into
// the window's J slice (row: its P half's first, the Q half L behind; NULL: the
// injections alone) and S_o
__device__ __noinline__ void ybus_row(const EwArgs &a, const longlong2 *sU, const double2 *sW, int o, int b, int p,
                                      int kd, double *row, int L, int d, double *P, double *Q)
{
    auto cosine = [&](int j, double &s) {
        const longlong2 u = sU[j];
        const double c = fix_q62_or_nan(u.x);
        s = u.x == kFixNaN ? c : q62_to_double(u.y);
        return c;
    };
    double so;
    const double co = cosine(b, so);
    const double v = sW[b].x, Vr = v * co, Vi = v * so;
    double Ir = 0.0, Ii = 0.0, dTr = 0.0, dTi = 0.0, dVr = 0.0, dVi = 0.0;
#pragma unroll 1
    for (int k = 0; k < d; ++k) {   // in column order
        const bool own = k == kd;
        double2 y;
        int j = b;
        if (own) {
            y = a.yd[o];
        } else {
            int2 f = a.tloc[p];
            j = f.x;
            y = make_double2(0.0, 0.0);
            for (;; f = a.tloc[p]) {   // the entry's parallel run, as k_ybus_values sums it
                const double2 c = a.tcoup[p++];
                y.x += c.x;
                y.y += c.y;
                if (!(f.y & EW_MORE)) break;
            }
        }
        double s;
        const double c = cosine(j, s), vj = sW[j].x;
        const double YUr = fma(y.x, c, -y.y * s), YUi = fma(y.x, s, y.y * c);
        const double sVr = fma(Vr, YUr, Vi * YUi), sVi = fma(Vi, YUr, -Vr * YUi);   // V conj(YU)
        const double sTr = vj * sVi, sTi = -vj * sVr;
        Ir = fma(vj, YUr, Ir);
        Ii = fma(vj, YUi, Ii);
        if (own) {
            dTr = sTr;
            dTi = sTi;
            dVr = sVr;
            dVi = sVi;
        } else if (row) {
            row[k] = sTr;
            row[k + d] = sVr;
            row[L + k] = sTi;
            row[L + k + d] = sVi;
        }
    }
    const double Sr = fma(Vr, Ir, Vi * Ii), Si = fma(Vi, Ir, -Vr * Ii);
    if (row) {
        row[kd] = dTr - Si;                                   // + j S
        row[kd + d] = dVr + fma(Ir, co, Ii * so);             // + conj(I) U
        row[L + kd] = dTi + Sr;
        row[L + kd + d] = dVi + fma(Ir, so, -Ii * co);
    }
    *P = Sr;
    *Q = Si;
}

// One window per CTA; with PERSIST the CTAs loop over the windows
// (grid-strided), so that the first windows' outputs leave while later
// windows are evaluated (outputs in host memory, where the host link is the
// bound).
template <bool JAC, bool PERSIST, bool RED = false, bool YBUS = false>
__device__ __forceinline__ void ew_windows(const EwArgs &a)
{
    extern __shared__ __align__(16) char smem[];
    const EwSmem sp = ew_smem_plan(a.max_nbus, a.max_nt, JAC ? a.max_L : 0, JAC, a.max_nph);
    int4 *sbm = reinterpret_cast<int4 *>(smem + sp.bm);
    double2 *syd = reinterpret_cast<double2 *>(smem + sp.yd);   // Yd, or (Jacobian) v conj(Yd)
    double2 *skg = reinterpret_cast<double2 *>(smem + sp.kg);
    double *jst = reinterpret_cast<double *>(smem + sp.jst);
    double *spq = reinterpret_cast<double *>(smem + sp.pq);
    longlong2 *sA = reinterpret_cast<longlong2 *>(smem + sp.ph);             // own buses: V in block floating point
    longlong2 *sU = sA + a.max_nph;                                          // 2^62 (cos, sin)
    double2 *sW = reinterpret_cast<double2 *>(sU + a.max_nph);               // (v, 1/v)
    int *sord = reinterpret_cast<int *>(smem + sp.ord);                     // reduction thread -> bus
    ITrig *tab = reinterpret_cast<ITrig *>(smem + sp.total);
    const int tid = threadIdx.x, TB = blockDim.x;
    // programmatic dependent launch: the next kernel in the stream may start
    // its CTAs as these exit (it waits before it reads or writes anything
    // this kernel may still touch, see below)
    pdl_launch_dependents();
    for (int w = blockIdx.x; w < a.nwin; w += gridDim.x) {
#ifdef PF_PHASE_PROBE
        const bool probe = !PERSIST && !RED && w < kProbeMaxWin;
        const unsigned long long gt0 = probe && tid == 0 ? probe_gtimer() : 0ull;
        const long long pt0 = clock64();
        long long pt[5] = {0, 0, 0, 0, 0};
        unsigned long long gtw = 0ull;
#endif
        if (PERSIST) __syncthreads();   // the previous window's shared-memory readers are done
        // two levels of dependent loads: the window's records (descriptor, the
        // bus of the thread's first phasor slot), then everything they index
        const int *sbus = a.slotbus + (long long)w * a.max_nph;
        const int o0 = tid < a.max_nph ? sbus[tid] : 0;
        const int4 d0 = a.desc[2 * w], d1 = a.desc[2 * w + 1];
        // the sine/cosine table is requested with the first level: issued after
        // the second-level gathers it would arrive at the end of the kernel's
        // whole input burst, and every warp waits for it at the barrier below
        const bool load_tab = !PERSIST || w == (int)blockIdx.x;
        const ITrig *trig = a.trig + (blockIdx.x % kITrigCopies) * kITrigN;
        ITrig tv0 = {0ull, 0ull};
        if (load_tab && tid < kITrigN) tv0 = trig[tid];
        const int b0 = d0.x, nbus = d0.y, b1 = b0 + nbus, t0 = d0.z, nt = d0.w;
        const int r0 = d1.x, L = JAC ? d1.y : 0, nph = d1.z;

        // ---- loads of topology data (fixed when the grid's layout is built;
        // no kernel writes them): the bus thread's metadata (a window has at
        // most blockDim.x buses), kept in registers until the phasors are done
        // so its latency hides behind them, and the first terminal's slots ----
        int4 bmo = make_int4(0, 0, 0, 0);
        int ordo = 0;
        if (tid < nbus) {
            bmo = a.bmeta[b0 + tid];
            ordo = a.rorder[b0 + tid];
        }
        int2 nq = make_int2(0, 0);
        int ol = 0;
        if (tid < nt) {
            nq = a.tloc[t0 + tid];
            ol = a.town[t0 + tid];   // made window-local at first use: nothing before the
                                     // barrier below may wait for a second-level load
        }
        // ---- the previous kernel in the stream may still run (programmatic
        // dependent launch): the state, the parameter-dependent constants and
        // the outputs are read and written only after it has completed; their
        // lines are only brought into L2 before (prefetches return no data) ----
        if (tid < nph) {
            prefetch_l2(a.va + o0);
            prefetch_l2(a.vm + o0);
        }
        if (tid < nbus) prefetch_l2(a.yd + b0 + tid);
        if (tid < nt) {
            prefetch_l2(a.tcfx + t0 + tid);
            prefetch_l2(a.tce + t0 + tid);
        }
        pdl_wait();
#ifdef PF_PHASE_PROBE
        if (probe && tid == 0) gtw = probe_gtimer();
#endif
        double th = 0.0, v = 0.0;
        if (tid < nph) {
            th = a.va[o0];
            v = a.vm[o0];
        }
        double2 ydo = make_double2(0.0, 0.0);
        if (tid < nbus) ydo = a.yd[b0 + tid];
        longlong2 yf = make_longlong2(0, 0);
        int ey = 0;
        if (tid < nt) {
            yf = a.tcfx[t0 + tid];
            ey = a.tce[t0 + tid];
        }
        if (load_tab) {
            if (tid < kITrigN) tab[tid] = tv0;
            for (int k = tid + TB; k < kITrigN; k += TB) tab[k] = trig[k];
        }
        __syncthreads();
        PF_PROBE_MARK(0);

        // ---- phasor table of the window (Sec. IV-B.1 step 1, own and ghost buses) ----
        for (int j = tid; j < nph; j += TB) {
            if (j != tid) {
                const int o = sbus[j];
                th = a.va[o];
                v = a.vm[o];
            }
            int64_t C, S;
            int_sincos_q62(th, tab, &C, &S);
            sU[j] = make_longlong2(C, S);
            double iv = 0.0;
            if (j < nbus) {
                int64_t ar, ai;
                fix_phasor(C, S, v, &ar, &ai);
                sA[j] = make_longlong2(ar, ai);
                if (YBUS && (ar == kFixNaN || !ybus_mid(fix_vexp(v)))) bmo.z |= kYbusSlowRow;   // j = tid is the bus
            }
            if (JAC) {
                // 1/v is read for the window's own buses only: warps of ghost
                // slots skip it (a warp-uniform branch), mixed warps form it
                // for all lanes; and v conj(Yd) of the reduction, formed once per
                // bus here (where the FP64 pipe is idle) instead of by both
                // threads of its pair (slot j < nbus is bus j, whose Yd thread j
                // holds)
                if (__any_sync(__activemask(), j < nbus)) {
                    iv = fast_rcp(v);
                    if (j < nbus) syd[j] = make_double2(v * ydo.x, neg(v * ydo.y));   // v conj(Yd)
                }
            }
            sW[j] = make_double2(v, iv);
        }
        if (tid < nbus) {
            sbm[tid] = bmo;
            if (!JAC) syd[tid] = ydo;
            sord[tid] = ordo;
        }
        __syncthreads();
        PF_PROBE_MARK(1);

        // ---- evaluation: one terminal per thread.  With a Jacobian nothing but
        // the staged entries is kept for the sums (a second copy of K and G and
        // the slot positions were 36 bytes a terminal and three more stores; with
        // them and the parallel runs in the sums' loop 70,000 buses took 8.55 us,
        // 410,000 42.9, without 7.5 and 38.7) ----
        int runs = 0;
        for (int i = tid; i < nt; i += TB) {
            if (i != tid) {
                yf = a.tcfx[t0 + i];
                ey = a.tce[t0 + i];
                nq = a.tloc[t0 + i];
                ol = a.town[t0 + i];
            }
            ol -= b0;
            if (JAC && (nq.y & EW_ACCUM)) continue;   // with the first branch of its parallel run
            // G = conj(Yc) V_o conj(U_q) = dS_t/dv_q on the integer pipe (FP64
            // products for the values the fixed-point form does not hold)
            const longlong2 A = sA[ol], uq = sU[nq.x];
            const double vo = sW[ol].x, vq = sW[nq.x].x;
            double Gr, Gi;
            if (YBUS) {
                // magnitudes whose products might leave the doubles' range, and
                // non-finite angles: the row goes the general way
                if (!(ybus_mid(ey) && ybus_mid_or_zero(vq) && uq.x != kFixNaN) || A.x == kFixNaN ||
                    !fix_G_fast(A.x, A.y, vo, uq.x, uq.y, yf.x, yf.y, ey, &Gr, &Gi)) {
                    Gr = Gi = 0.0;
                    sbm[ol].z |= kYbusSlowRow;
                }
            } else if (A.x == kFixNaN || uq.x == kFixNaN || ey == 0 ||
                       !fix_G_fast(A.x, A.y, vo, uq.x, uq.y, yf.x, yf.y, ey, &Gr, &Gi)) {
                const longlong2 uo = sU[ol];
                const double2 yc = a.tcoup[t0 + i];
                fix_G(A.x, A.y, vo, uo.x, uo.y, uq.x, uq.y, 0, 0, 0, yc.x, yc.y, &Gr, &Gi);
            }
            const double Kr = vq * Gr, Ki = vq * Gi;   // K_t = v_q G
            if (JAC) {
                runs |= nq.y;
                const int4 bm = sbm[ol];
                const int pos = bm.x + (nq.y & EW_KMASK), d = bm.y;
                jst[pos] = Ki;           // J11 = Re(-j K)
                jst[pos + d] = Gr;       // J12
                jst[L + pos] = neg(Kr);  // J21 = Im(-j K)
                jst[L + pos + d] = Gi;   // J22
            } else {
                skg[i] = make_double2(Kr, Ki);
            }
        }
        // the later branches of parallel runs, in their order, onto the entries
        // that this thread wrote (apart from the loop above, which has no
        // registers to spare for them)
        if (JAC && !YBUS && (runs & EW_MORE))
            for (int i = tid; i < nt; i += TB) {
                int p = t0 + i;
                const int2 f = a.tloc[p];
                if ((f.y & EW_ACCUM) || !(f.y & EW_MORE)) continue;
                const int o = a.town[p] - b0;
                const longlong2 A = sA[o], uq = sU[f.x];
                const double vo = sW[o].x, vq = sW[f.x].x;
                const int4 bm = sbm[o];
                double *e = jst + bm.x + (f.y & EW_KMASK);
                int more;
                do {
                    ++p;
                    const longlong2 y = a.tcfx[p];
                    const int ye = a.tce[p];
                    more = a.tloc[p].y & EW_MORE;
                    double Gr, Gi;
                    if (A.x == kFixNaN || uq.x == kFixNaN || ye == 0 ||
                        !fix_G_fast(A.x, A.y, vo, uq.x, uq.y, y.x, y.y, ye, &Gr, &Gi)) {
                        const longlong2 uo = sU[o];
                        const double2 yc = a.tcoup[p];
                        fix_G(A.x, A.y, vo, uo.x, uo.y, uq.x, uq.y, 0, 0, 0, yc.x, yc.y, &Gr, &Gi);
                    }
                    e[0] += vq * Gi;
                    e[bm.y] += Gr;
                    e[L] -= vq * Gr;
                    e[L + bm.y] += Gi;
                } while (more);
            }
        __syncthreads();
        PF_PROBE_MARK(2);

        // ---- reduction: its terminals in sorted order onto every bus ----
        const int pqs = (int)sp.pqs, par = b0 & 1;
        bool slow_row = false;
        if (JAC) {
            // two threads per bus: x = 2b' + im sums the real (im = 0) or imaginary
            // (im = 1) parts of K of bus b = sord[b'] and writes the entries that
            // depend on them only; the arithmetic is uniform across the pair (no
            // divergence), and with the buses taken by decreasing terminal count
            // the lanes of a warp loop about equally long
            for (int x = tid; x < 2 * nbus; x += TB) {
                const int b = sord[x >> 1], im = x & 1;
                const int4 bm = sbm[b];
                if (YBUS && bm.z < 0) {   // below
                    slow_row = true;
                    continue;
                }
                const int d = bm.y;
                // K along the staged row, past the diagonal; the sum starts from the first entry
                const double *row = jst + (im ? 0 : L) + bm.x;
                double sK = 0.0;
                if (d > 1) sK = row[bm.z == 0];
#pragma unroll 1
                for (int k = 1; k < d - 1; ++k) sK += row[k + (k >= bm.z)];
                sK = neg_if(sK, !im);
                const double2 vy = syd[b], vw = sW[b];   // v conj(Yd); v, 1/v
                const double vc = im ? vy.y : vy.x;
                const int pos = bm.x + bm.z;
                jst[(im ? 0 : L) + pos] = neg_if(sK, im);                  // Re / Im of j sum K
                jst[(im ? L : 0) + pos + d] = fma(sK, vw.y, fix_twice(vc));   // 2 v conj(Yd) + sum K / v
                spq[(im ? pqs : 0) + b + par] = fma(vw.x, vc, sK);            // S = v^2 conj(Yd) + sum K
            }
        } else {
            // two threads per bus as above
            const double *k1 = reinterpret_cast<const double *>(skg);   // K.x, K.y per terminal
            for (int x = tid; x < 2 * nbus; x += TB) {
                const int b = sord[x >> 1], im = x & 1;
                const int4 bm = sbm[b];
                const int tend = b + 1 < nbus ? sbm[b + 1].w : nt;
                int i = bm.w;
                double sK = 0.0;
                if (i < tend) sK = k1[2 * i++ + im];
                for (; i < tend; ++i) sK += k1[2 * i + im];
                const double2 y = syd[b];
                const double v = sW[b].x;
                if (YBUS && bm.z < 0)   // below
                    slow_row = true;
                else
                    spq[(im ? pqs : 0) + b + par] = fma(v * v, im ? neg(y.y) : y.x, sK);   // S = v^2 conj(Yd) + sum K
            }
        }
        // everything staged, the rows of the general way (over what the evaluation
        // wrote of them) last; ends with a barrier
        auto staged = [&]() {
            fence_proxy_async_smem();
            if (!YBUS) {
                __syncthreads();
                return;
            }
            if (!__syncthreads_or(slow_row)) return;
            __shared__ int nslow;
            if (tid == 0) nslow = 0;
            __syncthreads();
            if (tid < nbus && sbm[tid].z < 0) sord[atomicAdd(&nslow, 1)] = tid;   // the order of the sums is used up
            __syncthreads();
            for (int x = tid; x < nslow; x += TB) {
                const int b = sord[x];
                const int4 bm = sbm[b];
                ybus_row(a, sU, sW, b0 + b, b, t0 + bm.w, bm.z & ~kYbusSlowRow, JAC ? jst + bm.x : nullptr, L, bm.y,
                         spq + b + par, spq + pqs + b + par);
            }
            fence_proxy_async_smem();
            __syncthreads();
        };

        // ---- stores ----
        if (RED) {
            // J through a map from canonical positions (the reduced system's
            // CSC index, or a caller's pattern's position: Alg. 2's P_xy; -1
            // for an entry that is not kept), then the kept P and Q mismatches
            // to F, or P and Q themselves (no canonical J is written)
            __syncthreads();
            const long long p0 = 2 * (long long)r0, q0 = 2 * (long long)a.nnz + p0 - L;
            constexpr int U = 4;   // map loads in flight per thread and round (more spill at 48 registers)
            for (int base = tid; base < 2 * L; base += U * TB) {
                int k[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int x = base + u * TB;
                    k[u] = x < 2 * L ? a.jinv[(x < L ? p0 : q0) + x] : -1;
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (k[u] >= 0) a.Jr[k[u]] = jst[base + u * TB];
            }
            if (a.binv)
                for (int b = tid; b < nbus; b += TB) {
                    const int2 e = a.binv[b0 + b];
                    if (e.x >= 0) a.F[e.x] = spq[b + par] - a.Ps[b0 + b];
                    if (e.y >= 0) a.F[e.y] = spq[pqs + b + par] - a.Qs[b0 + b];
                }
            if (a.P)
                for (int b = tid; b < nbus; b += TB) {
                    a.P[b0 + b] = spq[b + par];
                    a.Q[b0 + b] = spq[pqs + b + par];
                }
        } else if (a.aligned) {
            staged();
            PF_PROBE_MARK(3);
            if (tid == 0) {
                if (JAC) {
                    bulk_s2g(a.J + 2 * (long long)r0, jst, 8u * (uint32_t)L);
                    bulk_s2g(a.J + 2 * (long long)a.nnz + 2 * (long long)r0, jst + L, 8u * (uint32_t)L);
                }
                if (a.P) {
                    store_range(a.P, spq, b0, b1);
                    store_range(a.Q, spq + pqs, b0, b1);
                }
                bulk_commit();
                bulk_wait_read();   // shared memory stays allocated until the copies have read it
            }
        } else {
            staged();
            if (JAC) {
                double *Jp = a.J + 2 * (long long)r0;
                double *Jq = a.J + 2 * (long long)a.nnz + 2 * (long long)r0;
                for (int x = tid; x < L; x += TB) {
                    Jp[x] = jst[x];
                    Jq[x] = jst[L + x];
                }
            }
            if (a.P)
                for (int b = tid; b < nbus; b += TB) {
                    a.P[b0 + b] = spq[b + par];
                    a.Q[b0 + b] = spq[pqs + b + par];
                }
        }
#ifdef PF_PHASE_PROBE
        if (probe && tid == 0) {
            pt[4] = clock64() - pt0;
            unsigned int smid;
            asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
            unsigned long long *o = g_phase_probe + (long long)w * kProbeSlots;
            o[0] = gt0;
            o[1] = probe_gtimer();
            o[2] = smid;
            for (int k = 0; k < 5; ++k) o[3 + k] = (unsigned long long)pt[k];
            o[8] = gtw;
        }
#endif
        if (!PERSIST) break;
    }
}

// At most 48 registers: 5 CTAs of 256 or 10 of 128 threads per SM.
template <bool JAC>
__global__ void __launch_bounds__(256, 5) k_ew(EwArgs a)
{
    ew_windows<JAC, false>(a);
}

// the same by the Ybus method (one launch)
template <bool JAC>
__global__ void __launch_bounds__(256, 5) k_ybus_win(const __grid_constant__ EwArgs a)
{
    ew_windows<JAC, false, false, true>(a);
}

// the Jacobian evaluation with its outputs in host memory (persistent CTAs)
__global__ void __launch_bounds__(256, 5) k_ew_host(EwArgs a)
{
    ew_windows<true, true>(a);
}

// the Jacobian evaluation with its values stored through a position map: the
// reduced Newton system, or a caller's pattern (Alg. 2)
__global__ void __launch_bounds__(256, 5) k_ew_red(EwArgs a)
{
    ew_windows<true, false, true>(a);
}

static bool al16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// persistent CTAs per SM of the host-output evaluation.  One: since the windows'
// evaluation got faster, a second CTA per SM only makes two overlapping evaluations
// get in each other's way on the host link.  70,000 buses, evaluations/s of
// eval_host_async on two streams / of eval_host: bulk stores 17,400-17,600 /
// 12,900, with two CTAs 16,800 / 12,870; plain stores 16,950-17,140 / 12,670, with
// two CTAs 16,400-16,700 / 12,650.
constexpr int kEwHostCtasPerSm = 1;

enum class EwOut { device, host, reduced, ybus };

template <bool JAC>
static cudaError_t launch_ew(Grid *g, const double *vm, const double *va, double *P, double *Q, double *J,
                             cudaStream_t s, EwOut out, const double *Ps = nullptr, const double *Qs = nullptr,
                             double *F = nullptr, double *Jr = nullptr, const int *jinv = nullptr,
                             const int2 *binv = nullptr)
{
    const EwDev &L = g->ew;
    if (L.nwin == 0) return cudaSuccess;
    const int max_nph = L.max_nph;
    const EwSmem sp = ew_smem_plan(L.max_nbus, L.max_nt, JAC ? L.max_L : 0, JAC, max_nph);
    const uint32_t smem = sp.total + kTrigSmem;
    // outputs in host memory: persistent CTAs (kEwHostCtasPerSm per SM) loop
    // over the windows, so the host link carries the first windows' outputs
    // while the later ones are evaluated
    const bool persist = out == EwOut::host && JAC;
    const bool red = out == EwOut::reduced && JAC, ybus = out == EwOut::ybus;
    uint32_t &conf = persist ? g->ew_smem_host
                     : red   ? g->ew_smem_red
                     : ybus  ? (JAC ? g->yb_smem_jac : g->yb_smem_inj)
                             : (JAC ? g->ew_smem_jac : g->ew_smem_inj);
    // conf: the largest size this grid has ensured (the process-wide limit
    // only grows, so a size ensured once stays valid)
    if (smem > 48u * 1024u && smem > conf) {
        cudaError_t e = ensure_dyn_smem(
            reinterpret_cast<const void *>(persist ? k_ew_host : red ? k_ew_red : ybus ? k_ybus_win<JAC> : k_ew<JAC>),
            smem);
        if (e != cudaSuccess) return e;
        conf = smem;
    }
    int grid = L.nwin;
    if (persist) {
        if (g->nsm == 0) {
            int dev = 0;
            cudaError_t e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g->nsm, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
        }
        grid = std::min(grid, kEwHostCtasPerSm * g->nsm);
    }
    EwArgs a = {};
    a.nnz = g->nnz;
    a.nwin = L.nwin;
    a.max_nbus = L.max_nbus;
    a.max_nt = L.max_nt;
    a.max_L = L.max_L;
    a.max_nph = max_nph;
    // bulk (TMA) stores, to host memory as well; plain coalesced ones where unaligned
    a.aligned = (!J || al16(J)) && (!P || (al16(P) && al16(Q)));
    a.desc = L.desc;
    a.slotbus = L.slotbus;
    a.bmeta = L.bmeta;
    a.rorder = L.rorder;
    a.town = g->town;
    a.yd = g->bus_yd;
    a.tcoup = g->tcoup;
    a.tcfx = ybus ? g->ytfx : g->tcfx;
    a.tce = ybus ? g->yte : g->tce;
    a.trig = trig_table();
    a.tloc = L.tloc;
    a.vm = vm;
    a.va = va;
    a.P = P;
    a.Q = Q;
    a.J = J;
    if (red) {
        a.jinv = jinv;
        a.binv = binv;
        a.Ps = Ps;
        a.Qs = Qs;
        a.F = F;
        a.Jr = Jr;
    }
    // the device-output kernels are launched as programmatic dependents of
    // the previous kernel in the stream (their prologue overlaps its end)
    if (persist) {
        k_ew_host<<<(unsigned)grid, (unsigned)L.tb, smem, s>>>(a);
        return cudaGetLastError();
    }
    if (red) return launch_k(k_ew_red, grid, L.tb, smem, s, true, a);
    if (ybus) return launch_k(k_ybus_win<JAC>, grid, L.tb, smem, s, true, a);
    return launch_k(k_ew<JAC>, grid, L.tb, smem, s, true, a);
}

cudaError_t ew_blocks_per_sm(int tb, size_t smem, int *per_sm)
{
    if (smem > 48u * 1024u) {
        cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void *>(k_ew<true>), smem);
        if (e != cudaSuccess) return e;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_ew<true>, tb, smem);
}

cudaError_t launch_jac_ew(Grid *g, const double *vm, const double *va, double *P, double *Q, double *J,
                          cudaStream_t s, bool host_out)
{
    return launch_ew<true>(g, vm, va, P, Q, J, s, host_out ? EwOut::host : EwOut::device);
}

cudaError_t launch_jac_ew_reduced(Grid *g, const double *vm, const double *va, const double *Ps, const double *Qs,
                                  double *F, double *Jr, cudaStream_t s)
{
    return launch_ew<true>(g, vm, va, nullptr, nullptr, nullptr, s, EwOut::reduced, Ps, Qs, F, Jr, g->red_jinv,
                           g->red_binv);
}

cudaError_t launch_jac_ew_mapped(Grid *g, const double *vm, const double *va, double *P, double *Q, const int *map,
                                 double *Jt, cudaStream_t s)
{
    return launch_ew<true>(g, vm, va, P, Q, nullptr, s, EwOut::reduced, nullptr, nullptr, nullptr, Jt, map,
                           nullptr);
}

cudaError_t launch_inj_ew(Grid *g, const double *vm, const double *va, double *P, double *Q, cudaStream_t s)
{
    return launch_ew<false>(g, vm, va, P, Q, nullptr, s, EwOut::device);
}

cudaError_t launch_ybus_win(Grid *g, bool jac, const double *vm, const double *va, double *P, double *Q, double *J,
                            cudaStream_t s)
{
    return jac ? launch_ew<true>(g, vm, va, P, Q, J, s, EwOut::ybus)
               : launch_ew<false>(g, vm, va, P, Q, nullptr, s, EwOut::ybus);
}

}  // namespace pf

PF_API pf_status pf_phase_probe_read(uint64_t *out, int32_t max_windows, int32_t *nwin)
{
#ifdef PF_PHASE_PROBE
    using namespace pf;
    if (!out || max_windows < 0) return set_error(PF_EINVAL, "pf_phase_probe_read: NULL output or negative size");
    const int n = max_windows < kProbeMaxWin ? max_windows : kProbeMaxWin;
    if (n > 0)
        PF_CUDA(cudaMemcpyFromSymbol(out, g_phase_probe, (size_t)n * kProbeSlots * sizeof(unsigned long long)));
    if (nwin) *nwin = n;
    return PF_OK;
#else
    (void)out;
    (void)max_windows;
    if (nwin) *nwin = 0;
    return pf::set_error(PF_EUNSUPPORTED, "pf_phase_probe_read: library built without -DPF_PHASE_PROBE");
#endif
}

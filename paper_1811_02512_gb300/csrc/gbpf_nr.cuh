// gbpf_nr.cuh -- the Newton-Raphson power flow of one case (Section III of
// arxiv 1811.02512) as device code shared by the Newton-Raphson kernels
// (gbpf_nr.cu) and the fast decoupled kernels, which fall back to it inside
// the same launch for cases the fast decoupled iteration leaves unconverged.
//
// Unknowns: (theta_i, V_i) of every non-slack bus i, one 2 x 2 block per
// entry of the bus-graph pattern of B' (the same ordering, elimination tree
// and levels).  The V unknown of a PV bus is pinned by an identity row and
// column, which keeps the block pattern equal to the bus graph.  The
// Jacobian is factorised without pivoting as J = L D U (unit block-lower L,
// unit block-upper U, 2 x 2 block diagonal D), column by column in level
// order with the same gather lists as the scalar LDL^T, and solved with the
// TMA-staged sweeps: J x = b uses L by rows and U by columns; J^T y = g uses
// U^T by rows and L^T by columns with the same factors (the adjoint).
#pragma once

#include "gbpf_device.cuh"

namespace gbpf {

// Arguments of the Newton-Raphson device code (by value in the kernels'
// parameters; the fast decoupled kernels carry one for their fallback).
struct NrArgs {
    DevNet dn;
    DevCases dc;
    DevMat m;          // pattern of B' (non-slack buses)
    void *F;           // [ncase][jstride] block factors (T)
    double *A;         // [ncase][jstride] FP64 Jacobian: D, Lc (J_rc), Uc (J_cr) regions
    int *fstat;        // [ncase] factor status of the last factorisation
    double tol;
    int max_iter;
    int flat;
    unsigned spin;
    int ir_max;
    double ir_tol, ir_abs;
    double *vm, *va;
    double *ef;        // [ncase][4 nbus]: e, f, P, Q
    double *xg;        // [ncase][6 nbus]: rhs (2n), refined x (2n), FP32 work (2n)
    double *bmax;      // [ncase][16]
    pf_case_result *res;
    const double *gva, *gvm;    // adjoint right-hand side per bus
    double *dJdP, *dJdQ;        // adjoint outputs per bus
    int use_smem;
    unsigned *jdone;   // [ncase][n] column done flags
    unsigned *jsync;   // [ncase][2] column counter, abort flag
    unsigned epoch0;   // factorisation k of this launch publishes epoch0 + k
    int fchunk;        // update terms staged per warp and pass (fits the shared memory)
    MultiSteps js;     // steps of the substitutions for blocks of kMultiThreads
};

// Fills `a` for launch L inside a kernel of 512 threads whose dynamic shared
// memory starts with the staging ring and holds `smem` bytes: the factor
// scratch after the ring takes as many staged update terms per warp as fit
// (32 to 128), the solve vector shares it when it fits.  Returns the
// reservation this needs: `smem`, or more when 32 terms do not fit.
size_t nr_args_within(const NrLaunch &L, size_t smem, NrArgs &a);

namespace {

constexpr int kNrChunkMax = 128;  // update terms staged per warp and pass in the block factor (at most)

// ------------------------------------------------------------ 2 x 2 blocks

template <class T>
struct B2 {
    T a, b, c, d;  // [[a, b], [c, d]]
};

// Blocks are read and written by 16-byte accesses: every block array starts
// at a multiple of four elements of a 16-byte aligned base.
__device__ __forceinline__ B2<float> ld2(const float *p) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return B2<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ B2<double> ld2(const double *p) {
    const double2 u = reinterpret_cast<const double2 *>(p)[0], v = reinterpret_cast<const double2 *>(p)[1];
    return B2<double>{u.x, u.y, v.x, v.y};
}

// A block written by another SM during this launch: read through L2.
__device__ __forceinline__ B2<float> ldcg2(const float *p) {
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(p));
    return B2<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ B2<double> ldcg2(const double *p) {
    const double2 u = __ldcg(reinterpret_cast<const double2 *>(p)), v = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
    return B2<double>{u.x, u.y, v.x, v.y};
}

__device__ __forceinline__ void st2(float *p, const B2<float> &m) {
    *reinterpret_cast<float4 *>(p) = make_float4(m.a, m.b, m.c, m.d);
}
__device__ __forceinline__ void st2(double *p, const B2<double> &m) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(m.a, m.b);
    reinterpret_cast<double2 *>(p)[1] = make_double2(m.c, m.d);
}

template <class T>
__device__ __forceinline__ B2<T> mul2(const B2<T> &x, const B2<T> &y) {
    return B2<T>{x.a * y.a + x.b * y.c, x.a * y.b + x.b * y.d, x.c * y.a + x.d * y.c,
                 x.c * y.b + x.d * y.d};
}

// Injection terms of branch-aware admittance entry (i, k) of case `outage`:
// the base Y entry at Ybus position p minus the outaged branch's share.
__device__ __forceinline__ void y_entry(const DevNet &dn, int outage, int i, int k, int p,
                                        double &G, double &B) {
    G = p >= 0 ? dn.G[p] : 0.0;
    B = p >= 0 ? dn.B[p] : 0.0;
    if (outage < 0 || !dn.bstatus[outage]) return;
    const int f = dn.bf[outage], t = dn.bt[outage];
    if (!((i == f || i == t) && (k == f || k == t))) return;
    const double r = dn.br[outage], x = dn.bx[outage], bc = dn.bb[outage], tp = dn.btap[outage];
    const double den = r * r + x * x;
    const double ys_re = r / den, ys_im = -x / den;
    if (i != k) {
        G += ys_re / tp;
        B += ys_im / tp;
    } else if (i == f) {
        G -= ys_re / (tp * tp);
        B -= (ys_im + 0.5 * bc) / (tp * tp);
    } else {
        G -= ys_re;
        B -= ys_im + 0.5 * bc;
    }
}

// Off-diagonal Jacobian block J_ik = d(P_i, Q_i)/d(theta_k, V_k) from the
// rectangular voltages; PV rows/columns pinned.
__device__ __forceinline__ B2<double> jac_off(double G, double B, double ei, double fi, double ek,
                                              double fk, double vk, bool pv_i, bool pv_k) {
    const double a = ei * ek + fi * fk;  // V_i V_k cos(theta_ik)
    const double b = fi * ek - ei * fk;  // V_i V_k sin(theta_ik)
    B2<double> J;
    J.a = G * b - B * a;                 // dP_i / dtheta_k
    J.b = (G * a + B * b) / vk;          // dP_i / dV_k
    J.c = -(G * a + B * b);              // dQ_i / dtheta_k
    J.d = (G * b - B * a) / vk;          // dQ_i / dV_k
    if (pv_i) { J.c = 0.0; J.d = 0.0; }
    if (pv_k) { J.b = 0.0; J.d = 0.0; }
    return J;
}

__device__ __forceinline__ B2<double> jac_diag(double G, double B, double P, double Q, double v,
                                               bool pv) {
    B2<double> J;
    J.a = -Q - B * v * v;     // dP_i / dtheta_i
    J.b = P / v + G * v;      // dP_i / dV_i
    J.c = P - G * v * v;      // dQ_i / dtheta_i
    J.d = Q / v - B * v;      // dQ_i / dV_i
    if (pv) { J.b = 0.0; J.c = 0.0; J.d = 1.0; }
    return J;
}
// Rectangular voltages of the CTA's bus slice.
__device__ void nr_rect(const NrArgs &a, int c, int i0, int i1) {
    const int nbus = a.dn.nbus;
    const double *vm = a.vm + (long long)c * nbus;
    const double *va = a.va + (long long)c * nbus;
    double *e = a.ef + (long long)c * 4 * nbus;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        double s, co;
        sincos(va[i], &s, &co);
        e[i] = vm[i] * co;
        e[nbus + i] = vm[i] * s;
    }
}

// Injections, mismatch and Newton right-hand side of the slice; returns the
// CTA maximum (NaN wins).
__device__ double nr_mismatch_slice(const NrArgs &a, int c, int i0, int i1, double *red) {
    const DevNet &dn = a.dn;
    const int nbus = dn.nbus;
    const double *e = a.ef + (long long)c * 4 * nbus;
    const double *f = e + nbus;
    double *P = const_cast<double *>(e) + 2 * nbus;
    double *Q = P + nbus;
    double *rhs = a.xg + (long long)c * 6 * nbus;
    const int outage = a.dc.outage[c];
    double mx = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        double p, q;
        bus_injection(dn, i, outage, e, f, p, q);
        P[i] = p;
        Q[i] = q;
        const int t = dn.btype[i];
        const long long idx = (long long)c * nbus + i;
        const double dP = (t != PF_BUS_SLACK) ? a.dc.Psp[idx] - p : 0.0;
        const double dQ = (t == PF_BUS_PQ) ? a.dc.Qsp[idx] - q : 0.0;
        double l = fmax(fabs(dP), fabs(dQ));
        if (dP != dP || dQ != dQ) l = __longlong_as_double(0x7ff8000000000000ll);
        mx = nan_max(mx, l);
        const int k = a.m.new_of_bus[i];
        if (k >= 0) {
            rhs[2 * k] = dP;
            rhs[2 * k + 1] = dQ;
        }
    }
    return block_max(mx, red);
}

// FP64 Jacobian of case c into A: the diagonal blocks of the slots [s0, s1)
// of the (n + nnz) slot range and the lower / upper blocks of the others.
__device__ void nr_assemble(const NrArgs &a, int c, int s0, int s1) {
    const DevNet &dn = a.dn;
    const DevMat &m = a.m;
    const int nbus = dn.nbus;
    const double *e = a.ef + (long long)c * 4 * nbus;
    const double *f = e + nbus;
    const double *P = e + 2 * nbus;
    const double *Q = e + 3 * nbus;
    const double *vm = a.vm + (long long)c * nbus;
    double *A = a.A + (long long)c * m.jstride;
    const int outage = a.dc.outage[c];
    for (int s = s0 + threadIdx.x; s < s1; s += blockDim.x) {
        if (s < m.n) {
            const int i = m.bus[s];
            double G, B;
            y_entry(dn, outage, i, i, dn.ydiag[i], G, B);
            st2(A + m.jD + 4 * s, jac_diag(G, B, P[i], Q[i], vm[i], dn.btype[i] == PF_BUS_PV));
        } else {
            const int p = s - m.n;
            int col = 0;
            {  // column of CSC slot p: binary search in Cp
                int lo = 0, hi = m.n;
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (m.Cp[mid] <= p) lo = mid; else hi = mid;
                }
                col = lo;
            }
            const int r = m.Cr[p];
            const int i = m.bus[r], k = m.bus[col];
            const bool pvi = dn.btype[i] == PF_BUS_PV, pvk = dn.btype[k] == PF_BUS_PV;
            double G, B;
            y_entry(dn, outage, i, k, m.src[m.n + p], G, B);
            st2(A + m.jLc + 4 * p, jac_off(G, B, e[i], f[i], e[k], f[k], vm[k], pvi, pvk));
            y_entry(dn, outage, k, i, m.srcT[p], G, B);
            st2(A + m.jUc + 4 * p, jac_off(G, B, e[k], f[k], e[i], f[i], vm[i], pvk, pvi));
        }
    }
}

// Sums the eight values of v over the warp by halving: each of the first
// three exchanges leaves a lane half of its values, so nine additions do
// what eight butterflies take forty for (an FP64 addition holds its SM
// sub-partition's unit for 64 cycles).  Lane 4 q receives the sum of v[q].
template <class T>
__device__ __forceinline__ T warp_sum8(const T (&v)[8]) {
    const int lane = threadIdx.x & 31;
    T a[4], b[2], c;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const T o = __shfl_xor_sync(0xffffffffu, lane & 16 ? v[i] : v[i + 4], 16);
        a[i] = (lane & 16 ? v[i + 4] : v[i]) + o;
    }
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const T o = __shfl_xor_sync(0xffffffffu, lane & 8 ? a[i] : a[i + 2], 8);
        b[i] = (lane & 8 ? a[i + 2] : a[i]) + o;
    }
    const T o = __shfl_xor_sync(0xffffffffu, lane & 4 ? b[0] : b[1], 4);
    c = (lane & 4 ? b[1] : b[0]) + o;
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    return c;
}

// The top levels [l0, nlev) of the block factor, whose few columns carry most
// of the update terms: a warp per target, so that a column's targets spread
// over every warp of the cluster, and one cluster barrier per level.  The
// columns' entries stay unnormalised until the end (Lu_ic = L_ic D_c, Uu_ci =
// D_c U_ci), so that no target waits for its column's diagonal,
//   Lu_ic = A_ic - sum_k L_ik (M_k U_kc),  Uu_ci = A_ci - sum_k (L_ck M_k) U_ki,
// with M_k = D_k for the normalised columns below l0 and D_k^-1 for those of
// the top.  Bound by the latency of a level: the lists, the blocks and the
// barrier.  A warp reads its next target's first terms ahead of the barrier.
// Newton run and adjoint of a 20,000-bus grid, FP32 factors: 144.8 ms with a
// warp per column throughout (and 21 refinement solves in the adjoint),
// 61.9 ms with this form (and the refinement's stop, nr_solve).
template <class T, int C>
__device__ void block_factor_top(const NrArgs &a, int c, int rank, T *F, const double *Aj, double piv) {
    const DevMat &m = a.m;
    constexpr int kw = C > 1 ? 1 : 0;
    const int lane = threadIdx.x & 31, nw = int(blockDim.x >> 5);
    const int gw = rank * nw + int(threadIdx.x >> 5), W = C * nw;
    const int ct = m.jct[kw], l0 = m.jl0[kw];
    T *D = F + m.jD, *Di = F + m.jDi, *Lc = F + m.jLc, *Uc = F + m.jUc;
    T *Lr = F + m.jLr, *Ur = F + m.jUr;
    if (l0 >= m.nlev) return;
    const int tend = m.jlt[m.nlev];
    // next target of this warp and its first terms' indices
    int lo = 0, hi = 0, col = 0;
    int4 e0 = make_int4(0, 0, 0, 0), e1 = e0;
    auto fetch = [&](int t) {
        lo = m.gp[t];
        hi = m.gp[t + 1];
        col = m.jtcol[t - m.jg0];
        if (lo + lane < hi) e0 = __ldg(m.gl + lo + lane);
        if (lo + 32 + lane < hi) e1 = __ldg(m.gl + lo + 32 + lane);
    };
    int ta = m.jlt[l0], te = m.jlt[l0 + 1];
    if (ta + gw < te) fetch(ta + gw);
    for (int l = l0; l < m.nlev; l++) {
        const int tn = l + 1 < m.nlev ? m.jlt[l + 2] : tend;
        for (int t = ta + gw; t < te; t += W) {
            if (t != ta + gw) fetch(t);
            const bool diag = col < 0;
            const int cc = diag ? ~col : col;
            const int p = t - cc - 1;  // CSC position of an off-diagonal target
            const int q = lane >> 2;   // component of [L-side | U-side] this lane's group ends with
            double src = 0.0;
            if (diag) src = q < 4 ? Aj[m.jD + 4 * cc + q] : 0.0;
            else src = q < 4 ? Aj[m.jLc + 4 * p + q] : Aj[m.jUc + 4 * p + q - 4];
            T v[8];
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] = T(0);
            auto term = [&](const B2<T> &Lx, const B2<T> &Mk, const B2<T> &Uy, const B2<T> &Ly, const B2<T> &Ux) {
                const B2<T> x = mul2(Lx, mul2(Mk, Uy));
                v[0] += x.a; v[1] += x.b; v[2] += x.c; v[3] += x.d;
                if (!diag) {
                    const B2<T> y = mul2(mul2(Ly, Mk), Ux);
                    v[4] += y.a; v[5] += y.b; v[6] += y.c; v[7] += y.d;
                }
            };
            for (int g = lo; g < hi; g += 64) {  // two terms per lane in flight
                const int g0 = g + lane, g1 = g0 + 32;
                if (g != lo) {
                    if (g0 < hi) e0 = __ldg(m.gl + g0);
                    if (g1 < hi) e1 = __ldg(m.gl + g1);
                }
                B2<T> A0, A1, A2, A3, A4, B0, B1, B2_, B3, B4;
                if (g0 < hi) {
                    A0 = ldcg2(Lc + 4 * e0.x); A1 = ldcg2((e0.z < ct ? D : Di) + 4 * e0.z);
                    A2 = ldcg2(Uc + 4 * e0.y); A3 = ldcg2(Lc + 4 * e0.y); A4 = ldcg2(Uc + 4 * e0.x);
                }
                if (g1 < hi) {
                    B0 = ldcg2(Lc + 4 * e1.x); B1 = ldcg2((e1.z < ct ? D : Di) + 4 * e1.z);
                    B2_ = ldcg2(Uc + 4 * e1.y); B3 = ldcg2(Lc + 4 * e1.y); B4 = ldcg2(Uc + 4 * e1.x);
                }
                if (g0 < hi) term(A0, A1, A2, A3, A4);
                if (g1 < hi) term(B0, B1, B2_, B3, B4);
            }
            const T s = T(src) - warp_sum8<T>(v);
            if (diag) {
                const B2<T> Dc{__shfl_sync(0xffffffffu, s, 0), __shfl_sync(0xffffffffu, s, 4),
                               __shfl_sync(0xffffffffu, s, 8), __shfl_sync(0xffffffffu, s, 12)};
                if (lane == 0) {
                    const T det = Dc.a * Dc.d - Dc.b * Dc.c;
                    st2(D + 4 * cc, Dc);
                    st2(Di + 4 * cc, B2<T>{Dc.d / det, -Dc.b / det, -Dc.c / det, Dc.a / det});
                    const double dd = double(det);
                    if (!isfinite(dd) || !isfinite(double(Dc.a)) || !isfinite(double(Dc.d)))
                        atomicCAS(a.fstat + c, PF_OK, PF_ERR_NONFINITE);
                    else if (fabs(dd) <= piv)
                        atomicCAS(a.fstat + c, PF_OK, PF_ERR_SINGULAR);
                }
            } else if ((lane & 3) == 0) {
                if (q < 4) Lc[4 * p + q] = s;
                else Uc[4 * p + q - 4] = s;
            }
        }
        ta = te;
        te = tn;
        if (ta + gw < te) fetch(ta + gw);
        cluster_sync<C>();
    }
    // normalise the top's columns and write their rows
    for (int t = m.jlt[l0] + rank * int(blockDim.x) + int(threadIdx.x); t < tend; t += C * int(blockDim.x)) {
        const int cc = m.jtcol[t - m.jg0];
        if (cc < 0) continue;
        const int p = t - cc - 1;
        const B2<T> inv = ldcg2(Di + 4 * cc);
        const B2<T> L = mul2(ldcg2(Lc + 4 * p), inv), U = mul2(inv, ldcg2(Uc + 4 * p));
        const int r = m.Cpos[p];
        st2(Lc + 4 * p, L);
        st2(Uc + 4 * p, U);
        st2(Lr + 4 * r, L);
        st2(Ur + 4 * r, U);
    }
}

// Block LDU factor of the Jacobian of case c (Section III.B with 2 x 2
// blocks, no pivoting; the pivot check is on det(D_c) against the largest
// diagonal-block entry) by all C blocks of its cluster, driven by the
// elimination tree's dependencies: every warp of the cluster takes
// columns in level order from a counter, waits until the columns of row c of
// L are done (their flags hold `epoch`), then computes each target block of
// column c with a lane per target from the gather lists of the pattern
// (Section III.B, 2 x 2 blocks),
//   A_ic - sum_k L_ik (D_k U_kc),  A_ci - sum_k (L_ck D_k) U_ki,
// publishes D_c, D_c^-1, L_ic = A_ic D_c^-1, U_ci = D_c^-1 A_ci (by column
// and by row) and its own flag.  Every wait is bounded; one that gives up
// raises the case's abort flag.  The columns of the top levels follow level
// by level (block_factor_top).  Cluster-uniform status.
template <class T, int C>
__device__ int cluster_block_factor(const NrArgs &a, int c, int rank, T *F, const double *Aj,
                                    unsigned char *scratch, double *red, unsigned epoch) {
    const DevMat &m = a.m;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chunk = a.fchunk;
    const int sa = 8 * (m.max_col + 1) + 8 * chunk;
    T *accL = reinterpret_cast<T *>(scratch) + warp * sa;
    T *accU = accL + 4 * (m.max_col + 1);
    T *termL = accU + 4 * (m.max_col + 1);
    T *termU = termL + 4 * chunk;
    T *D = F + m.jD, *Di = F + m.jDi, *Lc = F + m.jLc, *Uc = F + m.jUc;
    T *Lr = F + m.jLr, *Ur = F + m.jUr;
    unsigned *done = a.jdone + (long long)c * m.n;
    unsigned *ctr = a.jsync + 2LL * c, *abort_flag = ctr + 1;
    // pivot tolerance: largest diagonal-block entry over the cluster
    const int nd = 4 * m.n, slice = (nd + C - 1) / C;
    double amax = 0.0;
    for (int j = rank * slice + int(threadIdx.x); j < min(nd, (rank + 1) * slice); j += blockDim.x)
        amax = fmax(amax, fabs(Aj[m.jD + j]));
    amax = block_max(amax, red);
    if (threadIdx.x == 0) {
        a.bmax[(long long)c * 16 + rank] = amax;
        if (rank == 0) {
            *ctr = 0u;
            *abort_flag = 0u;
            a.fstat[c] = PF_OK;
        }
    }
    cluster_sync<C>();
    amax = 0.0;
    for (int r = 0; r < C; r++) amax = fmax(amax, a.bmax[(long long)c * 16 + r]);
    const double piv = 1e-14 * amax * amax;
    const int ct = m.jct[C > 1 ? 1 : 0];  // columns from here on: block_factor_top
    for (;;) {
        unsigned col = 0;
        if (lane == 0) col = atomicAdd(ctr, 1u);
        col = __shfl_sync(0xffffffffu, col, 0);
        if (col >= unsigned(ct)) break;
        const int cc = int(col);
        bool ok = true;
        for (int q = m.Fp[cc] + lane; q < m.Fp[cc + 1] && ok; q += 32) {
            const unsigned *f = done + m.Fc[q];
            unsigned it = 0;
            unsigned v;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
                if (v == epoch) break;
                if (++it > a.spin || *reinterpret_cast<volatile unsigned *>(abort_flag)) {
                    ok = false;
                    break;
                }
                __nanosleep(32);
            }
        }
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) {
                atomicExch(abort_flag, 1u);
                atomicCAS(a.fstat + c, PF_OK, PF_ERR_TIMEOUT);
            }
            continue;
        }
        const int c0 = m.Cp[cc], cnt = m.Cp[cc + 1] - c0, tb = c0 + cc;
        for (int t = lane; t <= cnt; t += 32) {
            const double *src = t == 0 ? Aj + m.jD + 4 * cc : Aj + m.jLc + 4 * (c0 + t - 1);
            st2(accL + 4 * t, B2<T>{T(src[0]), T(src[1]), T(src[2]), T(src[3])});
            if (t > 0) {
                const double *us = Aj + m.jUc + 4 * (c0 + t - 1);
                st2(accU + 4 * t, B2<T>{T(us[0]), T(us[1]), T(us[2]), T(us[3])});
            }
        }
        // the column's update terms, a chunk at a time: evaluated with the
        // whole warp (a lane per term) into shared memory, then summed per
        // target with a lane per target in list order
        const int gb = m.gp[tb], ge = m.gp[tb + cnt + 1];
        for (int cb = gb; cb < ge; cb += chunk) {
            const int ce = min(ge, cb + chunk);
            // four terms per lane in flight: their indices, then their blocks
            for (int g0 = cb + lane; g0 < ce; g0 += 128) {
                int4 e[4];
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (g0 + 32 * u < ce) e[u] = __ldg(m.gl + g0 + 32 * u);
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int g = g0 + 32 * u;
                    if (g >= ce) continue;
                    const B2<T> Lx = ldcg2(Lc + 4 * e[u].x), Dk = ldcg2(D + 4 * e[u].z);
                    const B2<T> Uy = ldcg2(Uc + 4 * e[u].y), Ly = ldcg2(Lc + 4 * e[u].y);
                    const B2<T> Ux = ldcg2(Uc + 4 * e[u].x);
                    st2(termL + 4 * (g - cb), mul2(Lx, mul2(Dk, Uy)));
                    st2(termU + 4 * (g - cb), mul2(mul2(Ly, Dk), Ux));
                }
            }
            __syncwarp();
            for (int t = lane; t <= cnt; t += 32) {
                const int lo = max(m.gp[tb + t], cb), hi = min(m.gp[tb + t + 1], ce);
                if (lo >= hi) continue;
                B2<T> sl{T(0), T(0), T(0), T(0)}, su{T(0), T(0), T(0), T(0)};
                for (int g = lo; g < hi; g++) {
                    const B2<T> a2 = ld2(termL + 4 * (g - cb)), b2 = ld2(termU + 4 * (g - cb));
                    sl.a += a2.a; sl.b += a2.b; sl.c += a2.c; sl.d += a2.d;
                    su.a += b2.a; su.b += b2.b; su.c += b2.c; su.d += b2.d;
                }
                T *al = accL + 4 * t;
                al[0] -= sl.a; al[1] -= sl.b; al[2] -= sl.c; al[3] -= sl.d;
                if (t > 0) {
                    T *au = accU + 4 * t;
                    au[0] -= su.a; au[1] -= su.b; au[2] -= su.c; au[3] -= su.d;
                }
            }
            __syncwarp();
        }
        const B2<T> Dc = ld2(accL);
        const T det = Dc.a * Dc.d - Dc.b * Dc.c;
        const B2<T> inv{Dc.d / det, -Dc.b / det, -Dc.c / det, Dc.a / det};
        if (lane == 0) {
            st2(D + 4 * cc, Dc);
            st2(Di + 4 * cc, inv);
            const double dd = double(det);
            if (!isfinite(dd) || !isfinite(double(Dc.a)) || !isfinite(double(Dc.d)))
                atomicCAS(a.fstat + c, PF_OK, PF_ERR_NONFINITE);
            else if (fabs(dd) <= piv)
                atomicCAS(a.fstat + c, PF_OK, PF_ERR_SINGULAR);
        }
        for (int t = lane; t < cnt; t += 32) {
            const B2<T> L = mul2(ld2(accL + 4 * (1 + t)), inv);
            const B2<T> U = mul2(inv, ld2(accU + 4 * (1 + t)));
            st2(Lc + 4 * (c0 + t), L);
            st2(Uc + 4 * (c0 + t), U);
            const int q = m.Cpos[c0 + t];
            st2(Lr + 4 * q, L);
            st2(Ur + 4 * q, U);
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(done + cc), "r"(epoch) : "memory");
    }
    cluster_sync<C>();
    block_factor_top<T, C>(a, c, rank, F, Aj, piv);
    cluster_sync<C>();
    const int st = *reinterpret_cast<volatile int *>(a.fstat + c);
    cluster_sync<C>();
    return st;
}

// One substitution sweep over the steps of a matrix (MultiSteps; the scheme of
// sweep_multi): x_r = (dinv ? Dinv_r x_r : x_r) - sum over row r's blocks of
// B_e x_{idx_e}, transposed with TRANS.  The factor is read straight from L2,
// a step's ranges two steps and its first blocks one step ahead.  (Staged by
// bulk copies with a warp alone on the narrow levels, a solve of a 20,000-bus
// Jacobian in FP32 took 1.4 ms.)
template <class T, bool TRANS, bool DIAG>
__device__ __forceinline__ void sweep_block2(const int2 *steps, int ns, const int *ptr, const int *idx, const T *val,
                                             const T *dinv, T *x) {
    const int slot = threadIdx.x;
    if (ns <= 0) return;
    auto step_at = [&](int j) { return __ldg(steps + min(j, ns - 1)); };
    auto range = [&](const int2 &s, int &r, int &a, int &b) {
        const int q = slot >> (unsigned(s.x) >> 28);
        r = q < (s.y & 0x7fffffff) ? (s.x & 0xfffffff) + q : -1;
        a = b = 0;
        if (r >= 0) {
            a = ptr[r];
            b = ptr[r + 1];
        }
    };
    int2 s0 = step_at(0), s1 = step_at(1), s2 = step_at(2);
    int r0, a0, b0, r1, a1, b1, r2, a2, b2, i0 = 0, i1 = 0;
    B2<T> v0{T(0), T(0), T(0), T(0)}, v1 = v0;
    auto entry = [&](const int2 &s, int a, int b, int &i, B2<T> &v) {
        const int e = a + (slot & ((1 << (unsigned(s.x) >> 28)) - 1));
        if (e < b) {
            i = idx[e];
            v = ldcg2(val + 4LL * e);
        }
    };
    range(s0, r0, a0, b0);
    range(s1, r1, a1, b1);
    entry(s0, a0, b0, i0, v0);
    for (int j = 0; j < ns; j++) {
        const int2 s3 = step_at(j + 3);
        entry(s1, a1, b1, i1, v1);
        range(s2, r2, a2, b2);
        const int G = 1 << (unsigned(s0.x) >> 28), gl = slot & (G - 1);
        if (__any_sync(0xffffffffu, r0 >= 0)) {
            T p = T(0), q = T(0);
            auto mac = [&](const B2<T> &B, int i) {
                const T y0 = x[2 * i], y1 = x[2 * i + 1];
                p += B.a * y0;
                p += (TRANS ? B.c : B.b) * y1;
                q += (TRANS ? B.b : B.c) * y0;
                q += B.d * y1;
            };
            if (a0 + gl < b0) mac(v0, i0);
            for (int e = a0 + G + gl; e < b0; e += 2 * G) {  // two blocks in flight
                const bool two = e + G < b0;
                const int u = idx[e], w = two ? idx[e + G] : 0;
                const B2<T> B = ldcg2(val + 4LL * e);
                B2<T> D = B;
                if (two) D = ldcg2(val + 4LL * (e + G));
                mac(B, u);
                if (two) mac(D, w);
            }
            for (int o = G >> 1; o > 0; o >>= 1) {
                p += __shfl_xor_sync(0xffffffffu, p, o);
                q += __shfl_xor_sync(0xffffffffu, q, o);
            }
            if (r0 >= 0 && gl == 0) {
                T y0 = x[2 * r0], y1 = x[2 * r0 + 1];
                if (DIAG) {
                    const B2<T> D = ldcg2(dinv + 4LL * r0);
                    const T z0 = D.a * y0 + (TRANS ? D.c : D.b) * y1;
                    y1 = (TRANS ? D.b : D.c) * y0 + D.d * y1;
                    y0 = z0;
                }
                x[2 * r0] = y0 - p;
                x[2 * r0 + 1] = y1 - q;
            }
        }
        if (s0.y < 0) __syncthreads();
        s0 = s1; r0 = r1; a0 = a1; b0 = b1; i0 = i1; v0 = v1;
        s1 = s2; r1 = r2; a1 = a2; b1 = b2;
        s2 = s3;
    }
}

// J x = x (TRANS = false) or J^T x = x (TRANS = true) with the block factors.
template <class T, class X, bool TRANS>
__device__ bool block_solve2(Ring *R, unsigned char *stages, const DevMat &m, const T *F, X *x,
                             unsigned spin) {
    if (!staged_sweep<T, X, 2, TRANS>(R, stages, m.pfJ, m.npfJ, m.Fp, m.Fc,
                                      F + (TRANS ? m.jUr : m.jLr), nullptr, m.lvl_ptr, x, spin))
        return false;
    return staged_sweep<T, X, 2, TRANS>(R, stages, m.pbJ, m.npbJ, m.Cp, m.Cr,
                                        F + (TRANS ? m.jLc : m.jUc), F + m.jDi, m.lvl_ptr, x, spin);
}

// r = b - J x (TRANS: b - J^T x) for row r of the FP64 Jacobian A.
template <bool TRANS>
__device__ __forceinline__ void jac_residual_row(const DevMat &m, const double *A, const double *b,
                                                 const double *x, int r, double &r0, double &r1) {
    double s0 = b[2 * r], s1 = b[2 * r + 1];
    const double *D = A + m.jD + 4 * r;
    const double x0 = x[2 * r], x1 = x[2 * r + 1];
    if (!TRANS) {
        s0 -= D[0] * x0 + D[1] * x1;
        s1 -= D[2] * x0 + D[3] * x1;
    } else {
        s0 -= D[0] * x0 + D[2] * x1;
        s1 -= D[1] * x0 + D[3] * x1;
    }
    // the off-diagonal blocks of the row, columns ascending; fill blocks are
    // zero in J and left out (twice the entries on a 20,000-bus grid)
    for (int e = m.Ap[r]; e < m.Ap[r + 1]; e++) {
        const int j = m.Aj[e], p = m.Apos[e] - m.offLc;
        const B2<double> Bk = ld2(A + ((j < r) != TRANS ? m.jLc : m.jUc) + 4LL * p);  // J_rj, or J_jr for J^T
        const double y0 = x[2 * j], y1 = x[2 * j + 1];
        if (!TRANS) { s0 -= Bk.a * y0 + Bk.b * y1; s1 -= Bk.c * y0 + Bk.d * y1; }
        else { s0 -= Bk.a * y0 + Bk.c * y1; s1 -= Bk.b * y0 + Bk.d * y1; }
    }
    r0 = s0;
    r1 = s1;
}

// Refined block solve of case c in one block: x = J^-1 b (or J^-T b) into
// the refined-x region, with FP64 residuals against A when the factor is
// FP32 (or when `always_refine`, e.g. factors of an earlier state).
template <class T, bool TRANS>
__device__ bool nr_solve(const NrArgs &a, Ring *R, unsigned char *stages, T *xs, const T *F,
                         const double *A, int c, double *red, int &ir_steps, bool always_refine) {
    const DevMat &m = a.m;
    const int nbus = a.dn.nbus;
    const int N = 2 * m.n;
    double *b = a.xg + (long long)c * 6 * nbus;
    double *x64 = b + 2 * nbus;
    T *xv = xs ? xs : reinterpret_cast<T *>(x64 + 2 * nbus);
    const bool refine = always_refine || sizeof(T) != sizeof(double);
    double bn = 0.0;
    for (int r = threadIdx.x; r < N; r += blockDim.x) {
        xv[r] = T(b[r]);
        bn = fmax(bn, fabs(b[r]));
    }
    bn = block_max(bn, red);
    bool ok = true;
    constexpr double kStagnant = 1e-9;
    double first = 0.0, last = INFINITY;
    for (int k = 0;; k++) {
        if (a.js.steps && blockDim.x == kMultiThreads) {
            sweep_block2<T, TRANS, false>(a.js.steps, a.js.nf, m.Fp, m.Fc, F + (TRANS ? m.jUr : m.jLr), nullptr, xv);
            sweep_block2<T, TRANS, true>(a.js.steps + a.js.nf, a.js.nb, m.Cp, m.Cr, F + (TRANS ? m.jLc : m.jUc),
                                         F + m.jDi, xv);
        } else {
            ok = block_solve2<T, T, TRANS>(R, stages, m, F, xv, a.spin);
            if (!ok) break;
        }
        T dn = T(0);
        for (int r = threadIdx.x; r < N; r += blockDim.x) {
            x64[r] = (k == 0 ? 0.0 : x64[r]) + double(xv[r]);
            dn = fmax(dn, fabs(xv[r]));
        }
        // a refinement to the last bit (the adjoint's) ends when its
        // corrections no longer shrink: they are then the rounding of the
        // residual seen through the inverse, and further ones only replace
        // one rounding by another.  The corrections, not the residual, are
        // what tells: an ill-conditioned component is still converging when
        // its share of the residual is long below the rounding of the rest
        // (stopping on the residual left 1.5e-10 of error where this leaves
        // 4e-13 and all 21 solves 1.3e-12, on a 20,000-bus grid).  Only
        // corrections far below the first solution are that rounding: with a
        // factor that is hardly an inverse they shrink by less than a tenth
        // from the start, and all ir_max of them are needed.
        double step = 0.0;
        if (always_refine) step = block_max(double(dn), red);
        else __syncthreads();
        if (!refine || k >= a.ir_max) break;
        if (k == 0) first = step;
        if (always_refine && step > 0.9 * last && step <= kStagnant * first) break;
        last = step;
        double rn = 0.0;
        for (int r = threadIdx.x; r < m.n; r += blockDim.x) {
            double r0, r1;
            jac_residual_row<TRANS>(m, A, b, x64, r, r0, r1);
            xv[2 * r] = T(r0);
            xv[2 * r + 1] = T(r1);
            rn = nan_max(rn, fmax(fabs(r0), fabs(r1)));
        }
        rn = block_max(rn, red);
        if (!(rn > a.ir_tol * bn) || !(rn > a.ir_abs)) break;
        ir_steps++;
    }
    return ok;
}

// Newton-Raphson power flow of case c on the C CTAs of its cluster (this
// CTA is `rank`): mismatch, Jacobian assembly and factor spread over the
// cluster, the refined solve in CTA 0, until the mismatch is within a.tol or
// a.max_iter steps; writes the case's result (method PF_NR).  Shared memory:
// the staging ring at smem_raw, then the factor scratch (a.fchunk update
// terms per warp), which the solve vector shares when a.use_smem.  The ring
// R must be initialised; its phases run on from whatever used it before.
template <class T, int C>
__device__ __forceinline__ void nr_case(const NrArgs &a, int c, int rank, unsigned char *smem_raw,
                                        double *red, Ring *R) {
    const DevNet &dn = a.dn;
    const DevMat &m = a.m;
    const int nbus = dn.nbus;
    unsigned char *stages = smem_raw;
    unsigned char *scratch = smem_raw + kStages * kStageBytes;
    T *xs = a.use_smem ? reinterpret_cast<T *>(scratch) : nullptr;  // shares the factor scratch
    double *vm = a.vm + (long long)c * nbus;
    double *va = a.va + (long long)c * nbus;
    double *flag = a.bmax + (long long)c * 16 + 15;
    T *F = static_cast<T *>(a.F) + (long long)c * m.jstride;
    const double *A = a.A + (long long)c * m.jstride;
    const int slice = (nbus + C - 1) / C;
    const int i0 = rank * slice, i1 = min(nbus, i0 + slice);
    const int nslot = m.n + m.nnz;
    const int sslice = (nslot + C - 1) / C;
    const int s0 = rank * sslice, s1 = min(nslot, s0 + sslice);
    if (a.flat)
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const int t = dn.btype[i];
            vm[i] = (t == PF_BUS_PQ) ? 1.0 : dn.vset[i];
            va[i] = (t == PF_BUS_SLACK) ? dn.va0[i] : 0.0;
        }
    int status = PF_ERR_NOT_CONVERGED, iters = 0, ir_steps = 0;
    double mis = INFINITY;
    for (int it = 0;; it++) {
        nr_rect(a, c, i0, i1);
        cluster_sync<C>();
        const double mx = nr_mismatch_slice(a, c, i0, i1, red);
        if (threadIdx.x == 0) a.bmax[(long long)c * 16 + rank] = mx;
        cluster_sync<C>();
        mis = 0.0;
        for (int r = 0; r < C; r++) mis = nan_max(mis, a.bmax[(long long)c * 16 + r]);
        if (!isfinite(mis)) { status = PF_ERR_NONFINITE; break; }
        if (mis <= a.tol) { status = PF_OK; break; }
        if (it >= a.max_iter) break;
        nr_assemble(a, c, s0, s1);
        cluster_sync<C>();
        const int fs = cluster_block_factor<T, C>(a, c, rank, F, A, scratch, red, a.epoch0 + unsigned(it) + 1u);
        if (rank == 0) {
            bool ok = fs == PF_OK;
            if (ok) ok = nr_solve<T, false>(a, R, stages, xs, F, A, c, red, ir_steps, false);
            if (threadIdx.x == 0) {
                a.fstat[c] = fs;
                *flag = fs != PF_OK ? double(fs) : (ok ? 0.0 : double(PF_ERR_TIMEOUT));
            }
        }
        cluster_sync<C>();
        if (*flag != 0.0) { status = int(*flag); break; }
        const double *dx = a.xg + (long long)c * 6 * nbus + 2 * nbus;
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const int k = m.new_of_bus[i];
            if (k >= 0) {
                va[i] += dx[2 * k];
                if (dn.btype[i] == PF_BUS_PQ) vm[i] += dx[2 * k + 1];
            }
        }
        iters++;
    }
    if (rank == 0 && threadIdx.x == 0) {
        a.res[c].status = status;
        a.res[c].iters = iters;
        a.res[c].ir_steps = ir_steps;
        a.res[c].method = PF_NR;
        a.res[c].max_mismatch = mis;
    }
    cluster_sync<C>();
}

// The Newton-Raphson fallback of case c inside a fast decoupled kernel, out
// of line: the fast decoupled loop keeps its own register allocation, and
// the arguments are read where they are (a __grid_constant__ parameter or a
// global array).  The caller's status is cluster-uniform, so every CTA of
// the cluster enters.
template <class T, int C>
__device__ __noinline__ void nr_fallback(const NrArgs &a, int c, int rank, unsigned char *smem_raw,
                                         double *red, Ring *R) {
    nr_case<T, C>(a, c, rank, smem_raw, red, R);
}

}  // namespace

}  // namespace gbpf

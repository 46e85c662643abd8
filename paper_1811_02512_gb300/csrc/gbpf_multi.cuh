// gbpf_multi.cuh -- the fast decoupled power flow of K cases per thread block
// (Section III of arxiv 1811.02512), for batches whose solves all use the
// base factor (load cases, and outage cases in their low-rank form).
//
// One block per case (gbpf_fdpf.cuh) leaves an SM waiting on the level chain
// of the substitutions and on FP64 instructions.  Here a block keeps the
// solve vectors of K cases side by side in shared memory, so that one read of
// a factor entry, one level's latency and one barrier serve K cases, and the
// nodal work (mismatch, state update, FP64-accurate residual) runs on the
// integer pipe (gbpf_fx.cuh): no FP64 instruction is left on the iteration of
// an FP32 batch, and only the substitutions' multiply-adds on an FP64 one.
//
// The state of the block's cases lies case-fastest, [bus][cases], in the
// per-case scratch of the batch: e + jf as limbs (int4), 1/V, theta, V and
// the specified injections as int64, the right-hand side as double.  Every
// bus must stay in the fixed-point range (fx_state_ok and the steps' checks);
// a case that leaves it, or that wants the Newton-Raphson fallback, is marked
// in `redo` and k_fdpf runs it afterwards.
#pragma once

#include "gbpf_fdpf.cuh"

namespace gbpf {

struct MultiArgs {
    RunArgs r;
    int K = 1;                // cases per block
    int C = 1;                // blocks per case (a cluster; K = 1)
    int *redo = nullptr;      // [ncase] 0 done, 1 k_fdpf from the start, 2 its fallback only
    int2 *x = nullptr;        // [ncase][nbus] refined solutions (FP32)
    void *xg = nullptr;       // [ncase][xs0] solve vectors' rows kept in global memory
    MultiNet net;
    MultiSteps steps[2];
    // arrays of two: by the half-iteration's matrix
    DevMat m[2];
    const void *F[2], *TV[2], *TW[2], *Z[2];
    const double *Kq[2];
    int xs0[2];               // first row of the solve vector in shared memory
    int xstride = 0;          // rows of xg per case
    int zoff = 0;             // its elements there, after which the top's vector lies
    int soff = 0;             // bytes before the sweeps' steps there
};

constexpr int kMultiMax = 4;  // cases per block at most

// Half-iterations after which an outage case by rule goes to its own factors.
// Cases that converge take 13 to 40 here; one that does not would keep its
// block busy up to max_iter, to be run again all the same (one of 512 outages
// on 1,425 buses in FP64: 7 of 21 ms).
constexpr int kOwnLaterHalf = 48;

namespace {

extern __shared__ __align__(128) unsigned char multi_smem[];

// Cases one thread computes of a row: FP32 all K (one 16-byte shared-memory
// access serves four), FP64 one (an FP64 instruction costs its warp 64 cycles
// whatever it does, so lanes are filled with (row, case) pairs).
template <class T, int K>
constexpr int kNc = sizeof(T) == 4 ? K : 1;

template <class T, int NC>
struct alignas(sizeof(T) * NC) Vk {
    T v[NC];
};

// ------------------------------------------------------------ sweeps

// The solve vectors.  kXs: in shared memory.  kXg: rows [xs0, n) in shared
// memory, the rows below (the leaves of a grid too large for it, which a sweep
// touches once or twice) in global memory.  kXc: a cluster's, in global memory
// for the nodal work of all its blocks; the first block brings rows [xs0, n)
// to its shared memory for the sweeps and back (solve_multi).
constexpr int kXs = 0, kXg = 1, kXc = 2;
template <class T, int K, int XG>
struct XVec {
    T *xg;
    int xs0;
    __device__ __forceinline__ T *at(int r) const {
        T *xs = reinterpret_cast<T *>(multi_smem);
        if (XG == kXc) return xg + (long long)r * K;
        if (XG == kXg) return r < xs0 ? xg + (long long)r * K : xs + (r - xs0) * K;
        return xs + r * K;
    }
};

// The threads that share a case's nodal work: first index, stride, barrier.
template <int K, int XG>
__device__ __forceinline__ int first_multi() {
    return XG == kXc ? int(cluster_rank() * blockDim.x + threadIdx.x) : int(threadIdx.x) / K;
}
template <int K, int XG>
__device__ __forceinline__ int step_multi(const MultiArgs &ma) {
    return XG == kXc ? ma.C * int(blockDim.x) : int(blockDim.x) / K;
}
template <int XG>
__device__ __forceinline__ void sync_multi() {
    if (XG == kXc) cluster_sync<2>();
    else __syncthreads();
}

// One substitution sweep: x_r = (dinv ? dinv_r x_r : x_r) - sum over row r's
// entries of val_e x_{idx_e}.  Its steps (MultiSteps, in shared memory) take up
// to a block of rows each, a level in one or several.  The factor is read
// straight from L2 ahead of its use -- a step's entries one step and its row
// ranges two steps before it -- so that a level costs its gathers from shared
// memory and one memory latency at most.  (Staged through shared memory by
// bulk copies, 8 KB at a time and four in flight, the copies' latency bound
// the sweeps: 56 us forward and 47 backward for B' of 10,000 buses, 4 FP32
// cases, by clock stamps; 32 and 41 this way.)  512 threads: more warps add a
// step's fixed instructions, and at 64 registers spills that the small L1
// beside the solve vectors does not hold.
template <class T, int K, int XG>
__device__ __noinline__ void sweep_multi(const int2 *steps, int ns, const int *ptr, const int *idx, const T *val,
                                         const T *dinv, XVec<T, K, XG> x) {
    constexpr int NC = kNc<T, K>, SUB = K / NC;  // lanes per row and entry
    using V = Vk<T, NC>;
    const int slot = int(threadIdx.x) / SUB, k = threadIdx.x % SUB;
    if (ns <= 0) return;
    // {first row | log2 lanes per row << 28, rows | barrier << 31}
    int2 s0 = steps[0], s1 = steps[min(1, ns - 1)], s2;
    int r0, r1, r2;                       // this thread's rows of the steps, -1: none
    int a0 = 0, b0 = 0, a1 = 0, b1 = 0, a2 = 0, b2 = 0;  // their entries
    T d0 = T(1), d1 = T(1), d2 = T(1);
    int i0, i1, j0, j1;                   // the first two entries of the first two
    T v0, v1, u0, u1;
    auto range = [&](const int2 &s, int &r, int &a, int &b, T &d) {
        const int q = slot >> (unsigned(s.x) >> 28);
        r = q < (s.y & 0x7fffffff) ? (s.x & 0xfffffff) + q : -1;
        a = b = 0;
        if (r >= 0) {
            a = ptr[r];
            b = ptr[r + 1];
            if (dinv) d = dinv[r];
        }
    };
    auto entries = [&](const int2 &s, int a, int b, int &ia, int &ib, T &va, T &vb) {
        const int lg = unsigned(s.x) >> 28, G = 1 << lg, e = a + (slot & (G - 1));
        if (e < b) { ia = idx[e]; va = val[e]; }
        if (e + G < b) { ib = idx[e + G]; vb = val[e + G]; }
    };
    range(s0, r0, a0, b0, d0);
    range(s1, r1, a1, b1, d1);
    entries(s0, a0, b0, i0, i1, v0, v1);
    for (int j = 0; j < ns; j++) {
        s2 = steps[min(j + 2, ns - 1)];
        entries(s1, a1, b1, j0, j1, u0, u1);
        range(s2, r2, a2, b2, d2);
        const int G = 1 << (unsigned(s0.x) >> 28), gl = slot & (G - 1);
        if (__any_sync(0xffffffffu, r0 >= 0)) {
            V acc;
#pragma unroll
            for (int c = 0; c < NC; c++) acc.v[c] = T(0);
            auto mac = [&](T w, int i) {
                const V y = *reinterpret_cast<const V *>(x.at(i) + k * NC);
#pragma unroll
                for (int c = 0; c < NC; c++) acc.v[c] = fma(w, y.v[c], acc.v[c]);
            };
            if (a0 + gl < b0) mac(v0, i0);
            if (a0 + G + gl < b0) mac(v1, i1);
            for (int e = a0 + 2 * G + gl; e < b0; e += 2 * G) {  // two entries in flight
                const bool two = e + G < b0;
                const int p = idx[e], q = two ? idx[e + G] : 0;
                const T w = val[e], y = two ? val[e + G] : T(0);
                mac(w, p);
                if (two) mac(y, q);
            }
            for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < NC; c++) acc.v[c] += __shfl_xor_sync(0xffffffffu, acc.v[c], o * SUB);
            if (r0 >= 0 && gl == 0) {
                V &y = *reinterpret_cast<V *>(x.at(r0) + k * NC);
#pragma unroll
                for (int c = 0; c < NC; c++) y.v[c] = dinv ? fma(d0, y.v[c], -acc.v[c]) : y.v[c] - acc.v[c];
            }
        }
        if (s0.y < 0) __syncthreads();
        s0 = s1; r0 = r1; a0 = a1; b0 = b1; d0 = d1;
        i0 = j0; i1 = j1; v0 = u0; v1 = u1;
        s1 = s2; r1 = r2; a1 = a2; b1 = b2; d1 = d2;
    }
}

// One gather through the top's partitioned inverse (tail_inverse_solve): out
// row r = own(r) + sum over its entries val_e in[idx_e], a warp per row and
// four rows at a time, with the entries [ends[r], ends[r + 1]) spread over its
// lanes; a lane holds one row's range for the whole warp and the next rows'
// first entries are read ahead.
template <class T, int K, class Own>
__device__ __forceinline__ void top_gather_multi(const int *ends, const int *idx, const T *val, int nt, const T *in,
                                                 T *out, Own own) {
    constexpr int NC = kNc<T, K>, SUB = K / NC, G = 32 / SUB;
    constexpr int U = 4;
    using V = Vk<T, NC>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = int(blockDim.x >> 5);
    const int k = lane % SUB, gl = lane / SUB;
    int ra = 0, rb = 0;
    int a[U], b[U], i0[U], i1[U];
    T v0[U], v1[U];
    auto fetch = [&](int j) {  // the warp's rows j to j + U - 1
        if (j % 32 == 0) {
            const int r = warp + (j + lane) * nw;
            ra = r < nt ? ends[r] : 0;
            rb = r < nt ? ends[r + 1] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            a[u] = __shfl_sync(0xffffffffu, ra, (j + u) % 32);
            b[u] = __shfl_sync(0xffffffffu, rb, (j + u) % 32);
            if (a[u] + gl < b[u]) { i0[u] = idx[a[u] + gl]; v0[u] = val[a[u] + gl]; }
            if (a[u] + G + gl < b[u]) { i1[u] = idx[a[u] + G + gl]; v1[u] = val[a[u] + G + gl]; }
        }
    };
    fetch(0);
    for (int j = 0; warp + j * nw < nt; j += U) {
        V acc[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
#pragma unroll
            for (int c = 0; c < NC; c++) acc[u].v[c] = T(0);
            auto mac = [&](T l, int i) {
                const V x = *reinterpret_cast<const V *>(in + i * K + k * NC);
#pragma unroll
                for (int c = 0; c < NC; c++) acc[u].v[c] = fma(l, x.v[c], acc[u].v[c]);
            };
            if (a[u] + gl < b[u]) mac(v0[u], i0[u]);
            if (a[u] + G + gl < b[u]) mac(v1[u], i1[u]);
            for (int e = a[u] + 2 * G + gl; e < b[u]; e += 2 * G) {
                const bool two = e + G < b[u];
                const int j0 = idx[e], j1 = two ? idx[e + G] : 0;
                const T l0 = val[e], l1 = two ? val[e + G] : T(0);
                mac(l0, j0);
                if (two) mac(l1, j1);
            }
        }
        fetch(j + U);
#pragma unroll
        for (int u = 0; u < U; u++) {
#pragma unroll
            for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < NC; c++) acc[u].v[c] += __shfl_xor_sync(0xffffffffu, acc[u].v[c], o * SUB);
            const int r = warp + (j + u) * nw;
            if (gl == 0 && r < nt)
#pragma unroll
                for (int c = 0; c < NC; c++) out[r * K + k * NC + c] = acc[u].v[c] + own(r, k * NC + c);
        }
    }
}

// L D L^T x = x for the K cases of x (level order).  With the top's inverse:
// the levels below the top, the top rows' entries below it, the two gathers
// of the top, the levels below it backward.
template <class T, int K, int XG>
__device__ __forceinline__ void solve_block(const MultiArgs &ma, int which, T *z, const XVec<T, K, XG> &x) {
    const DevMat &m = ma.m[which];
    const MultiSteps &st = ma.steps[which];
    const int2 *steps = reinterpret_cast<const int2 *>(multi_smem + ma.soff) + (which ? ma.steps[0].n() : 0);
    const T *F = static_cast<const T *>(ma.F[which]), *Di = F + m.offDi;
    sweep_multi<T, K, XG>(steps, st.nf, m.Fp, m.Fc, F + m.offLr, nullptr, x);
    if (st.np > 0) {
        const T *tv = static_cast<const T *>(ma.TV[which]), *tw = static_cast<const T *>(ma.TW[which]);
        sweep_multi<T, K, XG>(steps + st.nf, st.np, m.PPp, m.PPc, tv + m.tv_p, nullptr, x);
        T *xt = x.at(m.t0);
        top_gather_multi<T, K>(m.twfe, m.twfj, tw, m.nt, xt, z, [&](int r, int c) { return xt[r * K + c]; });
        __syncthreads();
        top_gather_multi<T, K>(m.twbe, m.twbj, tw + m.tw_boff, m.nt, z, xt,
                               [&](int r, int c) { return z[r * K + c] * Di[m.t0 + r]; });
        __syncthreads();
    }
    sweep_multi<T, K, XG>(steps + st.nf + st.np, st.nb, m.Cp, m.Cr, F + m.offLc, Di, x);
}

// The same for a block's or a cluster's cases: the cluster's sweeps run on its
// first block, which copies the rows it keeps in shared memory in and out.
template <class T, int K, int XG>
__device__ __forceinline__ void solve_multi(const MultiArgs &ma, int which, T *z, const XVec<T, K, XG> &x) {
    if constexpr (XG == kXc) {
        if (cluster_rank() == 0) {
            T *xs = reinterpret_cast<T *>(multi_smem);
            const int n = ma.m[which].n - x.xs0;
            for (int r = threadIdx.x; r < n; r += blockDim.x) xs[r] = x.xg[x.xs0 + r];
            __syncthreads();
            solve_block<T, 1, kXg>(ma, which, z, XVec<T, 1, kXg>{x.xg, x.xs0});
            __syncthreads();
            for (int r = threadIdx.x; r < n; r += blockDim.x) x.xg[x.xs0 + r] = xs[r];
        }
        cluster_sync<2>();
    } else {
        solve_block<T, K, XG>(ma, which, z, x);
    }
}

// ------------------------------------------------------------ the block's state

template <int K>
struct alignas(8) MultiShared {  // K = 1: pairs of 8 bytes (totals_multi)
    unsigned long long key[K];  // mismatch maxima
    int left[K];                // a bus left the fixed-point range
    int over[K];                // a mismatch above the tolerance
    unsigned bmax[K], rmax[K];  // FP32 norms (bits) of the right-hand side and the residual
    double s0[K], s1[K];        // low-rank corrections
    int more;                   // cases (bits) that need another correction
};

// All in position order, [position][kk].
struct MultiState {
    int kk;             // cases of this block
    int4 *ef;           // e + jf
    long long *ps, *qs; // specified injections in their bus's units
    long long *th, *vv; // theta, V: units 2^-60
    long long *b;       // right-hand side in its bus's units
    long long *iv;      // 1/V: units 2^-60
    int2 *x;            // refined solution: limbs, units 2^-60
};

// A cluster's maxima: after its barrier every block reads all blocks' words
// and forms the same totals; the words stay until the next barrier.
__device__ __forceinline__ unsigned long long cl_word(const void *p, unsigned rank) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];"
                 : "=l"(v) : "r"(cl_mapa(uint32_t(__cvta_generic_to_shared(p)), rank)) : "memory");
    return v;
}
template <int K, int XG>
__device__ __forceinline__ void totals_multi(const MultiArgs &ma, const MultiShared<K> &sh, MultiShared<K> &tot) {
    if constexpr (XG == kXc) {
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            const unsigned r = lane < ma.C ? unsigned(lane) : 0u;
            unsigned long long w[3];
            w[0] = cl_word(&sh.key[0], r);
            w[1] = cl_word(&sh.left[0], r);  // {left, over}
            w[2] = cl_word(&sh.bmax[0], r);  // {bmax, rmax}
            unsigned v[4] = {unsigned(w[1]), unsigned(w[1] >> 32), unsigned(w[2]), unsigned(w[2] >> 32)};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long q = __shfl_xor_sync(0xffffffffu, w[0], o);
                w[0] = q > w[0] ? q : w[0];
            }
#pragma unroll
            for (int u = 0; u < 4; u++) v[u] = __reduce_max_sync(0xffffffffu, v[u]);
            if (lane == 0) {
                tot.key[0] = w[0];
                tot.left[0] = int(v[0]);
                tot.over[0] = int(v[1]);
                tot.bmax[0] = v[2];
                tot.rmax[0] = v[3];
            }
        }
        __syncthreads();
    }
}

// max over the block's threads of the K lanes' keys into dst (cleared).
template <int K, class U>
__device__ __forceinline__ void lane_max(U v, U *dst) {
#pragma unroll
    for (int o = 16; o >= K; o >>= 1) {
        const U w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    if ((threadIdx.x & 31) < K && v) atomicMax(dst + (threadIdx.x & 31), v);
}

// The mismatch of the cases in `mask` (as cluster_mismatch, the arithmetic of
// fx_bus_current): the right-hand side dP/V or dQ/V in x and, for refinement,
// in st.b; after the next barrier in sh.over whether a bus is above the
// tolerance and, when `full`, the maxima in sh.key.  Bound by the L1's
// accesses, one per 128-byte line a warp's load touches: the row tables and
// the bus's own words are contiguous over the warp's positions, and only the
// neighbours' e + jf are gathered (32 / K lines a load).
template <class T, int K, int XG>
__device__ __forceinline__ void mismatch_multi(const MultiArgs &ma, const MultiState &st, MultiShared<K> &sh,
                                               const XVec<T, K, XG> &x, int c0, int which, bool full, unsigned mask) {
    const RunArgs &a = ma.r;
    const DevNet &dn = a.dn;
    const int nbus = dn.nbus, k = threadIdx.x % K, step = step_multi<K, XG>(ma), kk = st.kk;
    const bool mine = k < kk && ((mask >> k) & 1u);
    int of = -1, ot = -1, outage = mine ? a.dc.outage[c0 + k] : -1;
    if (outage >= 0 && dn.bstatus[outage]) {
        of = dn.bf[outage];
        ot = dn.bt[outage];
    }
    const int2 *esl = ma.net.esl;
    const int4 *ecol = ma.net.ecol, *eY = ma.net.eY, *meta = ma.net.meta;
    const int *row = ma.net.row[which];
    const long long *tol = ma.net.tol;
    const int4 *ef = st.ef + k;
    const bool wantP = full || which == 0, wantQ = full || which == 1;
    const bool keep_b = sizeof(T) == 4 && a.ir_max > 0;
    unsigned long long mx = 0ull;
    unsigned bm = 0u;
    bool over = false;
    // two positions at a time: their loads overlap
    constexpr int U = 2;
    if (mine)
        for (int p0 = first_multi<K, XG>(); p0 < nbus; p0 += U * step) {
            int2 ch[U];
            int4 mt[U], v[U], col[U];
            int r[U], p[U];
            long long ps[U], qs[U], ivi[U], lim[U];
            FxAcc ir[U], ii[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                p[u] = min(p0 + u * step, nbus - 1);  // the last one twice: the same values again
                ch[u] = esl[p[u] >> 5];
                mt[u] = meta[p[u]];
                r[u] = row[p[u]];
                lim[u] = tol[p[u]];
                const int at = p[u] * kk + k;
                ps[u] = wantP ? st.ps[at] : 0;
                qs[u] = wantQ ? st.qs[at] : 0;
                ivi[u] = st.iv[at];
                v[u] = ef[p[u] * kk];
                ir[u] = ii[u] = FxAcc{0, 0};
            }
#pragma unroll
            for (int u = 0; u < U; u++) col[u] = ecol[ch[u].x * 32 + (p[u] & 31)];
            auto term = [&](int u, const int4 &y, const int4 &w) {
                fx_mac(ir[u], y.x, y.y, w.x, w.y);
                fx_mac(ir[u], -y.z, -y.w, w.z, w.w);
                fx_mac(ii[u], y.x, y.y, w.z, w.w);
                fx_mac(ii[u], y.z, y.w, w.x, w.y);
            };
            auto chunk = [&](int u, int c, const int4 &q) {
                const int4 *Y = eY + c * 128 + (p[u] & 31);
                const int4 w0 = ef[q.x * kk], w1 = ef[q.y * kk], w2 = ef[q.z * kk], w3 = ef[q.w * kk];
                const int4 y0 = Y[0], y1 = Y[32], y2 = Y[64], y3 = Y[96];
                term(u, y0, w0);
                term(u, y1, w1);
                term(u, y2, w2);
                term(u, y3, w3);
                fx_carry(ir[u]);
                fx_carry(ii[u]);
            };
#pragma unroll
            for (int u = 0; u < U; u++) chunk(u, ch[u].x, col[u]);
#pragma unroll
            for (int u = 0; u < U; u++) {
                for (int c = ch[u].x + 1; c < ch[u].x + ch[u].y; c++) chunk(u, c, ecol[c * 32 + (p[u] & 31)]);
                const int i = mt[u].x, sc = mt[u].z + 2;
                if (i == of || i == ot) {  // takes the outaged branch's terms out
                    const bool from = i == of;
                    const double *t = dn.bry + 8LL * outage;
                    const int q = mt[u].z;
                    const FxLimbs gs = fx_split(-fx_from_double(t[from ? 0 : 2], q));
                    const FxLimbs bs = fx_split(-fx_from_double(t[from ? 1 : 3], q));
                    const FxLimbs gm = fx_split(-fx_from_double(t[4], q)), bo = fx_split(-fx_from_double(t[5], q));
                    term(u, make_int4(gs.h, gs.l, bs.h, bs.l), v[u]);
                    term(u, make_int4(gm.h, gm.l, bo.h, bo.l), ef[ma.net.pos[from ? ot : of] * kk]);
                }
                const long long cr = fx_sum<3>(ir[u]), ci = fx_sum<3>(ii[u]);
                long long dP = 0, dQ = 0;
                if (wantP && mt[u].y != PF_BUS_SLACK) dP = ps[u] - fx_power(false, v[u], cr, ci);
                if (wantQ && mt[u].y == PF_BUS_PQ) dQ = qs[u] - fx_power(true, v[u], cr, ci);
                const long long ap = dP < 0 ? -dP : dP, aq = dQ < 0 ? -dQ : dQ;
                const long long big = ap > aq ? ap : aq;
                over |= big > lim[u];
                if (full) {
                    const unsigned long long key = abs_key(fx_to_double(big, sc));
                    mx = key > mx ? key : mx;
                }
                if (r[u] >= 0) {
                    // dP / V in the bus's units: the rounding is that of dP itself
                    const FxLimbs g = fx_split(which == 0 ? dP : dQ), h = fx_split(ivi[u]);
                    FxAcc s{0, 0};
                    fx_mac(s, g.h, g.l, h.h, h.l);
                    const long long b = fx_sum<0>(s);
                    if constexpr (sizeof(T) == 4) {
                        const float f = fx_to_float(b, sc);
                        x.at(r[u])[k] = f;
                        if (keep_b) st.b[p[u] * kk + k] = b;
                        const unsigned fb = __float_as_uint(f) & 0x7fffffffu;
                        bm = fb > bm ? fb : bm;
                    } else {
                        x.at(r[u])[k] = fx_to_double(b, sc);
                    }
                    if (big >= (1ll << 60)) sh.left[k] = 1;  // beyond the limbs of d
                }
            }
        }
    if (over) sh.over[k] = 1;
    __syncwarp();
    if (full) lane_max<K>(mx, sh.key);
    if constexpr (sizeof(T) == 4) lane_max<K>(bm, sh.bmax);
}

// x + z0 s0 + z1 s1, each s an unevaluated sum of two floats: the products'
// and sums' errors are carried along, so the result is rounded once, as the
// FP64 form's.
__device__ __forceinline__ float lowrank_add(float x, float z0, float2 s0, float z1, float2 s1) {
    const float p = __fmul_rn(z0, s0.x), pe = fmaf(z0, s0.x, -p) + z0 * s0.y;
    const float q = __fmul_rn(z1, s1.x), qe = fmaf(z1, s1.x, -q) + z1 * s1.y;
    const float s = __fadd_rn(x, p), sb = __fadd_rn(s, -x);
    const float se = __fadd_rn(__fadd_rn(x, -__fadd_rn(s, -sb)), __fadd_rn(p, -sb));
    const float t = __fadd_rn(s, q), tb = __fadd_rn(t, -s);
    const float te = __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -tb)), __fadd_rn(q, -tb));
    return __fadd_rn(t, __fadd_rn(__fadd_rn(se, te), __fadd_rn(pe, qe)));
}
__device__ __forceinline__ double lowrank_add(double x, double z0, double s0, double z1, double s1) {
    return x + z0 * s0 + z1 * s1;
}

// Woodbury correction of the outage cases in `mask` (see LowRank).
template <class T, int K, int XG>
__device__ __forceinline__ void lowrank_multi(const MultiArgs &ma, MultiShared<K> &sh, const MultiState &st,
                                              const XVec<T, K, XG> &x, int c0, int which, unsigned mask) {
    const RunArgs &a = ma.r;
    const T *Zb = static_cast<const T *>(ma.Z[which]);
    if (!Zb) return;
    const DevMat &m = ma.m[which];
    const int n = m.n, k = threadIdx.x % K, step = step_multi<K, XG>(ma);
    const int inst = k < st.kk ? a.dc.inst[c0 + k] : 0;
    const bool on = inst > 0 && ((mask >> k) & 1u);
    if (int(threadIdx.x) < K && on) {
        const int e = a.dc.inst_outage[inst];
        const int p0 = m.br_slot[3 * e], p1 = m.br_slot[3 * e + 1];
        const double y0 = p0 >= 0 ? double(x.at(p0)[k]) : 0.0, y1 = p1 >= 0 ? double(x.at(p1)[k]) : 0.0;
        const double *Kq = ma.Kq[which] + 8LL * inst;
        sh.s0[k] = Kq[0] * y0 + Kq[1] * y1;
        sh.s1[k] = Kq[2] * y0 + Kq[3] * y1;
    }
    sync_multi<XG>();
    if (on) {
        const T *z0 = Zb + (long long)inst * 2 * n, *z1 = z0 + n;
        const double d0 = sh.s0[k], d1 = sh.s1[k];
        if constexpr (sizeof(T) == 4) {
            const float2 f0 = make_float2(float(d0), float(d0 - double(float(d0))));
            const float2 f1 = make_float2(float(d1), float(d1 - double(float(d1))));
            for (int r = first_multi<K, XG>(); r < n; r += step)
                x.at(r)[k] = lowrank_add(x.at(r)[k], z0[r], f0, z1[r], f1);
        } else {
            for (int r = first_multi<K, XG>(); r < n; r += step)
                x.at(r)[k] = lowrank_add(x.at(r)[k], z0[r], d0, z1[r], d1);
        }
    }
    sync_multi<XG>();
}

// FP32: the residual r = b - A x of the cases in `mask`, its norm into
// sh.rmax.  STORED: x = st.x, and r goes into the solve vector as the next
// right-hand side; else x is the FP32 solution in the solve vector, read from
// shared memory, and only the norm is formed.  The rows of A are in fixed
// point on the admittance pattern and x in the units of the state it updates,
// so the residual is as accurate as an FP64 one.
template <int K, int XG, bool STORED>
__device__ __forceinline__ void residual_multi(const MultiArgs &ma, MultiShared<K> &sh, const MultiState &st,
                                               const XVec<float, K, XG> &x, int c0, int which, unsigned mask) {
    const RunArgs &a = ma.r;
    const int nbus = a.dn.nbus, k = threadIdx.x % K, step = step_multi<K, XG>(ma), kk = st.kk;
    const int2 *esl = ma.net.esl, *eA = ma.net.eA[which], *qA = ma.net.qA[which];
    const int4 *ecol = STORED ? ma.net.ecol : ma.net.erow[which];
    const int *row = ma.net.row[which];
    const bool mine = k < kk && ((mask >> k) & 1u);
    unsigned rm = 0u;
    if (mine) {
        const int inst = a.dc.inst[c0 + k];
        const double *Kq = nullptr;
        int p0 = -1, p1 = -1;  // rows of the outaged branch
        if (ma.Z[0] && inst > 0) {
            const int e = a.dc.inst_outage[inst];
            Kq = ma.Kq[which] + 8LL * inst;
            p0 = ma.m[which].br_slot[3 * e];
            p1 = ma.m[which].br_slot[3 * e + 1];
        }
        auto value = [&](int i) {  // x at a position (STORED) or row
            if (STORED) {
                const int2 w = st.x[i * kk + k];
                return FxLimbs{w.x, w.y};
            }
            return fx_limbs60(x.at(i)[k]);
        };
        int left = 0;
        constexpr int U = 2;  // positions at a time
        for (int pb = first_multi<K, XG>(); pb < nbus; pb += U * step) {
            int r[U], p[U];
            int2 ch[U], q[U];
            int4 col[U];
            long long b[U];
            FxAcc s[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                p[u] = min(pb + u * step, nbus - 1);
                r[u] = row[p[u]];
                ch[u] = esl[p[u] >> 5];
                q[u] = qA[p[u]];  // units of the row's sum; their place above the right-hand side's
                b[u] = st.b[p[u] * kk + k];
                s[u] = FxAcc{0, 0};
            }
#pragma unroll
            for (int u = 0; u < U; u++) col[u] = ecol[ch[u].x * 32 + (p[u] & 31)];
            auto chunk = [&](int u, int c, const int4 &o) {
                const int2 *A = eA + c * 128 + (p[u] & 31);
                const int2 a0 = A[0], a1 = A[32], a2 = A[64], a3 = A[96];
                const FxLimbs w0 = value(o.x), w1 = value(o.y), w2 = value(o.z), w3 = value(o.w);
                fx_mac(s[u], a0.x, a0.y, w0.h, w0.l);
                fx_mac(s[u], a1.x, a1.y, w1.h, w1.l);
                fx_mac(s[u], a2.x, a2.y, w2.h, w2.l);
                fx_mac(s[u], a3.x, a3.y, w3.h, w3.l);
                fx_carry(s[u]);
            };
#pragma unroll
            for (int u = 0; u < U; u++) chunk(u, ch[u].x, col[u]);
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (r[u] < 0) continue;
                for (int c = ch[u].x + 1; c < ch[u].x + ch[u].y; c++) chunk(u, c, ecol[c * 32 + (p[u] & 31)]);
                // a right-hand side that the row's units cannot hold leaves
                const int up = min(max(q[u].y, 0), 63), dn = min(max(-q[u].y, 0), 63);
                const long long bs = (b[u] << up) >> dn;
                if (((bs << dn) >> up) != b[u] && up > 0) left = 1;
                long long res = bs - fx_sum<3>(s[u]);
                if (Kq && (r[u] == p0 || r[u] == p1)) {
                    // the outaged branch's share of the base row is added back
                    const int e = a.dc.inst_outage[inst];
                    auto val = [&](int rr, int bus) {
                        if (rr < 0) return 0.0;
                        const FxLimbs w = value(STORED ? ma.net.pos[bus] : rr);
                        return fx_to_double(fx_join(w.h, w.l), 60);
                    };
                    const double x0 = val(p0, a.dn.bf[e]), x1 = val(p1, a.dn.bt[e]);
                    const double share = r[u] == p0 ? Kq[4] * x0 + Kq[6] * x1 : Kq[6] * x0 + Kq[5] * x1;
                    if (!fx_fits(share, q[u].x)) left = 1;
                    res += fx_from_double(share, q[u].x);
                }
                const float f = fx_to_float(res, q[u].x);
                if (STORED) x.at(r[u])[k] = f;
                const unsigned fb = __float_as_uint(f) & 0x7fffffffu;
                rm = fb > rm ? fb : rm;
            }
        }
        if (left) sh.left[k] = 1;
    }
    __syncwarp();
    lane_max<K>(rm, sh.rmax);
    sync_multi<XG>();
}

// st.x = (first ? 0 : st.x) + the FP32 solution in x (0 at positions outside
// the matrix, which the residual's rows read).
template <int K, int XG>
__device__ __forceinline__ void accumulate_multi(const MultiArgs &ma, MultiShared<K> &sh, const MultiState &st,
                                                 const XVec<float, K, XG> &x, int which, bool first, unsigned mask) {
    const int nbus = ma.r.dn.nbus, k = threadIdx.x % K, step = step_multi<K, XG>(ma), kk = st.kk;
    const int *row = ma.net.row[which];
    if (k < kk && ((mask >> k) & 1u)) {
        bool left = false;
        int rn = first_multi<K, XG>() < nbus ? row[first_multi<K, XG>()] : -1;
        for (int p = first_multi<K, XG>(); p < nbus; p += step) {
            const int r = rn, at = p * kk + k;
            if (p + step < nbus) rn = row[p + step];
            if (r >= 0) {
                const float f = x.at(r)[k];
                left |= !(fabsf(f) < 1.75f);
                FxLimbs w = fx_limbs60(f);
                if (!first) {  // the sum keeps the parts' bound: limbs hold less than 2
                    const int2 o = st.x[at];
                    const long long sum = fx_join(w.h, w.l) + fx_join(o.x, o.y);
                    left |= (sum < 0 ? -sum : sum) >= 7ll << 58;
                    w = fx_split(sum);
                }
                st.x[at] = make_int2(w.h, w.l);
            } else if (first) {
                st.x[at] = make_int2(0, 0);
            }
        }
        if (left) sh.left[k] = 1;
    }
    sync_multi<XG>();
}

// The cases of `need` whose residual norm asks for another correction (block-
// uniform; clears the norms).
template <int K, int XG>
__device__ __forceinline__ unsigned more_multi(const MultiArgs &ma, MultiShared<K> &sh, MultiShared<K> &tot,
                                               unsigned need) {
    totals_multi<K, XG>(ma, sh, tot);
    if (threadIdx.x == 0) {
        unsigned more = 0u;
        for (int c = 0; c < K; c++)
            if ((need >> c) & 1u) {
                const double rn = double(__uint_as_float(tot.rmax[c])), bn = double(__uint_as_float(tot.bmax[c]));
                if (rn > ma.r.ir_tol * bn && rn > ma.r.ir_abs && !tot.left[c]) more |= 1u << c;
                if (XG != kXc) sh.rmax[c] = 0u;
            }
        tot.more = int(more);
    }
    sync_multi<XG>();
    if (XG == kXc && threadIdx.x == 0) sh.rmax[0] = 0u;  // read by every block; used after the next solve's barrier
    return unsigned(tot.more);
}

// The whole solve of one half-iteration for the cases in `mask`: x holds the
// right-hand sides.  Returns whether the solutions are in st.x (a correction
// was looked for beyond the first check), else they are in x.  irs counts the
// thread's case's corrections.  A tolerance within an FP32 solve's reach
// (1e-5) is first checked on the solution where it lies: most solves need no
// correction then.
template <class T, int K, int XG>
__device__ __forceinline__ bool halfsolve_multi(const MultiArgs &ma, MultiShared<K> &sh, MultiShared<K> &tot,
                                                const MultiState &st,
                                                const XVec<T, K, XG> &x, T *z, int c0, int which, unsigned mask,
                                                int &irs) {
    const RunArgs &a = ma.r;
    const int k = threadIdx.x % K;
    unsigned need = mask;
#pragma unroll 1
    for (int it = 0;; it++) {
        // the other cases' columns hold right-hand sides nobody reads the
        // solution of: solved along, not used
        solve_multi<T, K, XG>(ma, which, z, x);
        lowrank_multi<T, K, XG>(ma, sh, st, x, c0, which, need);
        if constexpr (sizeof(T) == 8) {
            return false;
        } else {
            if (a.ir_max == 0) return false;
            if (it == 0) {
                if (a.ir_tol >= 1e-5) {
                    residual_multi<K, XG, false>(ma, sh, st, x, c0, which, mask);
                    need = more_multi<K, XG>(ma, sh, tot, mask);
                    if (need == 0u) return false;
                }
                accumulate_multi<K, XG>(ma, sh, st, x, which, true, mask);
            } else {
                accumulate_multi<K, XG>(ma, sh, st, x, which, false, need);
            }
            if (it >= a.ir_max) return true;
            residual_multi<K, XG, true>(ma, sh, st, x, c0, which, need);
            need = more_multi<K, XG>(ma, sh, tot, need);
            if (need == 0u) return true;
            irs += int((need >> k) & 1u);
        }
    }
}

// The state update of the cases in `mask` from the solution.
template <class T, int K, int XG>
__device__ __forceinline__ void update_multi(const MultiArgs &ma, MultiShared<K> &sh, const MultiState &st,
                                             const XVec<T, K, XG> &xv, int which, unsigned mask, bool refined) {
    const RunArgs &a = ma.r;
    const int nbus = a.dn.nbus, k = threadIdx.x % K, step = step_multi<K, XG>(ma);
    const int *row = ma.net.row[which];
    if (!(k < st.kk && ((mask >> k) & 1u))) return;
    int left = 0;
    // the next position's words are read a round ahead: a round's chain is
    // then the arithmetic alone
    long long *sv = which == 0 ? st.th : st.vv;
    int rn = -1;
    int2 xn = make_int2(0, 0);
    long long svn = 0;
    int4 efn = make_int4(0, 0, 0, 0);
    auto ahead = [&](int p) {
        if (p >= nbus) return;
        const int at = p * st.kk + k;
        rn = row[p];
        if (refined) xn = st.x[at];
        svn = sv[at];
        efn = st.ef[at];
    };
    ahead(first_multi<K, XG>());
    for (int p = first_multi<K, XG>(); p < nbus; p += step) {
        const int r = rn, at = p * st.kk + k;
        const int2 w = xn;
        const long long s0 = svn;
        const int4 v = efn;
        ahead(p + step);
        if (r < 0) continue;
        long long d;  // units 2^-60, |d| < 2
        bool ok;
        if (refined) {  // checked as it was summed (accumulate_multi)
            d = fx_join(w.x, w.y);
            ok = true;
        } else {
            const T x = xv.at(r)[k];
            if constexpr (sizeof(T) == 4) {
                ok = fabsf(x) < 1.75f;
                const FxLimbs y = fx_limbs60(ok ? x : 0.0f);
                d = fx_join(y.h, y.l);
            } else {
                ok = fx_fits(x, 60);
                d = ok ? fx_from_double(x, 60) : 0;
            }
        }
        const unsigned long long ad = static_cast<unsigned long long>(d < 0 ? -d : d);
        if (which == 0) {
            const long long t4 = (s0 >> 2) + (d >> 2);  // the sum itself may not fit
            constexpr long long tmax = static_cast<long long>(kFxThMax * 64.0) << 52;
            if (!ok || t4 >= tmax || t4 <= -tmax) {
                left = 1;
                continue;
            }
            const long long t = s0 + d;
            st.th[at] = t;
            if (ad < 230584300921369395ull)  // 0.2
                st.ef[at] = fx_rotate<K>(v, d);
            else
                st.ef[at] = fx_polar60(st.vv[at], t);
        } else {
            const long long vn = s0 + d;
            if (!ok || !fx_v60_ok(vn)) {
                left = 1;
                continue;
            }
            st.vv[at] = vn;
            if (ad < (1ull << 58))
                st.ef[at] = fx_stretch(v, fx_mul60(d, st.iv[at]));
            else
                st.ef[at] = fx_polar60(vn, st.th[at]);
            st.iv[at] = fx_recip((vn + 2) >> 2);
        }
    }
    if (left) sh.left[k] = 1;
}

// ------------------------------------------------------------ kernel

// The whole power flow of the cases c0 .. c0 + K - 1.  sh: the block's words,
// tot: their totals (the same object unless a cluster's).
template <class T, int K, int XG>
__device__ __forceinline__ void multi_cases_run(const MultiArgs &ma, MultiShared<K> &sh, MultiShared<K> &tot, int c0) {
    const RunArgs &a = ma.r;
    const DevNet &dn = a.dn;
    const int nbus = dn.nbus, k = threadIdx.x % K, step = step_multi<K, XG>(ma);
    const int4 *meta = ma.net.meta;
    MultiState st;
    st.kk = min(K, a.dc.ncase - c0);
    {
        const long long nk = (long long)nbus * st.kk;
        double *p = a.ef + (long long)c0 * 4 * nbus, *q = a.xg + (long long)c0 * 3 * nbus;
        st.ef = reinterpret_cast<int4 *>(p);
        st.ps = reinterpret_cast<long long *>(p + 2 * nk);
        st.qs = st.ps + nk;
        st.th = reinterpret_cast<long long *>(q);
        st.vv = st.th + nk;
        st.b = st.vv + nk;
        st.iv = reinterpret_cast<long long *>(a.iv) + (long long)c0 * nbus;
        st.x = ma.x ? ma.x + (long long)c0 * nbus : nullptr;
    }
    const bool mine = k < st.kk;
    const long long cb = (long long)(c0 + k) * nbus;  // the case's vectors
    T *z = reinterpret_cast<T *>(multi_smem) + ma.zoff;  // the top's vector
    auto vec = [&](int w) {
        return XVec<T, K, XG>{XG != kXs ? static_cast<T *>(ma.xg) + (long long)c0 * ma.xstride : nullptr, ma.xs0[w]};
    };
    if (int(threadIdx.x) < K) {
        sh.key[k] = 0ull;
        sh.left[k] = 0;
        sh.bmax[k] = sh.rmax[k] = 0u;
    }
    {
        int2 *steps = reinterpret_cast<int2 *>(multi_smem + ma.soff);
        for (int w = 0; w < 2; w++) {
            for (int t = threadIdx.x; t < ma.steps[w].n(); t += blockDim.x) steps[t] = ma.steps[w].steps[t];
            steps += ma.steps[w].n();
        }
    }
    for (int w = 0; w < 2; w++)  // columns of absent cases are solved along: no stale bits
        for (int r = first_multi<K, XG>(); r < ma.m[w].n; r += step) vec(w).at(r)[k] = T(0);
    sync_multi<XG>();
    if (mine) {
        int left = 0;
        for (int i = first_multi<K, XG>(); i < nbus; i += step) {  // bus order: the caller's vectors are read in runs
            const int p = ma.net.pos[i];
            const int4 mt = meta[p];
            const int t = mt.y;
            const double vm = a.flat ? (t == PF_BUS_PQ ? 1.0 : dn.vset[i]) : a.vm[cb + i];
            const double va = a.flat ? (t == PF_BUS_SLACK ? dn.va0[i] : 0.0) : a.va[cb + i];
            const double psp = a.dc.Psp[cb + i], qsp = a.dc.Qsp[cb + i];
            if (!fx_state_ok(dn, i, vm, va, psp, qsp)) {
                left = 1;
                continue;
            }
            const int at = p * st.kk + k, sc = mt.z + 2;
            st.ps[at] = fx_from_double(psp, sc);
            st.qs[at] = fx_from_double(qsp, sc);
            st.th[at] = fx_from_double(va, 60);
            st.vv[at] = fx_from_double(vm, 60);
            st.ef[at] = fx_polar(vm, va);
            st.iv[at] = fx_recip(fx_from_double(vm, kFxV));
        }
        if (left) sh.left[k] = 1;
    }
    sync_multi<XG>();
    int status = PF_ERR_NOT_CONVERGED;  // of the thread's case, like the next three
    if (a.fs0[0] != PF_OK) status = a.fs0[0];
    else if (a.fs1[0] != PF_OK) status = a.fs1[0];
    int iters = 0, irs = 0, redo = 0;
    double mis = INFINITY;
    bool rotated = false;
    unsigned active = status == PF_ERR_NOT_CONVERGED ? (1u << st.kk) - 1u : 0u;
    totals_multi<K, XG>(ma, sh, tot);
    for (int c = 0; c < st.kk; c++)
        if (tot.left[c]) active &= ~(1u << c);
    if (mine && tot.left[k]) redo = 1;
    if (a.own_now)
        for (int c = 0; c < st.kk; c++)
            if (a.own_now[c0 + c]) active &= ~(1u << c);
#pragma unroll 1
    for (int h = 0; active; h++) {
        if (h == kOwnLaterHalf && a.own_now) {
            for (int c = 0; c < st.kk; c++)
                if (a.dc.inst[c0 + c] > 0) active &= ~(1u << c);
            if (!active) break;
        }
        // after the last half-iteration: a full evaluation alone
        const bool last = h >= 2 * a.max_iter;
        const int which = last ? 0 : h & 1;
        // the mismatch of this half; for cases at or below the tolerance
        // again in full at the exact state (e + jf from theta and V), which
        // decides.  Cases that converged, or left the fixed-point range,
        // leave `active`.
        unsigned mask = active;
#pragma unroll 1
        for (int full = 0; full < 2 && mask; full++) {
            if (full && rotated && mine && ((mask >> k) & 1u))
                for (int p = first_multi<K, XG>(); p < nbus; p += step) {
                    const int at = p * st.kk + k;
                    st.ef[at] = fx_polar60(st.vv[at], st.th[at]);
                }
            if (int(threadIdx.x) < K && ((mask >> k) & 1u)) {
                sh.key[k] = 0ull;
                sh.bmax[k] = 0u;
                sh.over[k] = 0;
            }
            sync_multi<XG>();
            mismatch_multi<T, K, XG>(ma, st, sh, vec(which), c0, which, full != 0, mask);
            sync_multi<XG>();
            totals_multi<K, XG>(ma, sh, tot);
            unsigned check = 0u;
            for (int c = 0; c < st.kk; c++) {
                if (!((mask >> c) & 1u)) continue;
                const bool in_tol =
                    full ? __longlong_as_double(static_cast<long long>(tot.key[c])) <= a.tol : tot.over[c] == 0;
                if (tot.left[c] || (full && in_tol)) active &= ~(1u << c);
                else if (!full && (in_tol || last)) check |= 1u << c;
            }
            if (mine && ((mask >> k) & 1u)) {
                if (full) mis = __longlong_as_double(static_cast<long long>(tot.key[k]));
                if (!((active >> k) & 1u)) {
                    if (tot.left[k]) redo = 1;
                    else status = PF_OK;
                }
            }
            sync_multi<XG>();
            mask = check;
        }
        if (last || !active) break;
        const bool refined = halfsolve_multi<T, K, XG>(ma, sh, tot, st, vec(which), z, c0, which, active, irs);
        update_multi<T, K, XG>(ma, sh, st, vec(which), which, active, refined);
        rotated = true;
        if ((active >> k) & 1u) iters++;
        sync_multi<XG>();
    }
    sync_multi<XG>();
    if (!mine) return;
    if (redo == 0 && status != PF_OK && a.fallback && status == PF_ERR_NOT_CONVERGED) redo = 2;
    const bool later = a.own_now && a.dc.inst[c0 + k] > 0 && status != PF_OK;  // the status tells the host
    if (later) redo = 0;
    if (int(threadIdx.x) < K && (XG != kXc || cluster_rank() == 0)) {
        ma.redo[c0 + k] = redo;
        if (redo == 0) {
            pf_case_result &o = a.res[c0 + k];
            o.status = status;
            o.iters = iters;
            o.ir_steps = irs;
            o.method = PF_FDPF;
            o.max_mismatch = mis;
        }
    }
    if (redo == 1 || later) return;  // the start state stays as it was
    for (int i = first_multi<K, XG>(); i < nbus; i += step) {
        const int p = ma.net.pos[i], t = meta[p].y, at = p * st.kk + k;
        if (ma.net.row[1][p] >= 0) a.vm[cb + i] = fx_to_double(st.vv[at], 60);
        else if (a.flat) a.vm[cb + i] = t == PF_BUS_PQ ? 1.0 : dn.vset[i];
        if (ma.net.row[0][p] >= 0) a.va[cb + i] = fx_to_double(st.th[at], 60);
        else if (a.flat) a.va[cb + i] = t == PF_BUS_SLACK ? dn.va0[i] : 0.0;
    }
}

template <class T, int K, int XG>
__global__ void __launch_bounds__(kMultiThreads, 1) k_fdpf_multi(const __grid_constant__ MultiArgs ma) {
    __shared__ MultiShared<K> sh;
    multi_cases_run<T, K, XG>(ma, sh, sh, int(blockIdx.x) * K);
}

// One case per cluster of ma.C blocks: the nodal work -- mismatch, residual,
// update, three quarters of an iteration on one block -- over all of them, the
// sweeps on the first, whose level chain bounds it then.  The sums are those of
// one block; the iterates may differ in the last bits (fx_rotate's choice by
// warp).  One FP32 case of 40,000 buses,
// refined to 1e-10, factors included: 10.9 ms on one block, 7.1 on 16.
template <class T>
__global__ void __launch_bounds__(kMultiThreads, 1) k_fdpf_multi_cl(const __grid_constant__ MultiArgs ma) {
    __shared__ MultiShared<1> sh, tot;
    multi_cases_run<T, 1, kXc>(ma, sh, tot, int(blockIdx.x) / ma.C);
    cluster_sync<2>();  // the blocks' words are read until here
}

// The grids of a pack, one per block (kXg) or cluster (kXc) at a time: they
// are taken from a counter in the order given (largest first).  The grid's
// arguments are copied to shared memory.
template <class T, int XG>
__global__ void __launch_bounds__(kMultiThreads, 1)
    k_fdpf_multi_pack(const MultiArgs *args, const int *order, int ngrid, unsigned *counter) {
    __shared__ MultiShared<1> sh, tot;
    __shared__ __align__(16) unsigned char raw[sizeof(MultiArgs)];
    __shared__ __align__(8) int next[2];
    const MultiArgs &ma = *reinterpret_cast<const MultiArgs *>(raw);
    for (;;) {
        if (threadIdx.x == 0 && (XG != kXc || cluster_rank() == 0)) {
            const unsigned q = atomicAdd(counter, 1u);
            next[0] = q < unsigned(ngrid) ? order[q] : -1;
        }
        sync_multi<XG>();
        const int g = XG == kXc ? int(unsigned(cl_word(next, 0))) : next[0];
        if (g < 0) break;
        const int *src = reinterpret_cast<const int *>(args + g);
        for (int t = threadIdx.x; t < int(sizeof(MultiArgs) / 4); t += blockDim.x) reinterpret_cast<int *>(raw)[t] = src[t];
        __syncthreads();
        if (ma.K > 0) multi_cases_run<T, 1, XG>(ma, sh, XG == kXc ? tot : sh, 0);
        sync_multi<XG>();
    }
    sync_multi<XG>();  // the first block's words are read until here
}

// k_lowrank_z (the columns of Z = A^-1 U of the outage instances) with the
// solves of K columns per block on the planned sweeps: a column per block on
// the staged sweeps took 669 us for 512 outages of 10,000 buses in FP32.
template <class T, int K>
__global__ void __launch_bounds__(kMultiThreads, 1)
    k_lowrank_z_multi(const __grid_constant__ MultiArgs ma, int which, T *Z) {
    const DevMat &m = ma.m[which];
    const DevCases &dc = ma.r.dc;
    const int n = m.n, k = threadIdx.x % K, c0 = int(blockIdx.x) * K, ncol = 2 * (dc.ninst - 1);
    int2 *steps = reinterpret_cast<int2 *>(multi_smem + ma.soff);
    for (int w = 0; w < 2; w++) {
        for (int t = threadIdx.x; t < ma.steps[w].n(); t += blockDim.x) steps[t] = ma.steps[w].steps[t];
        steps += ma.steps[w].n();
    }
    int p = -1;
    if (c0 + k < ncol) {
        const int e = dc.inst_outage[1 + (c0 + k) / 2];
        if (e >= 0 && ma.r.dn.bstatus[e]) p = m.br_slot[3 * e + (c0 + k) % 2];
    }
    const XVec<T, K, kXs> x{nullptr, 0};
    for (int r = int(threadIdx.x) / K; r < n; r += int(blockDim.x) / K) x.at(r)[k] = T(r == p ? 1 : 0);
    __syncthreads();
    solve_block<T, K, kXs>(ma, which, reinterpret_cast<T *>(multi_smem) + ma.zoff, x);
    __syncthreads();
    for (int c = 0; c < K && c0 + c < ncol; c++)
        for (int r = threadIdx.x; r < n; r += blockDim.x) Z[(2LL + c0 + c) * n + r] = x.at(r)[c];
}

// A launch in clusters of C blocks (C = 1: plain) with `smem` bytes each.
template <class... P, class... A>
cudaError_t launch_clustered(void (*k)(P...), int blocks, int C, size_t smem, cudaStream_t s, const A &...args) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(blocks));
    cfg.blockDim = dim3(kMultiThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(C);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// Clusters of C blocks that can be resident at once.
template <class T>
int multi_clusters_t(int C, size_t smem) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(C));
    cfg.blockDim = dim3(kMultiThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(C);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int least = 1 << 30;
    auto active = [&](auto *k) {
        int n = 0;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k, &cfg);
        if (e != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        least = n < least ? n : least;
    };
    active(k_fdpf_multi_cl<T>);
    active(k_fdpf_multi_pack<T, kXc>);
    return least;
}

template <class T>
cudaError_t multi_pack_t(const MultiArgs *args, const int *order, int ngrid, unsigned *counter, size_t smem, int groups,
                         int C, cudaStream_t s) {
    return launch_clustered(C > 1 ? k_fdpf_multi_pack<T, kXc> : k_fdpf_multi_pack<T, kXg>, groups * C, C, smem, s, args,
                            order, ngrid, counter);
}

template <class T>
cudaError_t multi_run_t(const MultiArgs &a, size_t smem, cudaStream_t s) {
    const int blocks = (a.r.dc.ncase + a.K - 1) / a.K * a.C;
    auto *k = a.C > 1 ? k_fdpf_multi_cl<T>
              : a.K == 4 ? k_fdpf_multi<T, 4, kXs>
              : a.K == 2 ? k_fdpf_multi<T, 2, kXs>
              : a.xs0[0] > 0 || a.xs0[1] > 0 ? k_fdpf_multi<T, 1, kXg> : k_fdpf_multi<T, 1, kXs>;
    return launch_clustered(k, blocks, a.C, smem, s, a);
}

template <class T>
cudaError_t multi_lowrank_t(const MultiArgs &a, int which, void *Z, size_t smem, cudaStream_t s) {
    auto *k = a.K == 4 ? k_lowrank_z_multi<T, 4> : a.K == 2 ? k_lowrank_z_multi<T, 2> : k_lowrank_z_multi<T, 1>;
    return launch_clustered(k, (2 * (a.r.dc.ninst - 1) + a.K - 1) / a.K, 1, smem, s, a, which, static_cast<T *>(Z));
}

}  // namespace

cudaError_t multi_lowrank_f64(const MultiArgs &a, int which, void *Z, size_t smem, cudaStream_t s);
cudaError_t multi_lowrank_f32(const MultiArgs &a, int which, void *Z, size_t smem, cudaStream_t s);
int multi_clusters_f64(int C, size_t smem);
int multi_clusters_f32(int C, size_t smem);
cudaError_t multi_run_f64(const MultiArgs &a, size_t smem, cudaStream_t s);
cudaError_t multi_run_f32(const MultiArgs &a, size_t smem, cudaStream_t s);
cudaError_t multi_pack_f64(const MultiArgs *args, const int *order, int ngrid, unsigned *counter, size_t smem,
                           int groups, int C, cudaStream_t s);
cudaError_t multi_pack_f32(const MultiArgs *args, const int *order, int ngrid, unsigned *counter, size_t smem,
                           int groups, int C, cudaStream_t s);

}  // namespace gbpf

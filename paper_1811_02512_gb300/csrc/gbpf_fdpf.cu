// gbpf_fdpf.cu -- launchers of the power-flow iteration kernels
// (gbpf_fdpf.cuh; the kernels themselves are instantiated per precision in
// gbpf_fdpf64.cu and gbpf_fdpf32.cu).
#include "gbpf_fdpf.cuh"
#include "gbpf_multi.cuh"

namespace gbpf {

namespace {
// The sliced rows of a MultiNet from the current admittance matrix, a thread
// per position: the fixed-point admittances, and with `refine` the rows of B'
// and B'' (entries joining two of the matrix's buses) in units that take the
// row's sum of magnitudes to at most 2^58.
__global__ void k_multi_rows(DevNet dn, MultiNet N, int refine, double tol) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= dn.nbus) return;
    const int2 ch = N.esl[p >> 5];
    const int sl = p & 31, unit = N.meta[p].z + 2;  // the mismatch's units
    N.tol[p] = fx_fits(tol, unit) ? fx_from_double(tol, unit) : 1ll << 62;
    for (int c = ch.x; c < ch.x + ch.y; c++)
        for (int u = 0; u < 4; u++) {
            const int q = N.esrc[(4 * c + u) * 32 + sl];
            N.eY[(4 * c + u) * 32 + sl] = q >= 0 ? dn.Yx[q] : make_int4(0, 0, 0, 0);
        }
    if (!refine) return;
    for (int w = 0; w < 2; w++) {
        auto value = [&](int c, int u) {
            const int q = N.esrc[(4 * c + u) * 32 + sl];
            const int4 col = N.ecol[c * 32 + sl];
            const int o = u == 0 ? col.x : u == 1 ? col.y : u == 2 ? col.z : col.w;
            if (q < 0 || N.row[w][p] < 0 || N.row[w][o] < 0) return 0.0;
            return w == 0 ? dn.Bp[q] : -dn.B[q];
        };
        double l1 = 0.0;
        for (int c = ch.x; c < ch.x + ch.y; c++)
            for (int u = 0; u < 4; u++) l1 += fabs(value(c, u));
        const int ex = int((unsigned(__double2hiint(l1)) >> 20) & 0x7ffu) - 1022;  // l1 < 2^ex
        const int sc = kFxRow - min(max(ex, -400), 400);
        N.qA[w][p] = make_int2(sc + 3, sc + 3 - unit);
        for (int c = ch.x; c < ch.x + ch.y; c++)
            for (int u = 0; u < 4; u++) {
                const FxLimbs v = fx_split(fx_from_double(value(c, u), sc));
                N.eA[w][(4 * c + u) * 32 + sl] = make_int2(v.h, v.l);
            }
    }
}
}  // namespace

// ------------------------------------------------------------ launchers

cudaError_t launch_fdpf_pack(const RunArgs *args_dev, const int *order_dev, int ngrid,
                             unsigned *counter_dev, int prec, size_t smem, int nsm, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(counter_dev, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const int blocks = ngrid < nsm ? ngrid : nsm;
    return prec == PF_FP64 ? fdpf_pack_f64(args_dev, order_dev, ngrid, counter_dev, smem, blocks, s)
                           : fdpf_pack_f32(args_dev, order_dev, ngrid, counter_dev, smem, blocks, s);
}

// Fills the run arguments of one grid of a pack (the single-case form of
// launch_fdpf's arguments); use_smem is decided by the caller.
void fill_run_args(RunArgs &a, const DevNet &dn, const DevCases &dc, const DevMat *m, const void *F0,
                   const void *F1, const void *TV0, const void *TV1, const double *A0,
                   const double *A1, const int *fstat0, const int *fstat1, const pf_run_opts &o,
                   double *vm, double *va, double *ef, double *iv, double *xg, double *bmax,
                   pf_case_result *res) {
    a.TV0 = m[0].npf2 > 0 ? TV0 : nullptr;
    a.TV1 = m[1].npf2 > 0 ? TV1 : nullptr;
    a.TW0 = a.TW1 = nullptr;
    a.Z0 = a.Z1 = nullptr;
    a.K0 = a.K1 = nullptr;
    a.iv = iv;
    a.A0 = A0;
    a.A1 = A1;
    a.ir_max = o.ir_max;
    a.ir_tol = o.ir_tol;
    a.ir_abs = o.ir_abs > 0 ? o.ir_abs : 0.01 * o.tol;
    a.dn = dn;
    a.dc = dc;
    a.m0 = m[0];
    a.m1 = m[1];
    a.F0 = F0;
    a.F1 = F1;
    a.fs0 = fstat0;
    a.fs1 = fstat1;
    a.tol = o.tol;
    a.max_iter = o.max_iter;
    a.flat = o.flat_start;
    a.spin = o.spin_limit > 0 ? unsigned(o.spin_limit) : kDefaultSpin;
    a.vm = vm;
    a.va = va;
    a.ef = ef;
    a.xg = xg;
    a.bmax = bmax;
    a.res = res;
    a.use_smem = 0;
    a.fallback = 0;
    a.redo = a.list = a.own_now = nullptr;
    a.nlist = 0;
}

size_t run_args_bytes() { return sizeof(RunArgs); }

size_t fill_multi_args(MultiArgs &ma, const RunArgs &a, const MultiLaunch &ml, const DevMat *m, const void *Z0,
                       const void *Z1, const double *K0, const double *K1, int prec);

cudaError_t launch_pack(const PackGrid *grids, int ngrid, int prec, const pf_run_opts &o,
                        const int *order_host, void *args_dev, void *margs_dev, int *order_dev, unsigned *counter_dev,
                        size_t smem_optin, int nsm, cudaStream_t s) {
    // the launch reserves shared memory for the largest grid whose solve
    // vector fits; larger grids keep theirs in global scratch
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float);
    const size_t ring = size_t(kStages) * kStageBytes;
    int ns = 0;
    for (int g = 0; g < ngrid; g++) {
        const int nm = grids[g].m[0].n > grids[g].m[1].n ? grids[g].m[0].n : grids[g].m[1].n;
        if (ring + elt * size_t(nm) + 2048 <= smem_optin && nm > ns) ns = nm;
    }
    std::vector<RunArgs> A(static_cast<size_t>(ngrid));
    for (int g = 0; g < ngrid; g++) {
        const PackGrid &p = grids[g];
        fill_run_args(A[g], p.dn, p.dc, p.m, p.F0, p.F1, p.TV0, p.TV1, p.A0, p.A1, p.fs0, p.fs1, o,
                      p.vm, p.va, p.ef, p.iv, p.xg, p.bmax, p.res);
        const int nm = p.m[0].n > p.m[1].n ? p.m[0].n : p.m[1].n;
        A[g].use_smem = nm <= ns;
        A[g].TW0 = p.m[0].npf3 > 0 && A[g].TV0 ? p.TW0 : nullptr;
        A[g].TW1 = p.m[1].npf3 > 0 && A[g].TV1 ? p.TW1 : nullptr;
    }
    // the several-cases-per-block kernel, one grid per block, takes every grid
    // it fits; k_fdpf_pack below the others and what it left
    std::vector<MultiArgs> M(static_cast<size_t>(ngrid));
    size_t msmem = 0;
    bool any = false, wide = true;
    int nbus_max = 0;
    for (int g = 0; g < ngrid; g++) {
        const PackGrid &p = grids[g];
        M[g].K = 0;
        if (p.ml.K > 0) {
            const size_t need = fill_multi_args(M[g], A[g], p.ml, p.m, nullptr, nullptr, nullptr, nullptr, prec);
            if (need + sizeof(MultiArgs) + 1024 > smem_optin) {
                M[g].K = 0;
            } else {
                msmem = need > msmem ? need : msmem;
                any = true;
                wide = wide && p.ml.C > 1;  // its solve vector has room for a cluster's
                nbus_max = p.dn.nbus > nbus_max ? p.dn.nbus : nbus_max;
                A[g].redo = p.ml.redo;
                k_multi_rows<<<(p.dn.nbus + 127) / 128, 128, 0, s>>>(p.dn, p.ml.net, prec == PF_FP32 && o.ir_max > 0, o.tol);
            }
        }
        A[g].TW0 = A[g].TW1 = nullptr;
    }
    const int C = any && wide ? multi_cluster_size(ngrid, nbus_max, nsm, prec, msmem) : 1;
    for (MultiArgs &x : M) x.C = C;
    cudaError_t e = cudaMemcpyAsync(args_dev, A.data(), sizeof(RunArgs) * size_t(ngrid),
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(order_dev, order_host, sizeof(int) * size_t(ngrid), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && any)
        e = cudaMemcpyAsync(margs_dev, M.data(), sizeof(MultiArgs) * size_t(ngrid), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // A and M are released on return
    if (e != cudaSuccess) return e;
    if (any) {
        e = cudaMemsetAsync(counter_dev, 0, sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
        const int blocks = ngrid < nsm ? ngrid : nsm;
        const MultiArgs *ma = static_cast<const MultiArgs *>(margs_dev);
        e = prec == PF_FP64 ? multi_pack_f64(ma, order_dev, ngrid, counter_dev, msmem, blocks, C, s)
                            : multi_pack_f32(ma, order_dev, ngrid, counter_dev, msmem, blocks, C, s);
        if (e != cudaSuccess) return e;
    }
    return launch_fdpf_pack(static_cast<const RunArgs *>(args_dev), order_dev, ngrid, counter_dev, prec,
                            ring + elt * size_t(ns), nsm, s);
}

// The arguments of the several-cases-per-block kernel from those of k_fdpf;
// returns its dynamic shared memory.
size_t fill_multi_args(MultiArgs &ma, const RunArgs &a, const MultiLaunch &ml, const DevMat *m, const void *Z0,
                       const void *Z1, const double *K0, const double *K1, int prec) {
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float);
    const int nmax = m[0].n > m[1].n ? m[0].n : m[1].n, nt = m[0].nt > m[1].nt ? m[0].nt : m[1].nt;
    ma.r = a;
    ma.K = ml.K;
    ma.C = ml.C;
    ma.redo = ml.redo;
    ma.net = ml.net;
    ma.x = ml.x;
    ma.xg = ml.xg;
    for (int w = 0; w < 2; w++) {
        ma.steps[w] = ml.steps[w];
        ma.m[w] = m[w];
        ma.F[w] = w == 0 ? a.F0 : a.F1;
        ma.TV[w] = w == 0 ? a.TV0 : a.TV1;
        ma.TW[w] = w == 0 ? a.TW0 : a.TW1;
        ma.Z[w] = w == 0 ? Z0 : Z1;
        ma.Kq[w] = w == 0 ? K0 : K1;
        ma.xs0[w] = m[w].n > nmax - ml.xs0 ? m[w].n - (nmax - ml.xs0) : 0;
    }
    ma.xstride = ma.C > 1 ? nmax : ma.xs0[0] > ma.xs0[1] ? ma.xs0[0] : ma.xs0[1];
    ma.zoff = ((nmax - ml.xs0) * ma.K + 3) & ~3;  // 16-byte accesses
    ma.soff = int((elt * (size_t(ma.zoff) + size_t(nt) * size_t(ma.K)) + 15) & ~size_t(15));
    return multi_smem_bytes(ml, m, prec);
}

cudaError_t launch_lowrank_z_multi(const MultiLaunch &ml, const DevNet &dn, const DevCases &dc, const DevMat *m, int which,
                                   int prec, const void *F, const void *TV, const void *TW, void *Z, cudaStream_t s) {
    RunArgs r = {};
    r.dn = dn;
    r.dc = dc;
    (which == 0 ? r.F0 : r.F1) = F;
    (which == 0 ? r.TV0 : r.TV1) = TV;
    (which == 0 ? r.TW0 : r.TW1) = TW;
    MultiArgs ma;
    const size_t smem = fill_multi_args(ma, r, ml, m, nullptr, nullptr, nullptr, nullptr, prec);
    return prec == PF_FP64 ? multi_lowrank_f64(ma, which, Z, smem, s) : multi_lowrank_f32(ma, which, Z, smem, s);
}

size_t multi_smem_bytes(const MultiLaunch &ml, const DevMat *m, int prec) {
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float);
    const int nmax = m[0].n > m[1].n ? m[0].n : m[1].n, nt = m[0].nt > m[1].nt ? m[0].nt : m[1].nt;
    const size_t zoff = size_t((nmax - ml.xs0) * ml.K + 3) & ~size_t(3);
    const size_t soff = (elt * (zoff + size_t(nt) * size_t(ml.K)) + 15) & ~size_t(15);
    return soff + sizeof(int2) * size_t(ml.steps[0].n() + ml.steps[1].n());
}

// A case alone on a block leaves the chip idle: 16 or 8 blocks share its nodal
// work while every case has its cluster at once.  The line: the cluster
// barriers, about ten a half-iteration, cost what that saves at some 2,000
// buses (one FP32 case, ir_tol 1e-10, cluster against block: 0.71 ms against
// 0.57 on 1,000 buses, 0.88 against 0.85 on 2,000, 1.08 against 1.18 on 3,000,
// 1.92 against 2.66 on 10,000, 7.1 against 10.9 on 40,000; FP64 8.6 against
// 12.3 on 40,000; nine cases of 10,000 buses 2.05 against 2.66).
int multi_cluster_size(int groups, int nbus, int num_sms, int prec, size_t smem, int most) {
    constexpr int kMultiClBuses = 2500;
    if (most == 0 && nbus < kMultiClBuses) return 1;
    for (int C : {16, 8})
        if ((most == 0 || C <= most) && groups * C <= num_sms &&
            (prec == PF_FP64 ? multi_clusters_f64(C, smem) : multi_clusters_f32(C, smem)) >= groups)
            return C;
    return 1;
}

size_t multi_args_bytes() { return sizeof(MultiArgs); }

// Cluster size of the power-flow kernel: a case spreads its nodal work over
// 16 (or 8) SMs when the batch is too small to fill the GPU with one block per
// case and such clusters can be resident; otherwise one block per case.
int fdpf_cluster_size(int ncase, int num_sms, int prec, size_t smem_optin, int nmax) {
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float);
    size_t smem = size_t(kStages) * kStageBytes + elt * size_t(nmax);
    if (smem + 2048 > smem_optin) smem = size_t(kStages) * kStageBytes;
    for (int C : {16, 8}) {
        if (ncase * C > num_sms) continue;
        if (prec == PF_FP64 ? fdpf_clusters_fit_f64(C, ncase, smem) : fdpf_clusters_fit_f32(C, ncase, smem))
            return C;
    }
    return 1;
}

cudaError_t launch_fdpf(const DevNet &dn, const DevCases &dc, const DevMat *m, int prec,
                        const void *F0, const void *F1, const void *TV0, const void *TV1,
                        const double *A0, const double *A1, const int *fstat0, const int *fstat1,
                        const pf_run_opts &o, double *vm, double *va, double *ef, double *iv,
                        double *xg, double *bmax, pf_case_result *res, size_t smem_optin,
                        size_t smem_per_sm, int cluster, int threads, cudaStream_t s, const void *Z0,
                        const void *Z1, const double *K0, const double *K1, const NrLaunch *fb,
                        const void *TW0, const void *TW1, const MultiLaunch *multi, const int *list, int nlist) {
    RunArgs a;
    a.redo = nullptr;
    a.list = list;
    a.nlist = nlist;
    a.own_now = multi && multi->K > 0 ? multi->own_now : nullptr;
    a.Z0 = Z0;
    a.Z1 = Z1;
    a.K0 = K0;
    a.K1 = K1;
    a.TV0 = m[0].npf2 > 0 ? TV0 : nullptr;
    a.TV1 = m[1].npf2 > 0 ? TV1 : nullptr;
    a.TW0 = m[0].npf3 > 0 && a.TV0 ? TW0 : nullptr;
    a.TW1 = m[1].npf3 > 0 && a.TV1 ? TW1 : nullptr;
    a.iv = iv;
    a.A0 = A0;
    a.A1 = A1;
    a.ir_max = o.ir_max;
    a.ir_tol = o.ir_tol;
    a.ir_abs = o.ir_abs > 0 ? o.ir_abs : 0.01 * o.tol;
    a.dn = dn;
    a.dc = dc;
    a.m0 = m[0];
    a.m1 = m[1];
    a.F0 = F0;
    a.F1 = F1;
    a.fs0 = fstat0;
    a.fs1 = fstat1;
    a.tol = o.tol;
    a.max_iter = o.max_iter;
    a.flat = o.flat_start;
    a.spin = o.spin_limit > 0 ? unsigned(o.spin_limit) : kDefaultSpin;
    a.vm = vm;
    a.va = va;
    a.ef = ef;
    a.xg = xg;
    a.bmax = bmax;
    a.res = res;
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float);
    const int nmax = m[0].n > m[1].n ? m[0].n : m[1].n;
    const size_t ring = size_t(kStages) * kStageBytes;
    size_t smem = ring + elt * size_t(nmax);
    a.use_smem = smem + 2048 <= smem_optin;
    // one block per case with fewer threads: as many blocks per SM as the
    // registers allow (64 per thread), the solve vector in shared memory
    // only when it does not lower that count
    if (cluster > 1 || (threads != 256 && threads != 128)) threads = kRunThreads;
    if (threads < kRunThreads) {
        const size_t blocks = size_t(65536 / (threads * 64)) < size_t(2048 / threads)
                                  ? size_t(65536 / (threads * 64)) : size_t(2048 / threads);
        const size_t budget = smem_per_sm / blocks;
        a.use_smem = smem + 2048 <= budget && smem + 2048 <= smem_optin;
    }
    if (!a.use_smem) smem = ring;
    a.fallback = 0;
    if (fb) {  // the Newton-Raphson fallback's factor scratch, when it fits
        const size_t need = nr_args_within(*fb, smem, a.nr);
        if (need + 2048 <= smem_optin) {
            smem = need;
            a.fallback = 1;
        }
    }
    if (multi && multi->K > 0) {
        // several cases per block first; the launch below takes what it left
        MultiArgs ma;
        const size_t ms = fill_multi_args(ma, a, *multi, m, Z0, Z1, K0, K1, prec);
        if (ms + 1024 > smem_optin) return cudaErrorInvalidConfiguration;
        k_multi_rows<<<(dn.nbus + 127) / 128, 128, 0, s>>>(dn, ma.net, prec == PF_FP32 && o.ir_max > 0, o.tol);
        const cudaError_t e = prec == PF_FP64 ? multi_run_f64(ma, ms, s) : multi_run_f32(ma, ms, s);
        if (e != cudaSuccess) return e;
        a.redo = multi->redo;
    }
    return prec == PF_FP64 ? fdpf_run_f64(a, smem, cluster, threads, s)
                           : fdpf_run_f32(a, smem, cluster, threads, s);
}

// Rows of one case's solve vector that may lie in global memory: those below
// the narrow top, and at most half of them all.
static bool multi_rows_out(const DevMat *m, long long x) {
    const int nmax = m[0].n > m[1].n ? m[0].n : m[1].n;
    return x <= m[0].n - m[0].nt && x <= m[1].n && 2 * x <= nmax;
}

bool multi_fit(MultiLaunch &ml, const DevMat *m, int prec, size_t room) {
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float), need = multi_smem_bytes(ml, m, prec);
    if (need <= room) return true;
    const long long x = ml.xs0 + (long long)((need - room) / elt) + 8;  // the sizes are rounded up
    if (ml.K != 1 || !multi_rows_out(m, x)) return false;
    ml.xs0 = int(x);
    return multi_smem_bytes(ml, m, prec) <= room;
}

int multi_cases(const DevMat *m, int prec, int ncase, int num_sms, size_t smem_optin, int *xs0) {
    const size_t elt = prec == PF_FP64 ? sizeof(double) : sizeof(float);
    const int nmax = m[0].n > m[1].n ? m[0].n : m[1].n;
    const int nt = m[0].nt > m[1].nt ? m[0].nt : m[1].nt;
    *xs0 = 0;
    constexpr int kMultiStepBytes = 8192;  // the sweeps' steps (a few levels' and blocks' worth per matrix)
    if (smem_optin < 32768) return 0;
    // elements of the solve vectors and the top's vector that fit
    const long long cap = (long long)((smem_optin - 2048 - kMultiStepBytes) / elt) - 4;
    if (nmax + nt > cap) {
        const long long x = nmax + nt - cap;  // one case, with rows in global memory
        if (!multi_rows_out(m, x)) return 0;
        *xs0 = int(x);
        return 1;
    }
    int K = 0;
    for (int k = 1; k <= kMultiMax && (long long)(nmax + nt) * k <= cap; k *= 2) {
        K = k;
        if ((ncase + k - 1) / k <= num_sms) break;
    }
    return K;
}

}  // namespace gbpf

"""GPU checks of the size-dependent code paths at the sizes where they change,
against the CPU oracle."""
import numpy as np
import pytest

from paper_1811_02512_gb300 import gbpf, gridgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _loaded(raw, lam=1.0 / 32):
    return raw.scaled_network(lam)


# ncase 1: a 16-block cluster per case; ncase 20: one block per case.  n = 3
# and 30 put every level in the top part of the block factor or nearly so.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ncase", [1, 20])
@pytest.mark.parametrize("n", [3, 30, 700])
def test_newton_factor_top_and_adjoint(oracle, n, ncase, prec):
    raw = gridgen.small_raw(n, 11) if n < 100 else gridgen.delaunay_raw(n, 11)
    case = _loaded(raw)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    g = gbpf.Grid(case)
    g.set_cases(ncase)
    vm = torch.zeros((ncase, n), dtype=torch.float64, device="cuda")
    va = torch.zeros_like(vm)
    st, res = gbpf.pf_run_to_tol(g.ctx, gbpf.run_opts(gbpf.PF_NR, p, tol=1e-11, max_iter=30), vm, va, ncase)
    assert st == gbpf.PF_OK
    J = torch.empty(ncase, dtype=torch.float64, device="cuda")
    gva, gvm, dP, dQ = (torch.empty_like(vm) for _ in range(4))
    gbpf.pf_objective(g.ctx, vm, va, J, gva, gvm)
    gbpf.pf_adjoint(g.ctx, p, vm, va, gva, gvm, dP, dQ, ncase)
    rc, vm0, va0, _, _ = oracle.power_flow(case, oracle.NR, tol=1e-12)
    assert rc == oracle.OK
    aP, aQ, _ = oracle.adjoint(case, vm0, va0)
    scale = max(np.abs(aP).max(), np.abs(aQ).max())
    # a mismatch of 1e-11 defines the state to the inverse Jacobian's norm
    # times that (the adjoint of a per-bus sum bounds it: below 1e3 here)
    for c in (0, ncase - 1):
        assert np.abs(vm[c].cpu().numpy() - vm0).max() <= 1e-8
        assert np.abs(va[c].cpu().numpy() - va0).max() <= 1e-8
        assert np.abs(dP[c].cpu().numpy() - aP).max() <= 1e-7 * scale
        assert np.abs(dQ[c].cpu().numpy() - aQ).max() <= 1e-7 * scale
    g.close()


def _flow(case, g, ncase, prec, tol=1e-11, **kw):
    vm = torch.zeros((ncase, case.n), dtype=torch.float64, device="cuda")
    va = torch.zeros_like(vm)
    opts = gbpf.run_opts(gbpf.PF_FDPF, prec, tol=tol, max_iter=300, **kw)
    st, res = gbpf.pf_run_to_tol(g.ctx, opts, vm, va, ncase)
    return st, res, vm.cpu().numpy(), va.cpu().numpy()


# Cases per block 1, 2 and 4 with a partial last block (152 SMs: 1
# case each up to 152, 2 up to 304, then 4), load and outage cases, small
# grids without and with a narrow top, and grids whose solve vector does not
# fit shared memory (FP64 above about 27,000 rows).  From 2,500 buses a few
# cases run on clusters: of 16 blocks up to 9 cases, of 8 up to 19.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,ncase,nout", [(3, 1, 0), (37, 153, 0), (700, 307, 2), (1425, 613, 5), (30000, 2, 0),
                                          (2500, 9, 2), (2503, 15, 2), (2800, 40, 2)])
def test_cases_per_block(oracle, n, ncase, nout, prec):
    raw = gridgen.small_raw(n, 5) if n < 100 else gridgen.delaunay_raw(n, 5)
    case = _loaded(raw, 1.0 / 256 if n > 5000 else 1.0 / 64 if n > 1500 else 1.0 / 32)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    sc = gridgen.scenarios(case, n_load=ncase - nout, n_outage=nout, seed=3)
    g = gbpf.Grid(case)
    g.set_cases(ncase, sc.load_scale, sc.outage)
    gbpf.pf_set_tuning(g.ctx, 1, 0, 0, 0, 2 if nout else 0, 0)
    for ir_tol in (1e-3, 1e-10) if prec == "fp32" else (1e-10,):
        st, res, vm, va = _flow(case, g, ncase, p, ir_tol=ir_tol)
        assert st == gbpf.PF_OK and np.all(res["status"] == gbpf.PF_OK)
        # every case's mismatch is within 1e-11; the state follows to the
        # inverse Jacobian's norm times that, below 1e3 on these grids
        for c in {0, 1 % ncase, ncase // 2, ncase - 1 - nout, ncase - 1}:
            rc, vm0, va0, _, _ = oracle.power_flow(gridgen.apply_scenario(case, sc, c), oracle.NR, tol=1e-12)
            assert rc == oracle.OK
            assert np.abs(vm[c] - vm0).max() <= 1e-8 and np.abs(va[c] - va0).max() <= 1e-8
    g.close()


# Cases that leave the fixed-point range of the iteration (a slack angle
# beyond it, a set-point beyond it) run on the FP64 form instead, beside
# cases that stay; given starts are kept for them.
@pytest.mark.parametrize("engine", [gbpf.PF_ENGINE_AUTO, gbpf.PF_ENGINE_BLOCK])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shift", [0.0, 7.0, 9.0, 1000.0])
def test_leaves_the_fixed_point_range(oracle, shift, prec, engine):
    case = _loaded(gridgen.delaunay_raw(300, 9))
    # the solution turns with the slack angle
    rc, vm0, va0, _, _ = oracle.power_flow(case, oracle.NR, tol=1e-12)
    assert rc == oracle.OK
    va0 = va0 + shift
    case.va = np.where(case.btype == gridgen.SLACK, shift, 0.0)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    g = gbpf.Grid(case)
    g.set_cases(1)
    vm = torch.ones((1, case.n), dtype=torch.float64, device="cuda")
    vm[0] = torch.as_tensor(np.where(case.btype == gridgen.PQ, 1.0, case.vset))
    va = torch.full_like(vm, shift)
    opts = gbpf.run_opts(gbpf.PF_FDPF, p, tol=1e-10, max_iter=300, flat_start=0, engine=engine)
    st, res = gbpf.pf_run_to_tol(g.ctx, opts, vm, va, 1)
    assert st == gbpf.PF_OK
    assert np.abs(vm[0].cpu().numpy() - vm0).max() <= 1e-7
    assert np.abs(va[0].cpu().numpy() - va0).max() <= 1e-7
    g.close()


# Outage cases by rule in their low-rank form: with every outage's own factors
# the same states, an outage that splits the grid reported as before, and the
# own factors there for pf_solve and pf_get_factor afterwards.
# The low-rank data of 20, 90 and 157 outages is solved for 1, 2 and 4 columns
# per block.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("count", [20, 90, 157])
def test_outages_by_rule(prec, count):
    case = _loaded(gridgen.delaunay_raw(500, 21), 1.0 / 64)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    cut = gridgen.bridges(case.n, case.f, case.t, case.status)
    ring = [k for k in range(case.m) if k not in set(cut)][:count]
    out = np.array(ring + [-1, ring[0]], dtype=np.int32)

    def run(branches, **tuning):
        g = gbpf.Grid(case)
        g.set_cases(len(branches), None, branches)
        gbpf.pf_set_tuning(g.ctx, **tuning)
        return (g,) + _flow(case, g, len(branches), p)

    g, st, res, vm, va = run(out)
    g1, st1, res1, vm1, va1 = run(out, outage=1)
    assert st == st1 == gbpf.PF_OK and np.array_equal(res["iters"], res1["iters"])
    # two runs of the same iteration: the difference is rounding, seen through
    # the inverse matrices (FP32: their 1e-7, on steps that end at 1e-11)
    assert np.abs(vm - vm1).max() <= 1e-10 and np.abs(va - va1).max() <= 1e-10
    n = g.info.n[0]
    rhs = torch.ones((len(out), n), dtype=torch.float64, device="cuda")
    x, x1 = rhs.clone(), rhs.clone()
    gbpf.pf_solve(g.ctx, gbpf.PF_MAT_BP, p, x, len(out))
    gbpf.pf_solve(g1.ctx, gbpf.PF_MAT_BP, p, x1, len(out))
    torch.cuda.synchronize()
    assert torch.equal(x, x1)
    assert all(np.array_equal(a, b) for a, b in zip(gbpf.pf_get_factor(g.ctx, 0, p, 3, g.info),
                                                    gbpf.pf_get_factor(g1.ctx, 0, p, 3, g1.info)))
    split = np.array([cut[0], -1], dtype=np.int32)
    seen = []
    for tuning in (dict(), dict(outage=1)):
        g2, st2, res2, _, _ = run(split, **tuning)
        assert st2 != gbpf.PF_OK and res2[0]["status"] == st2 and res2[1]["status"] == gbpf.PF_OK
        if prec == "fp64":
            assert st2 == gbpf.PF_ERR_SINGULAR
        seen.append([tuple(r) for r in res2[["status", "iters", "method"]]])
        g2.close()
    assert seen[0] == seen[1]


# The grids of a pack on clusters (up to 19 grids, the largest of 2,500 buses
# or more), one to a block, and more grids than SMs: the same states as each
# grid by itself.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sizes", [(2500, 120, 2011), (40, 7, 300), (40, 7) * 77])
def test_pack_on_clusters(prec, sizes):
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    cases = [_loaded(gridgen.small_raw(n, 3) if n < 100 else gridgen.delaunay_raw(n, 3), 1.0 / 64) for n in sizes]
    grids = [gbpf.Grid(c) for c in cases]
    for g in grids:
        g.set_cases(1)
    pk = gbpf.Pack(grids)
    opts = gbpf.run_opts(gbpf.PF_FDPF, p, tol=1e-11, ir_tol=1e-10, max_iter=300)
    vm = torch.zeros(sum(sizes), dtype=torch.float64, device="cuda")
    va = torch.zeros_like(vm)
    st, res = pk.run(opts, vm, va)
    assert st == gbpf.PF_OK and np.all(res["status"] == gbpf.PF_OK)
    for c, n, off in zip(cases, sizes, pk.offset):
        g = gbpf.Grid(c)
        g.set_cases(1)
        st, res, vm1, va1 = _flow(c, g, 1, p, ir_tol=1e-10, engine=gbpf.PF_ENGINE_BLOCK)
        assert st == gbpf.PF_OK
        # both mismatches are within 1e-11: the bound of test_cases_per_block
        assert np.abs(vm[off:off + n].cpu().numpy() - vm1[0]).max() <= 1e-8
        assert np.abs(va[off:off + n].cpu().numpy() - va1[0]).max() <= 1e-8
        g.close()
    pk.close()
    for g in grids:
        g.close()

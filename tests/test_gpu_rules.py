"""GPU checks of the mappings that a run takes by rule: the same outcome as the
mapping set by hand."""
import numpy as np
import pytest

from paper_1811_02512_gb300 import gbpf, gridgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(g, n, ncase, prec, **kw):
    vm = torch.zeros((ncase, n), dtype=torch.float64, device="cuda")
    va = torch.zeros_like(vm)
    st, res = gbpf.pf_run_to_tol(g.ctx, gbpf.run_opts(gbpf.PF_FDPF, prec, **kw), vm, va, ncase)
    return st, res, vm.cpu().numpy(), va.cpu().numpy()


def _launches(g, kind):
    return gbpf.pf_get_profile(g.ctx, kind, reset=True)[0]


# Outage batches with cases that do not converge: those alone run again, with
# their own factors, in the first call and in later ones (captured too); a load
# case that fails does not make them.  The outcome is that of own factors for
# every outage; what converged in the low-rank form is the same to rounding.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("fallback", [0, 1])
@pytest.mark.parametrize("bad", [(), (3,), (0, 40, 119), (5, 121), (121,), tuple(range(120))])
def test_outages_that_fail(bad, fallback, prec):
    case = gridgen.delaunay_raw(300, 21).scaled_network(1.0 / 64)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    cut = set(gridgen.bridges(case.n, case.f, case.t, case.status))
    out = np.array([k for k in range(case.m) if k not in cut][:120] + [-1, -1], np.int32)
    ncase = len(out)
    ls = np.ones((ncase, case.n))
    for b in bad:
        ls[b] *= 3000.0
    own = gbpf.Grid(case)
    own.set_cases(ncase, ls, out)
    gbpf.pf_set_tuning(own.ctx, outage=1)
    kw = dict(tol=1e-10, max_iter=60, fallback=fallback)
    st1, res1, vm1, va1 = _run(own, case.n, ncase, p, **kw)
    g = gbpf.Grid(case)
    g.set_cases(ncase, ls, out)
    fine = np.array([c not in bad for c in range(ncase)])
    again = any(out[b] >= 0 for b in bad)
    seen = []
    for call in range(4):
        _launches(g, gbpf.PF_K_RUN)
        st, res, vm, va = _run(g, case.n, ncase, p, **kw)
        assert _launches(g, gbpf.PF_K_RUN) == 1 + again, call
        assert (st == gbpf.PF_OK) == (len(bad) == 0) == (st1 == gbpf.PF_OK)
        assert np.array_equal(res["status"], res1["status"]) and np.array_equal(res["method"], res1["method"])
        assert np.abs(res["iters"] - res1["iters"])[fine].max(initial=0) <= 1
        # two mismatches of at most 1e-10, seen through the inverse Jacobian (below 1e3 here)
        assert np.abs(vm[fine] - vm1[fine]).max(initial=0) <= 1e-7 and np.abs(va[fine] - va1[fine]).max(initial=0) <= 1e-7
        seen.append((res, vm, va))
    for res, vm, va in seen[1:]:
        assert all(np.array_equal(res[f], seen[0][0][f]) for f in ("status", "iters", "ir_steps", "method"))
        assert np.array_equal(vm, seen[0][1], equal_nan=True) and np.array_equal(va, seen[0][2], equal_nan=True)
    # the batch's own factors for pf_solve, whatever the slots held
    n = g.info.n[1]
    x, x1 = (torch.ones((ncase, n), dtype=torch.float64, device="cuda") for _ in range(2))
    gbpf.pf_solve(g.ctx, gbpf.PF_MAT_BPP, p, x, ncase)
    gbpf.pf_solve(own.ctx, gbpf.PF_MAT_BPP, p, x1, ncase)
    torch.cuda.synchronize()
    assert torch.equal(x, x1)
    # ordinary loads for the same outages: every case in the low-rank form again
    g.set_cases(ncase, np.ones((ncase, case.n)), out)
    for _ in range(2):
        _launches(g, gbpf.PF_K_RUN)
        st, res, vm, va = _run(g, case.n, ncase, p, **kw)
        assert st == gbpf.PF_OK and np.all(res["method"] == gbpf.PF_FDPF)
    assert _launches(g, gbpf.PF_K_RUN) == 1
    g.close()
    own.close()


# With no memory left for what only a mapping by rule needs, the run takes the
# mapping that does without.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_no_room_for_the_mapping_by_rule(prec):
    case = gridgen.delaunay_raw(3000, 21).scaled_network(1.0 / 64)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    cut = set(gridgen.bridges(case.n, case.f, case.t, case.status))
    out = np.array([k for k in range(case.m) if k not in cut][:600], np.int32)
    ncase = len(out)
    g = gbpf.Grid(case)
    g.set_cases(ncase, None, out)
    gbpf.pf_set_tuning(g.ctx, outage=1)
    st1, res1, vm1, va1 = _run(g, case.n, ncase, p, tol=1e-8)  # storage of the own factors
    gbpf.pf_set_tuning(g.ctx)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    vm = torch.zeros((ncase, case.n), dtype=torch.float64, device="cuda")
    va = torch.zeros_like(vm)
    torch.cuda.synchronize()
    # the low-rank storage is 57 MB at least (FP32; 115 MB in FP64)
    take = torch.cuda.mem_get_info()[0] - (32 << 20)
    hold = torch.empty(take, dtype=torch.uint8, device="cuda")
    try:
        for _ in range(3):
            st, res = gbpf.pf_run_to_tol(g.ctx, gbpf.run_opts(gbpf.PF_FDPF, p, tol=1e-8), vm, va, ncase)
            assert st == st1 == gbpf.PF_OK, gbpf.pf_last_error(g.ctx)
            assert np.array_equal(res["iters"], res1["iters"])
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(vm.cpu().numpy(), vm1) and np.array_equal(va.cpu().numpy(), va1)
    g.close()


# What an untuned run takes can be set by hand and is among the tuner's
# candidates: the same bits from the mapping by rule and from its fields.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,ncase,cluster", [(3000, 1, 16), (3000, 12, 8), (900, 1, 1)])
def test_tuning_reaches_the_mapping_by_rule(n, ncase, cluster, prec):
    case = gridgen.delaunay_raw(n, 7).scaled_network(1.0 / 64)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    sc = gridgen.scenarios(case, n_load=ncase, n_outage=0, seed=3)
    g = gbpf.Grid(case)
    g.set_cases(ncase, sc.load_scale, sc.outage)
    out = []
    for tuning in (dict(engine=gbpf.PF_ENGINE_BLOCK),
                   dict(engine=gbpf.PF_ENGINE_BLOCK, cluster=cluster, factor=1, tail=3, outage=1)):
        gbpf.pf_set_tuning(g.ctx, **tuning)
        out.append(_run(g, n, ncase, p, tol=1e-8))
    assert out[0][0] == gbpf.PF_OK and np.array_equal(out[0][1], out[1][1])
    assert np.array_equal(out[0][2], out[1][2]) and np.array_equal(out[0][3], out[1][3])
    # asked for where the size would not have it: as many blocks, the same states to rounding
    if cluster == 1:
        gbpf.pf_set_tuning(g.ctx, engine=gbpf.PF_ENGINE_BLOCK, cluster=16, tail=3)
        st, res, vm, va = _run(g, n, ncase, p, tol=1e-8)
        assert st == gbpf.PF_OK and res["iters"][0] == out[0][1]["iters"][0]
        assert np.abs(vm - out[0][2]).max() <= 1e-9 and np.abs(va - out[0][3]).max() <= 1e-9
    g.close()


# A star has one level and no narrow top: the tuner tries form 3 there too.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_tuner_on_a_grid_without_a_top(prec):
    m = 400
    z = np.zeros(m + 1)
    case = gridgen.Case("star", np.array([gridgen.SLACK] + [gridgen.PQ] * m, np.int32),
                        np.r_[0.0, np.linspace(0.01, 0.1, m)], np.r_[0.0, np.full(m, 0.01)], z.copy(), z.copy(), z.copy(),
                        np.ones(m + 1), z.copy(), np.zeros(m, np.int32), np.arange(1, m + 1, dtype=np.int32),
                        np.full(m, 0.01), np.full(m, 0.05), np.zeros(m), np.zeros(m), np.ones(m, np.int32))
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    g = gbpf.Grid(case)
    g.set_cases(40)
    vm = torch.zeros((40, m + 1), dtype=torch.float64, device="cuda")
    va = torch.zeros_like(vm)
    _launches(g, gbpf.PF_K_RUN)
    t = gbpf.pf_autotune(g.ctx, gbpf.run_opts(gbpf.PF_FDPF, p, tol=1e-8), vm, va, reps=1)
    runs = _launches(g, gbpf.PF_K_RUN)
    assert t["tail"] in (2, 3) or t["engine"] == gbpf.PF_ENGINE_LANES
    # one block per case, two factor forms, three block sizes, tail 2 and 3,
    # each once untimed and once timed (the lane engine counts more launches)
    assert runs >= 2 * 2 * 3 * 2
    gbpf.pf_set_tuning(g.ctx, engine=gbpf.PF_ENGINE_BLOCK, cluster=1, factor=1, tail=3, outage=1, threads=512)
    st, res, vm1, va1 = _run(g, m + 1, 40, p, tol=1e-8)
    gbpf.pf_set_tuning(g.ctx, engine=gbpf.PF_ENGINE_BLOCK)
    st0, res0, vm0, va0 = _run(g, m + 1, 40, p, tol=1e-8)
    assert st == st0 == gbpf.PF_OK and np.array_equal(vm0, vm1) and np.array_equal(va0, va1)
    g.close()


# A case's result is its own: the same bits whatever other cases the batch
# holds (2 and 4 cases to a block).
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ncase", [201, 307])
def test_bits_do_not_depend_on_the_other_cases(ncase, prec):
    case = gridgen.delaunay_raw(700, 5).scaled_network(1.0 / 32)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    # every eighth case stays, the others take other loads (some too heavy ones)
    out = []
    for k in range(4):
        ls = np.random.default_rng(2).normal(1.0, 0.08, (ncase, case.n))
        rest = np.arange(ncase) % 8 != 0
        ls[rest] *= np.random.default_rng(10 + k).uniform(0.3, 1.3, (int(rest.sum()), 1))
        g = gbpf.Grid(case)
        g.set_cases(ncase, ls)
        st, res, vm, va = _run(g, case.n, ncase, p, tol=1e-10)
        assert np.all(res["status"][::8] == gbpf.PF_OK)
        out.append((res["iters"][::8], vm[::8], va[::8]))
        g.close()
    for its, vm, va in out[1:]:
        assert np.array_equal(its, out[0][0]) and np.array_equal(vm, out[0][1]) and np.array_equal(va, out[0][2])


# Grids of so many levels that the sweeps' steps take more shared memory than
# set aside: the solve vector gives way, alone and in a pack (whose kernel has
# less), instead of the whole run going to the one-case kernel.
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [52000, 70000])
def test_steps_of_many_levels_fit(n, prec):
    case = gridgen.delaunay_raw(n, 7).scaled_network(1.0 / 512)
    p = gbpf.PF_FP64 if prec == "fp64" else gbpf.PF_FP32
    g = gbpf.Grid(case)
    g.set_cases(1)
    alone, packed = [], []
    for tuning in (dict(tail=1, cluster=1), dict(), dict(tail=3, cluster=16)):
        gbpf.pf_set_tuning(g.ctx, engine=gbpf.PF_ENGINE_BLOCK, **tuning)
        alone.append(_run(g, n, 1, p, tol=1e-8, ir_tol=1e-3))
    pk = gbpf.Pack([g])
    for tuning in (dict(tail=1), dict()):
        gbpf.pf_set_tuning(g.ctx, **tuning)
        vm = torch.zeros(n, dtype=torch.float64, device="cuda")
        va = torch.zeros_like(vm)
        st, res = pk.run(gbpf.run_opts(gbpf.PF_FDPF, p, tol=1e-8, ir_tol=1e-3), vm, va)
        packed.append((st, res, vm.cpu().numpy()[None], va.cpu().numpy()[None]))
    pk.close()
    g.close()
    for st, res, vm, va in alone + packed:
        assert st == gbpf.PF_OK and abs(int(res["iters"][0]) - int(alone[0][1]["iters"][0])) <= 1
        # two mismatches within 1e-8, seen through the inverse Jacobian
        assert np.abs(vm - alone[0][2]).max() <= 1e-5 and np.abs(va - alone[0][3]).max() <= 1e-5
    if prec == "fp64" and n > 54000:  # half of the rows and the top do not fit shared memory
        return
    assert np.array_equal(alone[1][2], alone[2][2]) and np.array_equal(alone[1][3], alone[2][3])
    # not the one-case kernels, whose bits tail 1 gives
    assert not np.array_equal(alone[1][3], alone[0][3]) and not np.array_equal(packed[1][3], packed[0][3])

"""GPU checks of the fixed-point forms where their ranges end: what leaves them
takes the FP64 form, with the results that has."""
import numpy as np
import pytest

from paper_1811_02512_gb300 import gbpf, gridgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _chain(strong, weak, load):
    """Bus 0 (load) -- strong -- bus 1 -- weak -- bus 2 (slack), lossless, by 1/x."""
    z = np.zeros(3)
    return gridgen.Case("chain", np.array([gridgen.PQ, gridgen.PQ, gridgen.SLACK], np.int32), np.array([load, 0.0, 0.0]),
                        z.copy(), z.copy(), z.copy(), z.copy(), np.ones(3), z.copy(), np.array([0, 1], np.int32),
                        np.array([1, 2], np.int32), np.zeros(2), np.array([1 / strong, 1 / weak]), np.zeros(2),
                        np.zeros(2), np.ones(2, np.int32))


# FP32 holds strong + weak = 2^23 + 1.6 as 2^23 + 2 and strong as 2^23: a solve
# gives 1.3 / 2 of the step, one correction 0.35 of the rest, and each part may
# be in the range of a step's limbs where their sum is not.  The loads ask for
# steps of 1.6 to 3.2 rad, of which one correction leaves 1 - 0.35^2.
def test_refined_step_beyond_the_limbs():
    case = _chain(2.0 ** 23 + 0.3, 1.3, -1.3)
    want = np.linspace(1.6, 3.2, 33)
    ls = np.ones((33, 3))
    ls[:, 0] = want
    va = []
    for tuning in (dict(engine=gbpf.PF_ENGINE_BLOCK), dict(engine=gbpf.PF_ENGINE_BLOCK, cluster=1, tail=1, threads=512)):
        g = gbpf.Grid(case)
        g.set_cases(33, ls)
        gbpf.pf_set_tuning(g.ctx, **tuning)
        vm = torch.zeros((33, 3), dtype=torch.float64, device="cuda")
        th = torch.zeros_like(vm)
        gbpf.pf_run_to_tol(g.ctx, gbpf.run_opts(gbpf.PF_FDPF, gbpf.PF_FP32, tol=1e-8, max_iter=1, ir_max=1), vm, th, 33)
        va.append(th.cpu().numpy())
        g.close()
    # FP32 roundings of two solves of a step of at most 3.2
    assert np.abs(va[0] - va[1]).max() <= 8 * 3.2 * 2.0 ** -23
    assert np.abs(va[0][:, 0] - want * (1 - 0.35 ** 2)).max() <= 8 * 3.2 * 2.0 ** -23


# The FP32 factor holds the weak branch as `held` instead of weak, so every
# correction of the adjoint leaves 1 - weak / held of the error: 20 of them are
# all it has, and they are all taken.
@pytest.mark.parametrize("strong,weak,held", [(2.0 ** 23 + 0.45, 0.08, 1.0), (2.0 ** 23 + 0.4, 0.15, 1.0),
                                              (2.0 ** 23 + 0.3, 1.3, 2.0)])
def test_adjoint_of_a_poor_factor_takes_every_correction(strong, weak, held):
    g = gbpf.Grid(_chain(strong, weak, 0.0))
    g.set_cases(1)
    vm = torch.ones((1, 3), dtype=torch.float64, device="cuda")
    va, gvm, dP, dQ = (torch.zeros_like(vm) for _ in range(4))
    gva = torch.tensor([[1.0, 0.0, 0.0]], dtype=torch.float64, device="cuda")
    gbpf.pf_adjoint(g.ctx, gbpf.PF_FP32, vm, va, gva, gvm, dP, dQ, 1)
    # dJ/dP at bus 1 is 1 / weak; the 21 solves leave (1 - weak / held)^21 of
    # it, to FP32's rounding of the last correction and what it multiplies
    left = (1 - weak / held) ** 21
    assert abs(weak * dP[0, 1].item() - (1 - left)) <= 1e-5
    g.close()


def _states(case, vm, va, unaligned=False):
    """pf_mismatch, pf_objective and pf_branch_flows at one state."""
    g = gbpf.Grid(case)
    g.set_cases(1)
    vm, va = (torch.as_tensor(np.atleast_2d(a)).cuda() for a in (vm, va))
    dp, dq, gva, gvm = (torch.zeros_like(vm) for _ in range(4))
    mis, J, loss = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(3))
    store = torch.zeros(case.m * 4 + 1, dtype=torch.float64, device="cuda")
    flows = store[1:] if unaligned else store[:-1]
    gbpf.pf_mismatch(g.ctx, vm, va, dp, dq, mis, 1)
    gbpf.pf_objective(g.ctx, vm, va, J, gva, gvm)
    gbpf.pf_branch_flows(g.ctx, vm, va, 1, flows, loss)
    torch.cuda.synchronize()
    out = [t.cpu().numpy() for t in (dp[0], dq[0], mis, J, gva[0], gvm[0], flows.view(-1, 4), loss)]
    ybus = gbpf.pf_get_ybus(g.ctx, case.n, g.info.nnz_ybus)
    g.close()
    return out, ybus


# Flows and mismatches of small operands keep a double's relative accuracy: a
# lossless branch between small angles (P), low voltages, terms set apart by a
# tap, a resistive branch at a flat profile (Q).
@pytest.mark.parametrize("r,x,tap,v,th", [
    (0.0, 0.1, 0.0, 1.0, 1e-3), (0.0, 0.1, 0.0, 1.0, 1e-6), (0.0, 0.1, 0.0, 1.0, 1e-9), (1e-4, 0.1, 0.0, 1.0, 1e-6),
    (0.01, 0.1, 0.0, 0.3, 0.1), (0.01, 0.1, 0.0, 1e-3, 0.1), (0.01, 0.1, 0.0, 1e-6, 0.1), (0.01, 0.1, 0.0, 1e-9, 0.1),
    (0.01, 0.1, 1e-3, 1.0, 0.1), (0.01, 0.1, 1e3, 1.0, 0.1), (0.01, 0.1, 0.5, 1.0, 0.1), (0.1, 0.0, 0.0, 1.0, 1e-6)])
def test_small_operands_keep_their_digits(r, x, tap, v, th):
    case = _chain(10.0, 10.0, 0.0)
    case.r[:], case.x[:], case.tap[0] = r, x if x else 1e-30, tap
    vm, va = np.array([v, 1.1 * v, 1.0]), np.array([3 * th, -th, 0.0])
    (dp, dq, _, _, _, _, flows, _), _ = _states(case, vm, va)
    L = np.longdouble
    t = L(tap) if tap else L(1)
    den = L(case.r[0]) ** 2 + L(case.x[0]) ** 2
    g, b = L(case.r[0]) / den, -L(case.x[0]) / den
    Vf, Vt, d = L(vm[0]), L(vm[1]), L(va[0]) - L(va[1])
    h = 2 * np.sin(d / 2) ** 2  # 1 - cos d
    ff = Vf / t
    # S_f = ff conj(y (ff - Vt e^-jd)), S_t = Vt conj(y (Vt - ff e^jd))
    pf = ff * (g * (ff - Vt + Vt * h) - b * Vt * np.sin(d))
    qf = -ff * (b * (ff - Vt + Vt * h) + g * Vt * np.sin(d))
    pt = Vt * (g * (Vt - ff + ff * h) + b * ff * np.sin(d))
    qt = -Vt * (b * (Vt - ff + ff * h) - g * ff * np.sin(d))
    # an FP64 evaluation rounds a few times at the size of the terms of each sum
    y = abs(g) * max(abs(ff), abs(Vt)) + abs(b) * max(abs(ff), abs(Vt)) * min(1.0, abs(d))
    z = abs(b) * max(abs(ff), abs(Vt)) + abs(g) * max(abs(ff), abs(Vt)) * min(1.0, abs(d))
    for got, want, size in ((flows[0, 0], pf, ff * y), (flows[0, 1], qf, ff * z), (flows[0, 2], pt, Vt * y),
                            (flows[0, 3], qt, Vt * z), (-dp[0], pf, ff * y), (-dq[0], qf, ff * z)):
        assert abs(got - want) <= 16 * 2.0 ** -53 * size, (got, want)


# States outside the fixed-point range and rows beyond any scale, beside
# ordinary buses: the mismatch of the general FP64 entry point, flows and
# gradient as plain FP64 gives them, not-finite where those are.
@pytest.mark.parametrize("special", [dict(vm=0.3), dict(vm=2.5), dict(vm=0.0), dict(va=9.0), dict(va=-1e3), dict(vm=np.nan),
                                     dict(va=np.nan), dict(va=np.inf), dict(vm=np.inf), dict(x=1e-125), dict(x=1e-30)])
def test_states_outside_the_range(special):
    case = gridgen.delaunay_raw(300, 9).scaled_network(1.0 / 32)
    rng = np.random.default_rng(4)
    vm, va = 1.0 + 0.02 * rng.standard_normal(case.n), 0.1 * rng.standard_normal(case.n)
    where = np.array([5, 140, 299])
    if "x" in special:
        case.x[where], case.r[where] = special["x"], 0.3 * special["x"]
    vm[where] = special.get("vm", vm[where])
    va[where] = special.get("va", va[where])
    (dp, dq, mis, J, gva, gvm, flows, loss), (rp, col, G, B) = _states(case, vm, va, unaligned=True)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
    dp0, dq0, mis0 = t(np.zeros(case.n)), t(np.zeros(case.n)), t(np.zeros(1))
    st = gbpf.pf_mismatch_static(case.n, t(rp, torch.int32), t(col, torch.int32), t(G), t(B), t(case.btype, torch.int32),
                                 t(case.pg - case.pd), t(-case.qd), t(vm), t(va), dp0, dq0, mis0)
    assert st == gbpf.PF_OK
    torch.cuda.synchronize()
    dp0, dq0, mis0 = (a.cpu().numpy() for a in (dp0, dq0, mis0))
    with np.errstate(all="ignore"):
        v = np.nan_to_num(np.abs(vm), nan=0, posinf=0).max()
        row = np.add.reduceat(np.abs(G) + np.abs(B), rp[:-1]) * v * v  # each row's terms; 3.7 of them on average
        for got, want in ((dp, dp0), (dq, dq0)):
            assert np.array_equal(np.isfinite(got), np.isfinite(want))
            ok = np.isfinite(want)
            assert np.all(np.abs(got - want)[ok] <= 32 * 2.0 ** -53 * (row[ok] + 1.0))
        assert np.isfinite(mis[0]) == np.isfinite(mis0[0])
        V = vm * np.exp(1j * va)
        y = 1.0 / (case.r + 1j * case.x)
        tap = np.where(case.tap == 0, 1.0, case.tap)
        Vf, Vt = V[case.f], V[case.t]
        sf = Vf * np.conj((y + 0.5j * case.b) / tap ** 2 * Vf - y / tap * Vt)
        stt = Vt * np.conj((y + 0.5j * case.b) * Vt - y / tap * Vf)
        ref = np.stack([sf.real, sf.imag, stt.real, stt.imag], 1)
        size = (np.abs(y) + np.abs(case.b)) * np.maximum(np.abs(Vf), np.abs(Vt)) ** 2
        ok = np.isfinite(ref).all(1)
        assert np.array_equal(np.isfinite(flows).all(1), ok)
        assert np.all(np.abs(flows - ref)[ok] <= 64 * 2.0 ** -53 * size[ok, None])
        if "x" in special or not np.isfinite(vm).all() or not np.isfinite(va).all():
            return
        # dJ/dtheta, dJ/dV of sum (V - 1)^2 + sum P over the branches and shunts
        gt = np.zeros(case.n)
        gv = 2 * (vm - 1) + 2 * vm * case.gs
        for k in range(case.m):
            a, c, gk = case.f[k], case.t[k], y[k].real
            dth, tk = va[a] - va[c], tap[k]
            gt[a] += 2 * gk / tk * vm[a] * vm[c] * np.sin(dth)
            gt[c] -= 2 * gk / tk * vm[a] * vm[c] * np.sin(dth)
            gv[a] += 2 * gk * (vm[a] / tk ** 2 - vm[c] / tk * np.cos(dth))
            gv[c] += 2 * gk * (vm[c] - vm[a] / tk * np.cos(dth))
        for got, want in ((gva, gt), (gvm, gv)):
            assert np.all(np.abs(got - want) <= 64 * 2.0 ** -53 * (row + 1.0))


# Refinement asked for below the unit of the fixed-point residual (absolute
# targets of 1e-30 on rows that sum to 174): as many corrections as the form
# with the FP64 residual takes, alone and in a pack.
@pytest.mark.parametrize("ir_tol,ir_abs", [(1e-10, 0.0), (1e-10, 1e-30), (1e-14, 1e-30), (1e-3, 1e-30)])
def test_refinement_below_the_unit(ir_tol, ir_abs):
    case = gridgen.delaunay_raw(700, 5).scaled_network(1.0 / 32)
    opts = gbpf.run_opts(gbpf.PF_FDPF, gbpf.PF_FP32, tol=1e-8, ir_max=20, ir_tol=ir_tol, ir_abs=ir_abs)
    steps = []
    for tuning in (dict(cluster=1, tail=1, threads=512), dict(), None):
        g = gbpf.Grid(case)
        g.set_cases(1)
        vm = torch.zeros((1, case.n), dtype=torch.float64, device="cuda")
        va = torch.zeros_like(vm)
        if tuning is None:
            pk = gbpf.Pack([g])
            st, res = pk.run(opts, vm[0], va[0])
            pk.close()
        else:
            gbpf.pf_set_tuning(g.ctx, engine=gbpf.PF_ENGINE_BLOCK, **tuning)
            st, res = gbpf.pf_run_to_tol(g.ctx, opts, vm, va, 1)
        assert st == gbpf.PF_OK
        steps.append(int(res["ir_steps"][0]))
        g.close()
    # a solve whose residual lies at the target may go either way: one in ten
    assert max(steps) <= 1.1 * steps[0] + 2, steps

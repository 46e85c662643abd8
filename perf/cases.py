"""The workloads whose speed is followed, from the smallest grid to the largest.

Every case goes through the package's public entry points on one GPU.  The
grids are the seeded synthetic ones of ``gridgen``; a case names its topology
and its sizes, and the seed of ``prepare`` draws what changes from call to
call in use: the loads of every bus, the outaged branches, the states and the
right-hand sides.  ``exact`` recomputes a case in FP64 with plain torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1811_02512_gb300 import gbpf, gridgen

DEV = "cuda"
EXACT_MAX_BUS = 21000      # the dense Jacobian of a larger grid takes too long
EXACT_MAX_PACK_BUS = 6000  # the same for each grid of a pack
FLOW = dict(kind="flow", grid="delaunay", gseed=0, ncase=1, nout=0, precision="fp64", ir_tol=1e-10,
            tuned=False, fallback=False)


def listed():
    return [
        # the smallest call: an operator's 120-bus system solved once, mapping chosen by the autotuner
        dict(FLOW, name="flow120", grid="config0", n=120, tuned=True),
        # a regional grid solved as the quick start does it, without tuning
        dict(FLOW, name="flow2643", n=2643),
        # the headline: one 10,000-bus energy-management solve in FP64, tuned
        dict(FLOW, name="flow10k", grid="config1", n=10000, tuned=True),
        # a large interconnection with FP32 factors and the default refinement, untuned
        dict(FLOW, name="flow40k_fp32", n=40000, precision="fp32"),
        # a planning study: 512 load scenarios and 512 branch outages in one tuned FP32 launch
        dict(FLOW, name="batch10k_1024_fp32", grid="config1", n=10000, ncase=1024, nout=512,
             precision="fp32", ir_tol=1e-3, tuned=True),
        # a day of load profiles on a regional grid, FP64, untuned
        dict(FLOW, name="loads2643_288", n=2643, ncase=288),
        # N-1 screening of a small system, FP64, the NR fallback armed, untuned
        dict(FLOW, name="outages1425_512", n=1425, ncase=512, nout=512, fallback=True),
        # a queue of unequal grids solved in one packed launch, FP32 with refinement
        dict(kind="pack", name="pack10_fp32", first=30, ngrid=10, precision="fp32", ir_tol=1e-3),
        # a training step of a dispatch model: Newton-Raphson and the adjoint gradient
        dict(kind="grad", name="grad20k_fp32", grid="config3", gseed=0, n=20000, ncase=1, precision="fp32"),
        # the same on a regional grid for a few profiles, FP64 factors
        dict(kind="grad", name="grad1425_fp64", grid="delaunay", gseed=0, n=1425, ncase=4, precision="fp64"),
        # evaluation of given states: mismatch, objective with gradient, branch flows
        dict(kind="states", name="states10k_256", grid="config1", gseed=0, n=10000, ncase=256),
        # the linear-algebra entry points by themselves: both factors, then many right-hand sides
        dict(kind="solve", name="solve5k_64", grid="delaunay", gseed=0, n=5001, ncase=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow", "flow", "batch", "batch", "pack", "grad", "states", "solve"])
    gseed = rng.randrange(1, 1000)
    precision = rng.choice(["fp64", "fp32"])
    if kind == "flow":
        return dict(FLOW, n=_log(rng, 100, 40000), gseed=gseed, precision=precision,
                    ir_tol=rng.choice([1e-10, 1e-3]), tuned=rng.random() < 0.5)
    if kind == "batch":
        n = _log(rng, 100, 10000)
        ncase = _log(rng, 2, min(1024, 2_000_000 // n))
        nout = rng.choice([0, ncase // 2, min(ncase, n // 8)])
        return dict(FLOW, n=n, gseed=gseed, ncase=ncase, nout=nout, precision=precision,
                    ir_tol=rng.choice([1e-10, 1e-3]), tuned=rng.random() < 0.5)
    if kind == "pack":
        ngrid = rng.randrange(2, 11)
        sizes = [s for s, _ in gridgen.config4_sizes()]
        first = rng.choice([k for k in range(len(sizes) - ngrid) if sum(sizes[k:k + ngrid]) <= 190_000])
        return dict(kind="pack", first=first, ngrid=ngrid, precision=precision, ir_tol=rng.choice([1e-10, 1e-3]))
    if kind == "grad":
        n = _log(rng, 100, 20000 if precision == "fp32" else 3000)
        return dict(kind="grad", grid="delaunay", gseed=gseed, n=n, ncase=rng.randrange(1, 5) if n < 3000 else 1,
                    precision=precision)
    n = _log(rng, 100, 20000)
    return dict(kind=kind, grid="delaunay", gseed=gseed, n=n,
                ncase=_log(rng, 1, min(512, 2_500_000 // n if kind == "states" else 320_000 // n)))


# ---------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=64)
def _grid(grid, n, gseed):
    if grid == "delaunay":
        # loadings and network scalings under which a flat start converges for every seed tried
        lam = 1 / 32 if n <= 1000 else 1 / 64 if n <= 5000 else 1 / 128 if n <= 15000 else 1 / 256
        return gridgen.delaunay_raw(n, 1000 * gseed + n).scaled_network(lam)
    if grid == "multigrid":
        size, seed = gridgen.config4_sizes()[n]
        return gridgen.with_loading_factor(gridgen.delaunay_raw(size, seed, name=f"multigrid{n}"))
    return gridgen.config(int(grid[len("config"):]))


@functools.lru_cache(maxsize=64)
def _cycle_branches(grid, n, gseed):
    g = _grid(grid, n, gseed)
    cut = set(gridgen.bridges(g.n, g.f, g.t, g.status))
    return np.array([k for k in range(g.m) if k not in cut], dtype=np.int32)


def _load_scale(g, ncase, rng):
    """Per-bus factors ~ N(1, 0.08) of every load, as a forecast's error."""
    s = np.ones((ncase, g.n))
    pq = g.btype == gridgen.PQ
    s[:, pq] = rng.normal(1.0, 0.08, (ncase, int(pq.sum())))
    return s


def _scenarios(case, seed):
    """(grid, load_scale, outage): load cases first, then single-branch outages at the base load."""
    g = _grid(case["grid"], case["n"], case["gseed"])
    rng = np.random.default_rng(seed)
    scale = _load_scale(g, case["ncase"], rng)
    if case["nout"] == 0:
        return g, scale, None
    cand = _cycle_branches(case["grid"], case["n"], case["gseed"])
    out = np.full(case["ncase"], -1, dtype=np.int32)
    k = min(case["nout"], len(cand))
    out[case["ncase"] - k:] = rng.permutation(cand)[:k]
    scale[out >= 0] = scale[0]
    return g, scale, out


def _injections(case, seed):
    """Specified (Psp, Qsp) [ncase, n] of loads drawn around the grid's own."""
    g = _grid(case["grid"], case["n"], case["gseed"])
    scale = _load_scale(g, case["ncase"], np.random.default_rng(seed))
    return g, g.pg - g.pd * scale, -g.qd * scale


def _states(case, seed):
    g = _grid(case["grid"], case["n"], case["gseed"])
    rng = np.random.default_rng(seed + 1)
    vm = 1.0 + 0.02 * rng.standard_normal((case["ncase"], g.n))
    va = 0.1 * rng.standard_normal((case["ncase"], g.n))
    return vm, va


def _rhs(case, seed):
    g = _grid(case["grid"], case["n"], case["gseed"])
    rng = np.random.default_rng(seed)
    return [rng.standard_normal((case["ncase"], int(k)))
            for k in (np.sum(g.btype != gridgen.SLACK), np.sum(g.btype == gridgen.PQ))]


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV)


def _precision(case):
    return gbpf.PF_FP32 if case["precision"] == "fp32" else gbpf.PF_FP64


def _pack_grids(case):
    return [_grid("multigrid", k, 0) for k in range(case["first"], case["first"] + case["ngrid"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pack":
        cases = _pack_grids(case)
        rng = np.random.default_rng(seed)
        grids = [gbpf.Grid(c) for c in cases]
        for g in grids:
            g.set_cases(1, _load_scale(g.case, 1, rng))
        vm = torch.zeros(sum(g.nbus for g in grids), dtype=torch.float64, device=DEV)
        opts = gbpf.run_opts(gbpf.PF_FDPF, _precision(case), tol=1e-8, ir_tol=case["ir_tol"])
        return dict(kind=kind, pack=gbpf.Pack(grids), opts=opts, vm=vm, va=torch.zeros_like(vm))
    if kind == "flow":
        c, scale, out = _scenarios(case, seed)
        g = gbpf.Grid(c)
        g.set_cases(case["ncase"], scale, out)
        vm = torch.zeros((case["ncase"], c.n), dtype=torch.float64, device=DEV)
        va = torch.zeros_like(vm)
        opts = gbpf.run_opts(gbpf.PF_FDPF, _precision(case), tol=1e-8, ir_tol=case["ir_tol"],
                             fallback=int(case["fallback"]))
        if case["tuned"]:
            gbpf.pf_autotune(g.ctx, opts, vm, va, reps=3 if case["ncase"] == 1 else 1)
        return dict(kind=kind, grid=g, opts=opts, vm=vm, va=va)
    c = _grid(case["grid"], case["n"], case["gseed"])
    g = gbpf.Grid(c)
    ncase = case["ncase"]
    if kind == "grad":
        g.set_cases(ncase)
        _, psp, qsp = _injections(case, seed)
        return dict(kind=kind, grid=g, precision=_precision(case), psp=_dev(psp).requires_grad_(),
                    qsp=_dev(qsp).requires_grad_())
    if kind == "states":
        g.set_cases(ncase, _load_scale(c, ncase, np.random.default_rng(seed)))
        vm, va = _states(case, seed)
        return dict(kind=kind, grid=g, vm=_dev(vm), va=_dev(va))
    g.set_cases(ncase)
    return dict(kind=kind, grid=g, rhs=[_dev(b) for b in _rhs(case, seed)])


# ---------------------------------------------------------------- one pass

def run(state):
    kind = state["kind"]
    if kind == "flow":
        vm, va = state["vm"], state["va"]
        _, res = gbpf.pf_run_to_tol(state["grid"].ctx, state["opts"], vm, va, vm.shape[0])
        return dict(vm=vm, va=va, status=res["status"], iters=res["iters"])
    if kind == "pack":
        pack = state["pack"]
        _, res = pack.run(state["opts"], state["vm"], state["va"])
        cut = [slice(int(a), int(b)) for a, b in zip(pack.offset[:-1], pack.offset[1:])]
        return dict(vm=[state["vm"][s] for s in cut], va=[state["va"][s] for s in cut],
                    status=res["status"], iters=res["iters"])
    g = state["grid"]
    if kind == "grad":
        psp, qsp = state["psp"], state["qsp"]
        vm, va = gbpf.PowerFlowFn.apply(g, psp, qsp, state["precision"])
        J = gbpf.ObjectiveFn.apply(g, vm, va)
        dP, dQ = torch.autograd.grad(J.sum(), (psp, qsp))
        return dict(vm=vm.detach(), va=va.detach(), J=J.detach(), dP=dP, dQ=dQ)
    if kind == "states":
        vm, va = state["vm"], state["va"]
        ncase = vm.shape[0]
        dp, dq, gva, gvm = (torch.empty_like(vm) for _ in range(4))
        mis, J, loss = (torch.empty(ncase, dtype=torch.float64, device=vm.device) for _ in range(3))
        flows = torch.empty((ncase, g.case.m, 4), dtype=torch.float64, device=vm.device)
        stream = torch.cuda.current_stream()
        gbpf.pf_mismatch(g.ctx, vm, va, dp, dq, mis, ncase, stream)
        gbpf.pf_objective(g.ctx, vm, va, J, gva, gvm, stream)
        gbpf.pf_branch_flows(g.ctx, vm, va, ncase, flows, loss, stream)
        return dict(dp=dp, dq=dq, mis=mis, J=J, gva=gva, gvm=gvm, flows=flows, loss=loss)
    x = []
    stream = torch.cuda.current_stream()
    for which, b in zip((gbpf.PF_MAT_BP, gbpf.PF_MAT_BPP), state["rhs"]):
        gbpf.pf_factor(g.ctx, which, gbpf.PF_FP64, stream)
        x.append(b.clone())
        gbpf.pf_solve(g.ctx, which, gbpf.PF_FP64, x[-1], b.shape[0], stream=stream)
    return dict(x=x)


def work(case):
    """Bytes of the inputs and outputs, and operations of the method, per pass.

    With n buses the grids have 1.35 n branches, 3.7 n admittance entries and
    about 3.3 n (B') and 1.7 n (B'') entries in L; a fast decoupled solve
    takes about 16 half-iterations, a Newton one 4 steps of about 40 n block
    updates of 16 operations.
    """
    kind, ncase = case["kind"], case.get("ncase", 1)
    n = sum(s for s, _ in gridgen.config4_sizes()[case["first"]:case["first"] + case["ngrid"]]) \
        if kind == "pack" else case["n"]
    net = 60 * n + int(1.35 * n) * 48
    vec = 8 * n * ncase
    if kind in ("flow", "pack"):
        return {"bytes": net + 4 * vec, "flops": 16 * ncase * n * (8 * 3.7 + 21 + 4 * 2.5) + 40 * n}
    if kind == "grad":
        return {"bytes": net + 6 * vec, "flops": 4 * ncase * n * (640 + 100) + ncase * n * 200}
    if kind == "states":
        return {"bytes": net + 8 * vec + int(1.35 * n) * 32 * ncase, "flops": ncase * n * (3 * 8 * 3.7 + 100)}
    return {"bytes": net + 4 * vec, "flops": ncase * n * 4 * 5.0 + 40 * n}


# ---------------------------------------------------------------- FP64 by plain torch

class _Network:
    """One grid's branches in FP64: nodal powers and the dense Jacobian."""

    def __init__(self, g):
        t = functools.partial(torch.as_tensor, device=DEV)
        self.n, self.m = g.n, g.m
        self.f, self.t = t(g.f).long(), t(g.t).long()
        on = t(g.status).double()
        ys = on / torch.complex(t(g.r).double(), t(g.x).double())
        tap = t(np.where(g.tap == 0.0, 1.0, g.tap)).double()
        half = on * 0.5j * t(g.b).double()
        self.yff, self.ytt, self.yft = (ys + half) / tap ** 2, ys + half, -ys / tap
        self.ysh = torch.complex(t(g.gs).double(), t(g.bs).double())
        self.btype = t(g.btype)
        pv = np.where(g.btype == gridgen.PQ, 1.0, g.vset)
        self.v0, self.a0 = t(pv).double(), t(np.where(g.btype == gridgen.SLACK, g.va, 0.0)).double()
        self.th = torch.nonzero(self.btype != gridgen.SLACK)[:, 0]
        self.vq = torch.nonzero(self.btype == gridgen.PQ)[:, 0]

    def ends(self, V, out=None):
        """Complex power into the branches at both ends, [ncase, m] each."""
        Vf, Vt = V[:, self.f], V[:, self.t]
        sf = Vf * (self.yff * Vf + self.yft * Vt).conj()
        st = Vt * (self.ytt * Vt + self.yft * Vf).conj()
        if out is not None:
            c = torch.nonzero(out >= 0)[:, 0]
            sf[c, out[c]] = 0
            st[c, out[c]] = 0
        return sf, st

    def power(self, vm, va, out=None):
        V = torch.polar(vm, va)
        sf, st = self.ends(V, out)
        S = vm ** 2 * self.ysh.conj()
        return S.index_add(1, self.f, sf).index_add(1, self.t, st)

    def jacobian(self, vm, va):
        """d(P at non-slack, Q at PQ) / d(theta, V) at one state, dense."""
        V = torch.polar(vm, va)
        Y = torch.zeros((self.n, self.n), dtype=torch.complex64, device=DEV)
        for i, j, y in ((self.f, self.f, self.yff), (self.t, self.t, self.ytt), (self.f, self.t, self.yft),
                        (self.t, self.f, self.yft)):
            Y.index_put_((i, j), y.to(Y.dtype), accumulate=True)
        Y.diagonal().add_(self.ysh.to(Y.dtype))
        V = V.to(Y.dtype)
        I = Y @ V
        W = V[:, None] * (Y * V[None, :]).conj_physical_()  # S_ij = V_i conj(Y_ij V_j)
        del Y
        dth, dv = -1j * W, W / vm.to(torch.float32)[None, :]
        del W
        dth.diagonal().add_(1j * V * I.conj())
        dv.diagonal().add_((V / vm) * I.conj())
        th, vq = self.th, self.vq
        top = torch.cat([dth.real[th][:, th], dv.real[th][:, vq]], 1)
        low = torch.cat([dth.imag[vq][:, th], dv.imag[vq][:, vq]], 1)
        del dth, dv
        return torch.cat([top, low], 0)

    def unknowns(self, a, b):
        return torch.cat([a[..., self.th], b[..., self.vq]], -1)

    def spread(self, x):
        """An unknowns' vector [ncase, nu] as two bus vectors."""
        a = torch.zeros((x.shape[0], self.n), dtype=torch.float64, device=DEV)
        b = torch.zeros_like(a)
        a[:, self.th], b[:, self.vq] = x[:, :len(self.th)], x[:, len(self.th):]
        return a, b

    def branch_jacobian(self, out, vm, va):
        """d(P_f, P_t, Q_f, Q_t) / d(theta_f, theta_t, V_f, V_t) of each case's outaged branch."""
        k = out.clamp(min=0)

        Vf, Vt = torch.polar(vm, va)[self.f[k]], torch.polar(vm, va)[self.t[k]]
        If, It = self.yff[k] * Vf + self.yft[k] * Vt, self.ytt[k] * Vt + self.yft[k] * Vf
        zero = torch.zeros_like(Vf)
        rows = []
        for V, I, d in ((Vf, If, (self.yff[k], self.yft[k])), (Vt, It, (self.yft[k], self.ytt[k]))):
            own = (1, 0) if V is Vf else (0, 1)
            ends = (Vf, Vt)
            rows.append([1j * (ends[q] * own[q] * I.conj() - V * (d[q] * ends[q]).conj()) for q in (0, 1)]
                        + [(ends[q] * own[q] * I.conj() + V * (d[q] * ends[q]).conj()) / ends[q].abs() + zero
                           for q in (0, 1)])
        D = torch.stack([torch.stack(r, 1) for r in rows], 1)
        return torch.cat([D.real, D.imag], 1)


def _lu_solve(lu, b, adjoint=False):
    """Solves with an FP32 factor for rows of b [ncase, nu] (the caller refines in FP64)."""
    scale = b.abs().amax(1, keepdim=True).clamp(min=1e-300)
    x = torch.linalg.lu_solve(*lu, (b / scale).float().T.contiguous(), adjoint=adjoint).T
    return x.double() * scale


def _power_flow(net, P, Q, out=None):
    """States [ncase, n] with P, Q as specified: Newton steps with an FP32
    factor of the first case's Jacobian, each mismatch in FP64; the outaged
    branches enter the steps as corrections of low rank."""
    ncase = P.shape[0]
    vm, va = net.v0.repeat(ncase, 1), net.a0.repeat(ncase, 1)
    target = net.unknowns(P, Q)

    def mismatch(c):
        S = net.power(vm[c], va[c], None if out is None else out[c])
        return target[c] - net.unknowns(S.real, S.imag)

    base = slice(0, 1)
    for _ in range(4):
        lu = torch.linalg.lu_factor(net.jacobian(vm[0], va[0]))
        da, dv = net.spread(_lu_solve(lu, mismatch(base)))
        va[base] += da
        vm[base] += dv
    vm[1:], va[1:] = vm[0], va[0]
    if out is not None:
        place = torch.full((2, net.n), -1, dtype=torch.long, device=DEV)
        place[0, net.th] = torch.arange(len(net.th), device=DEV)
        place[1, net.vq] = torch.arange(len(net.vq), device=DEV) + len(net.th)
        k = out.clamp(min=0)
        at = torch.stack([place[0, net.f[k]], place[0, net.t[k]], place[1, net.f[k]], place[1, net.t[k]]], 1)
        have = (at >= 0) & (out >= 0)[:, None]
        at = at.clamp(min=0)
        M = net.branch_jacobian(out, vm[0], va[0]) * have[:, :, None] * have[:, None, :]
        E = torch.zeros((4 * ncase, target.shape[1]), dtype=torch.float64, device=DEV)
        E[torch.arange(4 * ncase, device=DEV), at.reshape(-1)] = have.reshape(-1).double()
        Z = _lu_solve(lu, torch.where(E.abs().sum(1, keepdim=True) > 0, E, 1e-30)).reshape(ncase, 4, -1)
        Z = Z * have[:, :, None]
        del E
        EZ = torch.gather(Z, 2, at[:, None, :].expand(-1, 4, -1)).transpose(1, 2) * have[:, :, None]
        K = torch.linalg.solve(torch.eye(4, dtype=torch.float64, device=DEV) - M @ EZ, M)
    best, stale = math.inf, 0
    for _ in range(200):
        F = mismatch(slice(None))
        worst = float(F.abs().max())
        best, stale = min(best, worst), 0 if worst < 0.95 * best else stale + 1
        if stale == 5:  # the steps no longer gain: rounding of the mismatch itself
            break
        x = _lu_solve(lu, F)
        if out is not None:
            x = x + torch.einsum("cku,ck->cu", Z, (K @ (torch.gather(x, 1, at) * have)[:, :, None])[:, :, 0])
        da, dv = net.spread(x)
        va += da
        vm += dv
    return vm, va


def _objective_grad(net, vm, va):
    """J = sum (V - 1)^2 + sum P, dJ/dV and dJ/dtheta at every bus."""
    vm, va = vm.detach().requires_grad_(), va.detach().requires_grad_()
    with torch.enable_grad():
        J = ((vm - 1) ** 2).sum(1) + net.power(vm, va).real.sum(1)
        gvm, gva = torch.autograd.grad(J.sum(), (vm, va))
    return J.detach(), gvm, gva


def _transposed_product(net, vm, va, y):
    """J^T y at the state, [ncase, nu]."""
    a, b = net.spread(y)
    vm, va = vm.detach().requires_grad_(), va.detach().requires_grad_()
    with torch.enable_grad():
        S = net.power(vm, va)
        gvm, gva = torch.autograd.grad((S.real * a + S.imag * b).sum(), (vm, va))
    return net.unknowns(gva, gvm)


def exact(case, seed):
    kind = case["kind"]
    if kind == "pack":
        rng = np.random.default_rng(seed)
        states = []
        for c in _pack_grids(case):
            scale = _load_scale(c, 1, rng)
            states.append(_power_flow(_Network(c), _dev(c.pg - c.pd * scale), _dev(-c.qd * scale))
                          if c.n <= EXACT_MAX_PACK_BUS else (None, None))
        if all(s[0] is None for s in states):
            return None
        flat = [[None if s[q] is None else s[q][0] for s in states] for q in (0, 1)]
        return dict(vm=flat[0], va=flat[1], status=None, iters=None)
    if case["n"] > EXACT_MAX_BUS:
        return None
    if kind == "flow":
        c, scale, out = _scenarios(case, seed)
        vm, va = _power_flow(_Network(c), _dev(c.pg - c.pd * scale), _dev(-c.qd * scale),
                             None if out is None else _dev(out).long())
        return dict(vm=vm, va=va, status=None, iters=None)
    c = _grid(case["grid"], case["n"], case["gseed"])
    net = _Network(c)
    if kind == "grad":
        _, psp, qsp = _injections(case, seed)
        vm, va = _power_flow(net, _dev(psp), _dev(qsp))
        J, gvm, gva = _objective_grad(net, vm, va)
        g = net.unknowns(gva, gvm)
        lu = torch.linalg.lu_factor(net.jacobian(vm[0], va[0]))
        y = torch.zeros_like(g)
        best, stale = math.inf, 0
        for _ in range(200):
            r = g - _transposed_product(net, vm, va, y)
            worst = float(r.abs().max())
            best, stale = min(best, worst), 0 if worst < 0.95 * best else stale + 1
            if stale == 5:
                break
            y = y + _lu_solve(lu, r, adjoint=True)
        dP, dQ = net.spread(y)
        return dict(vm=vm, va=va, J=J, dP=dP, dQ=dQ)
    if kind == "states":
        scale = _load_scale(c, case["ncase"], np.random.default_rng(seed))
        vm, va = (_dev(a) for a in _states(case, seed))
        S = net.power(vm, va)
        dp = torch.where(net.btype != gridgen.SLACK, _dev(c.pg - c.pd * scale) - S.real, 0.0)
        dq = torch.where(net.btype == gridgen.PQ, _dev(-c.qd * scale) - S.imag, 0.0)
        J, gvm, gva = _objective_grad(net, vm, va)
        sf, st = net.ends(torch.polar(vm, va))
        return dict(dp=dp, dq=dq, mis=torch.maximum(dp.abs().amax(1), dq.abs().amax(1)), J=J, gva=gva, gvm=gvm,
                    flows=torch.stack([sf.real, sf.imag, st.real, st.imag], 2), loss=S.real.sum(1))
    x = []
    series = _dev(c.status / c.x)
    for which, b in enumerate(_rhs(case, seed)):
        A = torch.zeros((c.n, c.n), dtype=torch.float64, device=DEV)
        if which == 0:  # B': 1/x between buses
            parts = ((net.f, net.f, series), (net.t, net.t, series), (net.f, net.t, -series), (net.t, net.f, -series))
        else:           # B'': -Im(Y)
            parts = ((net.f, net.f, -net.yff.imag), (net.t, net.t, -net.ytt.imag), (net.f, net.t, -net.yft.imag),
                     (net.t, net.f, -net.yft.imag))
            A.diagonal().sub_(net.ysh.imag)
        for i, j, v in parts:
            A.index_put_((i, j), v, accumulate=True)
        keep = net.th if which == 0 else net.vq
        A = A[keep][:, keep]
        lu = torch.linalg.lu_factor(A.float())
        b = _dev(b)
        y = torch.zeros_like(b)
        for _ in range(8):
            y = y + _lu_solve(lu, b - y @ A)
        x.append(y)
    return dict(x=x)

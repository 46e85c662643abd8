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

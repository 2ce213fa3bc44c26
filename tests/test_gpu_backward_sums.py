"""Long sums of the mixed adjoint: rounding errors that have one sign in every term do not average out,
so none may be left in the exponent gradient of a shell that thousands of quartets share."""
import numpy as np
import pytest
import torch

from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


def gradient(shells, q, precision):
    plan = api.eri_plan_create(shells, q, precision=precision)
    G = torch.ones(api.eri_output_bytes(plan, 0)[0] // 8, dtype=torch.float64, device="cuda")
    dR = torch.empty((shells.n, 3), dtype=torch.float64, device="cuda")
    da = torch.empty(len(shells.exps), dtype=torch.float64, device="cuda")
    api.eri_backward(plan, G, dR, da)
    api.eri_sync(plan)
    return dR.cpu().numpy(), da.cpu().numpy()


@pytest.mark.parametrize("place", [0, 3])
@pytest.mark.parametrize("above", [False, True])
def test_exponent_of_a_shared_shell(place, above):
    """E-term coefficient 3 / (4 alpha) halfway between two FP32 numbers: rounding it costs 2^-24 of every
    term (all are positive), times the ratio of the E-term to the gradient (at least 1).  The other
    roundings of a term, about ten of 2^-25 on average, differ between quartets and leave
    10 2^-25 / sqrt(6000) = 4e-9 of the sum; the bound lies between the two, at 2^-25."""
    rng = np.random.default_rng(11 + place)
    n = 64
    ulp = 2.0 ** -23
    coef = 1.0 + (20 + 0.5) * ulp + (0.02 if above else -0.02) * ulp  # 3 / (4 alpha), rounded down or up
    exps = np.exp(rng.uniform(np.log(0.3), np.log(3.0), n))
    exps[0] = 0.75 / coef
    shells = W.make_shellset(rng.uniform(-0.8, 0.8, (n, 3)), np.zeros(n, dtype=np.int32), list(exps[:, None]),
                             [np.ones(1)] * n)
    q = rng.integers(1, n, (6000, 4)).astype(np.int32)
    q[:, place] = 0
    want = gradient(shells, q, "fp64")[1][0]
    got = gradient(shells, q, "mixed")[1][0]
    assert abs(got - want) <= 2.0 ** -25 * abs(want)

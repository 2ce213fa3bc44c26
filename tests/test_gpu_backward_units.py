"""The adjoint over units: quartets of uneven contraction degree, so that the units of a group change
their quartet and their primitives at every kind of boundary (between two groups of units, at the end
of a batch and of a CTA's share), against the oracle derivative."""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cls,n", [((0, 0, 0, 0), 400), ((1, 1, 0, 0), 90), ((2, 1, 1, 0), 40), ((2, 2, 2, 2), 9),
                                   ((1, 2, 2, 2), 1), ((3, 0, 3, 1), 12), ((3, 3, 2, 0), 7)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_uneven_units(cls, n, precision):
    if precision == "fp64" and 3 in cls:
        pytest.skip("the FP64 adjoint serves shells up to d")
    rng = np.random.default_rng(n + sum(cls))
    degrees = (1, 4, 2, 5, 3)
    Ls = sorted(set(cls))
    L = [l for l in Ls for _ in degrees]
    ks = [k for _ in Ls for k in degrees]
    shells = W.make_shellset(rng.uniform(-1.5, 1.5, (len(L), 3)), L,
                             [0.25 * 1.8 ** np.arange(k) * rng.uniform(0.8, 1.2, k) for k in ks],
                             [rng.uniform(0.1, 1.0, k) for k in ks])
    q = np.stack([rng.integers(0, len(degrees), n) + len(degrees) * Ls.index(l) for l in cls], axis=1).astype(np.int32)
    sizes = oracle.quartet_sizes(shells, q)
    offs = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(sizes, out=offs[1:])
    G = rng.standard_normal(int(offs[-1]))
    plan = api.eri_plan_create(shells, q, precision=precision)  # one class: the caller's order
    dR = torch.empty((shells.n, 3), dtype=torch.float64, device="cuda")
    da = torch.empty(len(shells.exps), dtype=torch.float64, device="cuda")
    api.eri_backward(plan, torch.tensor(G, device="cuda"), dR, da)
    api.eri_sync(plan)
    rR, ra = oracle.eri_grad_batch(shells, q, G, offs)
    # of the largest component: the FP64 parity bound, and the mixed adjoint's
    tol = 1e-10 if precision == "fp64" else 2e-5
    assert np.max(np.abs(dR.cpu().numpy() - rR)) <= tol * np.abs(rR).max()
    assert np.max(np.abs(da.cpu().numpy() - ra)) <= tol * np.abs(ra).max()

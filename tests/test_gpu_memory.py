"""Device memory that a plan and its calls take: what their own classes need."""
import numpy as np
import pytest
import torch

from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20


def taken(f):
    """Device memory (bytes) that f() leaves taken, and its result; f has run once before, so that
    modules and the runtime's own pools are loaded."""
    f()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    r = f()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0], r


@pytest.mark.parametrize("precision,classes", [("mixed", [(0, 0, 0, 0), (1, 0, 0, 0), (1, 1, 0, 0)]),
                                               ("fp64", [(0, 0, 0, 0), (1, 0, 0, 0), (1, 0, 1, 0)]),
                                               ("fp64", [(4, 0, 0, 0), (0, 0, 0, 0)])])
def test_primitive_calls_without_scratch(precision, classes):
    """Classes whose kernels form everything in registers, and FP64 values of classes with a g shell,
    leave no scratch behind (654 MB where a class does need it)."""
    rng = np.random.default_rng(2)
    Ls = (0, 1, 2, 3, 4)
    pool = W.random_primitive_pool(rng, 8, Ls=Ls)
    q = np.concatenate([W.random_class_quartets(rng, c, 50, 8, Ls=Ls) for c in classes])
    out = torch.zeros(sum(50 * W.quartet_size(*c) for c in classes), dtype=torch.float64, device="cuda")
    packed, scales = torch.zeros(50000, dtype=torch.int32, device="cuda"), torch.zeros(200, device="cuda")

    def call():
        plan = api.eri_plan_create(pool, q, precision=precision)
        api.eri_compute(plan, out)
        if 4 not in classes[0]:
            api.eri_compute_compressed(plan, 16, packed, scales)
            api.eri_compute_compressed_batched(plan, 16, packed, scales)
        api.eri_sync(plan)
        return plan

    left, plan = taken(call)
    assert left < 32 * MB
    plan.destroy()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_small_contracted_plan(precision):
    """A contracted plan's scratch follows its classes: of these quartets of p and d shells, K = 2, a class
    has at most 12, 192 primitive quartets of up to 1,296 outputs and 117 record values, 2.2 MB in FP64 on a
    stream for each of 7 classes.  All of it is made with the plan."""
    rng = np.random.default_rng(4)
    pool = W.random_contracted_pool(rng, 2, K=2, Ls=(1, 2))
    q = np.array([(i, j, k, l) for i in range(4) for j in range(i + 1) for k in range(i + 1) for l in range(k + 1)],
                 dtype=np.int32)
    assert max(np.unique(pool.L[q], axis=0, return_counts=True)[1]) == 12

    left, plan = taken(lambda: api.eri_plan_create(pool, q, precision=precision))
    assert left < 32 * MB
    out = torch.empty(api.eri_output_bytes(plan, 0)[0] // 8, dtype=torch.float64, device="cuda")
    more, _ = taken(lambda: api.eri_compute(plan, out))
    assert more < 4 * MB
    plan.destroy()

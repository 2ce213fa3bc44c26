"""Classes with a g shell in one launch: a call over all classes runs them in sets, the same values and
codes bit for bit as a launch per class (the same tiles in the same order of operations), with s to f
classes beside them, with classes switched to FP64 and with packed tiles that share words."""
import itertools

import numpy as np
import pytest
import torch

from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu

LS = (0, 1, 2, 3, 4)
CLASSES = list(itertools.product(LS, repeat=4))


# few: one to three quartets of a class; many: more than a tile (64 quartets) of the small ones
@pytest.mark.parametrize("count", ["few", "many"])
@pytest.mark.parametrize("K,precision,bits", [(1, "mixed", 16), (1, "fp64", 0), (1, "mixed", 7), (2, "mixed", 12),
                                              (2, "fp64", 0)])
def test_sets_equal_the_per_class_launches(count, K, precision, bits):
    rng = np.random.default_rng(K + bits)
    pool = (W.random_primitive_pool(rng, 4, Ls=LS) if K == 1 else W.random_contracted_pool(rng, 4, K=K, Ls=LS))
    q = []
    for i, c in enumerate(CLASSES):
        n = 1 + i % 3 if count == "few" else 1 + min(200, 20000 // W.quartet_size(*c))
        if 4 in c or i % 5 == 0:
            q.append(W.random_class_quartets(rng, c, n, 4, Ls=LS))
    plan = api.eri_plan_create(pool, np.concatenate(q), precision=precision)
    ids = [W.class_id(*c) for c in CLASSES if 4 in c]
    if precision == "mixed":  # two sets' worth of classes in each precision
        for c in ids[::2]:
            api.eri_plan_set_class_precision(plan, c, "fp64")
    for c in ids:
        assert api.eri_plan_class_info(plan, c)[0] > 0
    if bits == 0:
        whole = torch.full((api.eri_output_bytes(plan, 0)[0] // 8,), -1.0, dtype=torch.float64, device="cuda")
        each = whole.clone()
        api.eri_compute(plan, whole)
        for i in range(625):
            api.eri_compute_class(plan, W.class_id(*CLASSES[i]), each)
        api.eri_sync(plan)
        assert torch.equal(whole, each)
        return
    nb, sb = api.eri_output_bytes(plan, bits)
    out = [(torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda"),
            torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")) for _ in range(2)]
    api.eri_compute_compressed(plan, bits, *out[0])
    for c in CLASSES:
        api.eri_compute_compressed_class(plan, W.class_id(*c), bits, *out[1])
    api.eri_sync(plan)
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])

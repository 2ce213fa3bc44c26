"""Tiles of the run-time-L kernel: their length follows the number of quartets and of streams, and in FP64
a class's recursion runs on lanes or on one thread.  The values of a call over one class, of a call over
all classes (other tiles) and the codes of both are the same bit for bit, and the values are the oracle's.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu

LS = (0, 1, 2, 3, 4)


# few planes (one thread per recursion), many planes and one quartet per tile (lanes), many planes and a
# full batch (one thread); one quartet, one per tile, one more than that, several per tile
@pytest.mark.parametrize("cls", [(4, 0, 0, 0), (0, 4, 2, 1), (4, 1, 2, 2), (4, 3, 3, 1), (4, 2, 4, 1)])
@pytest.mark.parametrize("n", [1, 304, 305, 1301])
def test_tiles(cls, n):
    rng = np.random.default_rng(n + sum(cls))
    pool = W.random_primitive_pool(rng, 6, Ls=LS)
    others = [c for c in [(4, 0, 1, 0), (4, 4, 0, 0), (1, 4, 0, 0), (3, 4, 0, 0)] if c != cls]
    q = np.concatenate([W.random_class_quartets(rng, cls, n, 6, Ls=LS)] +
                       [W.random_class_quartets(rng, c, 2, 6, Ls=LS) for c in others])
    neri, cid = W.quartet_size(*cls), W.class_id(*cls)
    plan = api.eri_plan_create(pool, q, precision="fp64")
    first = api.eri_plan_class_info(plan, cid)[3]
    whole = torch.full((api.eri_output_bytes(plan, 0)[0] // 8,), -1.0, dtype=torch.float64, device="cuda")
    each = whole.clone()
    api.eri_compute(plan, whole)
    api.eri_compute_class(plan, cid, each)
    api.eri_sync(plan)
    got = each[first:first + n * neri]
    assert torch.equal(whole[first:first + n * neri], got)
    some = np.unique(np.linspace(0, n - 1, 5).astype(int))
    ref, offs = oracle.eri_batch(pool, q[some])
    got = got.cpu().numpy().reshape(n, neri)
    for k, i in enumerate(some):  # parity bound of the FP64 path
        r = ref[offs[k]:offs[k + 1]]
        assert np.all(np.abs(got[i] - r) <= np.maximum(1e-12, 1e-10 * np.abs(r)))
    for precision in ("fp64", "mixed"):
        plan = api.eri_plan_create(pool, q, precision=precision)
        nb, sb = api.eri_output_bytes(plan, 11)
        out = [(torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda"),
                torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")) for _ in range(2)]
        api.eri_compute_compressed(plan, 11, *out[0])
        for c in [cls, *others]:
            api.eri_compute_compressed_class(plan, W.class_id(*c), 11, *out[1])
        api.eri_sync(plan)
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])

"""Contracted quartets longer than a span of the scratch, on neighbouring streams: a quartet's sum (in FP32
with its compensation) is carried through several spans, and each stream keeps its own.

[ff|ff] and [ff|fd] have quartets of up to 4,096 primitive quartets.  A call over sixteen classes gives
each stream a sixteenth of the scratch, one class at a time has all of it, and a quartet alone takes one
span; the values and codes are the same bit for bit."""
import numpy as np
import pytest
import torch

from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu

F, D = [0, 1, 2, 3], [4, 5]  # shells of the long quartets, by degree 8, 7, 8, 6 and 8, 5


def basis(rng):
    Ls = [3, 3, 3, 3, 2, 2] + [0, 1, 2]
    degrees = [8, 7, 8, 6, 8, 5] + [1, 2, 1]
    exps = [0.2 * 1.6 ** np.arange(k) * rng.uniform(0.8, 1.2, k) for k in degrees]
    return W.make_shellset(rng.uniform(-1.5, 1.5, (len(Ls), 3)), Ls, exps, [rng.uniform(0.1, 1.0, k) for k in degrees])


def quartets():
    """[ff|ff] and [ff|fd] of uneven length, and one quartet each of fourteen classes of s, p and d shells."""
    long = [(0, 2, 0, 2), (0, 1, 2, 3), (2, 2, 2, 0), (3, 0, 1, 2), (2, 0, 2, 1), (0, 0, 0, 0), (1, 1, 0, 2), (2, 3, 0, 0)]
    second = [(0, 2, 0, 4), (2, 2, 0, 5), (0, 0, 2, 4), (1, 2, 0, 4)]
    small = [(6 + a, 6 + b, 6 + c, 6 + d) for a in range(3) for b in range(3) for c in range(3) for d in range(3)][:14]
    return np.array(long + second + small, dtype=np.int32), len(long), len(second)


@pytest.mark.parametrize("precision,bits", [("fp64", 0), ("fp64", 12), ("mixed", 0), ("mixed", 16)])
def test_long_quartets_on_neighbouring_streams(precision, bits):
    shells = basis(np.random.default_rng(8))
    q, n_ff, n_fd = quartets()
    plan = api.eri_plan_create(shells, q, precision=precision)
    ffff, fffd = W.class_id(3, 3, 3, 3), W.class_id(3, 3, 3, 2)
    units = np.prod(shells.nprim[q], axis=1)
    # [ff|ff] takes more than one span of the whole scratch, so a share holds less than a sixteenth of its
    # units, and the quartets of 4,096 are cut twice at least
    assert len(np.unique(shells.L[q], axis=0)) == 16
    assert api.eri_plan_class_launches(plan, ffff) >= 8 and units[:n_ff].sum() < 16 * 4096 // 2
    assert units[:n_ff].max() == 4096 and units[n_ff:n_ff + n_fd].max() == 4096
    if bits == 0:
        outs = [[torch.full((api.eri_output_bytes(plan, 0)[0] // 8,), -1.0, dtype=torch.float64, device="cuda")]
                for _ in range(2)]
        api.eri_compute(plan, *outs[0])
        for c in range(256):
            api.eri_compute_class(plan, c, *outs[1])
    else:
        nb, sb = api.eri_output_bytes(plan, bits)
        outs = [[torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda"),
                 torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")] for _ in range(2)]
        api.eri_compute_compressed(plan, bits, *outs[0])
        for c in range(256):
            api.eri_compute_compressed_class(plan, c, bits, *outs[1])
    api.eri_sync(plan)
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    if bits:
        return
    # the long quartets alone, each in one span
    for cls, at, n in ((ffff, 0, n_ff), (fffd, n_ff, n_fd)):
        first, neri = api.eri_plan_class_info(plan, cls)[3], W.quartet_size(*W.class_of_id(cls))
        for i in range(n):
            alone = api.eri_plan_create(shells, q[at + i:at + i + 1], precision=precision)
            assert api.eri_plan_class_launches(alone, cls) == 4
            out = torch.empty(neri, dtype=torch.float64, device="cuda")
            api.eri_compute(alone, out)
            api.eri_sync(alone)
            assert torch.equal(out, outs[0][0][first + i * neri:first + (i + 1) * neri])
            alone.destroy()

"""Codes of the FP32 kernels against the values of the same kernels.

A mixed plan's values are FP32 numbers, and eps (Eq. 9), the scaling and the rounding (Eq. 10) are
FP32 operations, so the codes follow from the values exactly: eps = b_max / M, q = round half away of
x * (1 / eps).  The quartet counts sit at the edges of the kernels' tiles (one quartet, a ragged
tile, more tiles than CTAs of the grid) and the widths at those of the packing: whole bytes, groups
of eight codes, words gathered one by one, more than 22 bits.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu

# all outputs of one a per thread; of one (a, c); b-chunks; one quartet per tile
CLASSES = [((2, 1, 2, 0), 70001), ((2, 1, 2, 0), 1), ((2, 2, 2, 2), 9001), ((3, 2, 3, 2), 2603),
           ((3, 3, 3, 3), 1301), ((1, 3, 0, 1), 2000), ((3, 1, 1, 1), 3)]


@pytest.mark.parametrize("cls,n", CLASSES)
@pytest.mark.parametrize("bits", [3, 8, 11, 12, 16, 17, 20, 23, 24])
def test_codes_follow_from_the_values(cls, n, bits):
    rng = np.random.default_rng(n + bits)
    Ls = tuple(sorted(set(cls)))
    pool = W.random_primitive_pool(rng, 24, Ls=Ls)
    q = W.random_class_quartets(rng, cls, n, 24, Ls=Ls)
    plan = api.eri_plan_create(pool, q, precision="mixed")
    neri = W.quartet_size(*cls)
    out = torch.full((n * neri,), -1.0, dtype=torch.float64, device="cuda")
    nb, sb = api.eri_output_bytes(plan, bits)
    packed = torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda")
    scales = torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")
    api.eri_compute(plan, out)
    api.eri_compute_compressed(plan, bits, packed, scales)
    api.eri_sync(plan)
    x = out.cpu().numpy().reshape(n, neri)
    assert np.array_equal(x, x.astype(np.float32))
    x = x.astype(np.float32)
    M = np.float32(2 ** (bits - 1) - 1)
    bmax = np.abs(x).max(axis=1)
    eps = bmax / M
    np.testing.assert_array_equal(scales.cpu().numpy(), eps)
    keep = bmax > 1e-25  # the reciprocal of a smaller eps can leave the FP32 range
    with np.errstate(divide="ignore", over="ignore", invalid="ignore"):
        v = (x * (np.float32(1) / eps)[:, None]).astype(np.float64)
    want = np.clip(np.sign(v) * np.floor(np.abs(v) + 0.5), -float(M), float(M))
    words = packed.cpu().numpy().view(np.uint32)
    codes = oracle.unpack_bits(words, n * neri, bits).reshape(n, neri)
    np.testing.assert_array_equal(codes[keep], want[keep])
    used = (n * neri * bits + 31) // 32
    assert np.all(words[used:] == 0)  # zero up to the segment's end
    if n * neri * bits % 32:
        assert words[used - 1] >> (n * neri * bits % 32) == 0

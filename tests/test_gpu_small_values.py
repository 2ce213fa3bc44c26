"""Codes of quartets whose eps (Eq. 9) is a subnormal FP32 number.

Rounding eps there costs more than the half unit of a normal one, so x / eps of the largest value can
round to M + 1; the codes stay within +-M all the same (Eq. 10), at every width.  The values of the
quartets are scaled into that range by the coefficient of their first shell.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


def own_shells(rng, cls, n, coefs):
    """Quartet i over shells 4 i .. 4 i + 3, coefs[i] the coefficient of its first one."""
    m = 4 * n
    c = np.ones(m)
    c[::4] = coefs
    shells = W.make_shellset(rng.uniform(-1, 1, (m, 3)), np.tile(cls, n), list(rng.uniform(0.3, 3.0, (m, 1))),
                             list(c[:, None]))
    return shells, np.arange(m, dtype=np.int32).reshape(-1, 4)


# the rows kernel with all outputs of one a per thread and of one (a, c); a thread per quartet
@pytest.mark.parametrize("cls,n", [((2, 1, 2, 0), 12000), ((3, 2, 3, 2), 600), ((2, 1, 1, 0), 12000)])
@pytest.mark.parametrize("bits", [8, 16, 20, 21, 22, 23, 24])
def test_codes_stay_within_their_range(cls, n, bits):
    neri, M = W.quartet_size(*cls), 2 ** (bits - 1) - 1
    values = []
    coefs = np.ones(n)
    for step in range(2):
        shells, q = own_shells(np.random.default_rng(5), cls, n, coefs)
        plan = api.eri_plan_create(shells, q, precision="mixed")
        out = torch.empty(n * neri, dtype=torch.float64, device="cuda")
        api.eri_compute(plan, out)
        api.eri_sync(plan)
        values = out.cpu().numpy().reshape(n, neri)
        if step == 0:  # eps from 2^-128 (1 / eps near the largest FP32 number) to 2^-125
            coefs = M * 2.0 ** np.random.default_rng(9).uniform(-128, -125, n) / np.abs(values).max(axis=1)
    nb, sb = api.eri_output_bytes(plan, bits)
    packed = torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda")
    scales = torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")
    api.eri_compute_compressed(plan, bits, packed, scales)
    api.eri_sync(plan)
    x = values.astype(np.float32)
    assert np.array_equal(x, values)
    eps = np.abs(x).max(axis=1) / np.float32(M)
    np.testing.assert_array_equal(scales.cpu().numpy(), eps)
    with np.errstate(over="ignore"):
        inv = np.float32(1) / eps
    keep = np.isfinite(inv)
    assert keep.sum() > 0.9 * n and (eps[keep] < 2.0 ** -126).sum() > 0.5 * n
    v = (x[keep] * inv[keep, None]).astype(np.float64)
    want = np.clip(np.sign(v) * np.floor(np.abs(v) + 0.5), -M, M)
    codes = oracle.unpack_bits(packed.cpu().numpy().view(np.uint32), n * neri, bits).reshape(n, neri)
    np.testing.assert_array_equal(codes[keep], want)

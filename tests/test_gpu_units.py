"""Contracted quartets computed as units (primitive quartets) and summed afterwards.

A class's units are cut into spans that fill the scratch, and a quartet may be cut between two
spans.  The per-class call works in the whole scratch and the call over all classes in an eighth
of it, so they cut the same quartets at different places: the sums have to agree bit for bit, and
with the oracle on the quartets that are cut.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


def uneven_shells(rng, Ls, degrees):
    exps = [0.3 * 1.7 ** np.arange(k) * rng.uniform(0.8, 1.2, k) for k in degrees]
    coefs = [rng.uniform(0.1, 1.0, k) for k in degrees]
    return W.make_shellset(rng.uniform(-1.5, 1.5, (len(Ls), 3)), Ls, exps, coefs)


# [ff|ff]: 10,000 outputs, an eighth of the scratch holds about 1,000 (FP64) or 2,000 (FP32) units;
# [ss|ss]: one output, tiles of 128 quartets; [fs|ps]: odd code counts, shared words at tile edges
@pytest.mark.parametrize("L,degrees,n", [((3, 3, 3, 3), (6, 5, 1, 4), 14), ((0, 0, 0, 0), (1, 6, 3, 2), 300),
                                         ((3, 0, 1, 0), (1, 2, 1, 6, 3), 131)])
@pytest.mark.parametrize("precision,bits", [("fp64", 0), ("fp64", 12), ("mixed", 16), ("mixed", 7)])
def test_cut_quartets_sum_to_the_same(L, degrees, n, precision, bits):
    rng = np.random.default_rng(sum(L) + n)
    Ls, ks = [], []
    for l in sorted(set(L)):
        Ls += [l] * len(degrees)
        ks += list(degrees)
    shells = uneven_shells(rng, Ls, ks)
    by = {l: [i for i, x in enumerate(Ls) if x == l] for l in set(L)}
    q = np.stack([rng.choice(by[l], n) for l in L], axis=1).astype(np.int32)
    plan = api.eri_plan_create(shells, q, precision=precision)
    cls = W.class_id(*L)
    outs = []
    for whole in (False, True):
        if bits == 0:
            out = torch.full((api.eri_output_bytes(plan, 0)[0] // 8,), -1.0, dtype=torch.float64, device="cuda")
            api.eri_compute_class(plan, cls, out) if whole else api.eri_compute(plan, out)
            api.eri_sync(plan)
            outs.append((out.cpu().numpy(),))
        else:
            nb, sb = api.eri_output_bytes(plan, bits)
            packed = torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda")
            scales = torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")
            if whole:
                api.eri_compute_compressed_class(plan, cls, bits, packed, scales)
            else:
                api.eri_compute_compressed(plan, bits, packed, scales)
            api.eri_sync(plan)
            outs.append((packed.cpu().numpy(), scales.cpu().numpy()))
    for x, y in zip(*outs):
        np.testing.assert_array_equal(x, y)
    some = np.arange(n) if np.prod(L) == 0 else np.array([0, 6, n - 1])
    ref, offs = oracle.eri_batch(shells, q[some])
    neri = W.quartet_size(*L)
    for k, i in enumerate(some):
        r = ref[offs[k]:offs[k + 1]]
        if bits == 0:
            got = outs[0][0][i * neri:(i + 1) * neri]
            # parity bound of the FP64 path (1e-12 absolute, 1e-10 relative)
            assert np.all(np.abs(got - r) <= np.maximum(1e-12, 1e-10 * np.abs(r)))
            continue
        codes = oracle.unpack_bits(outs[0][0].view(np.uint32), n * neri, bits)[i * neri:(i + 1) * neri]
        eps = outs[0][1][i]
        # half a step, plus the path's own error: FP64 rounding, or 1e-5 of b_max in FP32
        own = 1e-10 if precision == "fp64" else 1e-5
        assert np.max(np.abs(codes * float(eps) - r)) <= 0.5 * eps * (1 + 1e-6) + own * np.abs(r).max()

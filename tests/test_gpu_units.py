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
    # a quartet of another class, so that the call over all classes divides the scratch
    other = 1 if set(L) == {0} else 0
    Ls.append(other)
    ks.append(2)
    shells = uneven_shells(rng, Ls, ks)
    by = {l: [i for i, x in enumerate(Ls[:-1]) if x == l] for l in set(L)}
    q = np.stack([rng.choice(by[l], n) for l in L], axis=1).astype(np.int32)
    plan = api.eri_plan_create(shells, np.concatenate([q, np.full((1, 4), len(Ls) - 1, dtype=np.int32)]),
                               precision=precision)
    cls = W.class_id(*L)
    fp64_first = api.eri_plan_class_info(plan, cls)[3]
    first = api.eri_plan_class_info(plan, cls)[2]
    outs = []
    for whole in (False, True):
        if bits == 0:
            out = torch.full((api.eri_output_bytes(plan, 0)[0] // 8,), -1.0, dtype=torch.float64, device="cuda")
            api.eri_compute_class(plan, cls, out) if whole else api.eri_compute(plan, out)
            api.eri_sync(plan)
            outs.append((out.cpu().numpy()[fp64_first:fp64_first + n * W.quartet_size(*L)],))
        else:
            nb, sb = api.eri_output_bytes(plan, bits)
            packed = torch.full((nb // 4,), -1, dtype=torch.int32, device="cuda")
            scales = torch.full((sb // 4,), -1.0, dtype=torch.float32, device="cuda")
            if whole:
                api.eri_compute_compressed_class(plan, cls, bits, packed, scales)
            else:
                api.eri_compute_compressed(plan, bits, packed, scales)
            api.eri_sync(plan)
            off, seg = api.eri_packed_class_offset(plan, bits, cls)
            outs.append((packed.cpu().numpy()[off // 4:(off + seg) // 4], scales.cpu().numpy()[first:first + n]))
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


def test_classes_cut_side_by_side():
    """Two classes on neighbouring streams, both cut inside quartets: each keeps its own carried sums."""
    rng = np.random.default_rng(6)
    shells = uneven_shells(rng, [2, 3, 3, 3, 3], [6, 6, 6, 6, 6])
    q = np.array([[1, 2, 3, 4], [4, 3, 2, 1], [1, 2, 3, 0], [2, 4, 1, 0]], dtype=np.int32)
    plan = api.eri_plan_create(shells, q, precision="fp64")
    n = api.eri_output_bytes(plan, 0)[0] // 8
    whole, each = (torch.full((n,), -1.0, dtype=torch.float64, device="cuda") for _ in range(2))
    api.eri_compute(plan, whole)
    for L in ((3, 3, 3, 3), (3, 3, 3, 2)):
        api.eri_compute_class(plan, W.class_id(*L), each)
    api.eri_sync(plan)
    np.testing.assert_array_equal(whole.cpu().numpy(), each.cpu().numpy())

"""Calls over all classes spread them over side streams; to the caller they stay work of the stream
that was passed: ordered after what was queued there before and before what is queued after, also
with two plans on two streams and inside a captured graph."""
import numpy as np
import pytest
import torch

from paper_2303_13632_gb300 import api, workloads as W

pytestmark = pytest.mark.gpu


def make_plan(K, precision, seed):
    rng = np.random.default_rng(seed)
    Ls = (0, 1, 2, 3)
    pool = (W.random_primitive_pool(rng, 8, Ls=Ls) if K == 1 else
            W.random_contracted_pool(rng, 8, K=K, Ls=Ls))
    cls = [W.class_of_id(c) for c in range(0, 256, 3)]
    q = np.concatenate([W.random_class_quartets(rng, c, 5, 8, Ls=Ls) for c in cls])
    return api.eri_plan_create(pool, q, precision=precision), cls


def by_class(plan, cls, n):
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    for c in cls:
        api.eri_compute_class(plan, W.class_id(*c), out)
    api.eri_sync(plan)
    return out


@pytest.mark.parametrize("K,precision", [(1, "fp64"), (1, "mixed"), (3, "fp64"), (3, "mixed")])
def test_calls_are_ordered_on_the_stream(K, precision):
    plans = [make_plan(K, precision, s) for s in (1, 2)]
    n = [api.eri_output_bytes(p, 0)[0] // 8 for p, _ in plans]
    want = [by_class(p, c, m).clone() for (p, c), m in zip(plans, n)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in plans]
    outs = [torch.zeros(m, dtype=torch.float64, device="cuda") for m in n]
    copies = [[], []]
    torch.cuda.synchronize()
    for _ in range(4):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                outs[i].fill_(-1.0)
                api.eri_compute(plans[i][0], outs[i], s)
                copies[i].append(outs[i].clone())
    torch.cuda.synchronize()
    for i in range(2):
        for c in copies[i]:
            assert torch.equal(c, want[i])


@pytest.mark.parametrize("K", [1, 2])
def test_captured_call(K):
    """A contracted plan's first call can be captured (it allocates nothing); a primitive plan's can
    once a call has made its scratch."""
    plan, cls = make_plan(K, "mixed", 3)
    n = api.eri_output_bytes(plan, 0)[0] // 8
    other = make_plan(K, "mixed", 5)[0]  # another plan's call loads the kernels
    api.eri_compute(other, torch.zeros(api.eri_output_bytes(other, 0)[0] // 8, dtype=torch.float64, device="cuda"))
    api.eri_sync(other)
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    want = by_class(plan, cls, n) if K == 1 else None
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        api.eri_compute(plan, out, s)
    if want is None:
        want = by_class(plan, cls, n)
    for _ in range(2):
        out.fill_(-1.0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)


def test_gradient_on_side_streams_matches_itself():
    """The adjoint's classes share dR and dalpha: sums in another order, FP64 rounding apart."""
    plan, _ = make_plan(2, "mixed", 4)
    n = api.eri_output_bytes(plan, 0)[0] // 8
    G = torch.randn(n, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    s = torch.cuda.Stream()
    got = []
    for st in (None, s, s):
        dR = torch.full((32, 3), 7.0, dtype=torch.float64, device="cuda")
        da = torch.full((64,), 7.0, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        api.eri_backward(plan, G, dR, da, st)
        api.eri_sync(plan, st)
        got.append((dR.cpu().numpy(), da.cpu().numpy()))
    for dR, da in got[1:]:
        np.testing.assert_allclose(dR, got[0][0], rtol=0, atol=1e-12 * np.abs(got[0][0]).max())
        np.testing.assert_allclose(da, got[0][1], rtol=0, atol=1e-12 * np.abs(got[0][1]).max())

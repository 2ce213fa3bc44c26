"""The work this library is timed on, through its public entry points.

`listed()` gives the fixed cases and `draw(rng)` further ones of the same ranges; `prepare` makes
what a program holds before the call (shells, quartet list, plan, output buffers), `run` is one
call as such a program makes it, `work` its unavoidable bytes and flops, and `exact` the same
result from a plain 64-bit evaluation in torch that shares nothing with the library.

Kinds of case:
  class     one quartet class of primitive shells, FP64 ERIs or n-bit codes (a building block of
            every larger job, and the smallest calls)
  sweep     all 256 classes of s..f shells in one plan (the bulk form: integrals of a large system
            computed and kept compressed, or delivered in FP64)
  step      one step of a geometry loop: a small contracted molecule is moved and its unique ERIs
            are recomputed in FP64
  molecule  contracted unique quartets of a larger molecule (an even share of the device's
            enumeration), as 16-bit codes: the CUDA-graph form, the single-launch work queue, or
            the per-class launches
  gradient  forward and backward through autograd (forces and exponent gradients of a contracted
            basis), in FP64 or with FP32 parameters and mixed arithmetic
  gshell    the 369 classes with a g shell, as codes
  fock      Coulomb and exchange matrices from stored 16-bit ERIs (one SCF iteration)
  chunks    codes re-laid into per-quartet 512-bit chunks
"""
import math

import numpy as np
import torch

from paper_2303_13632_gb300 import api
from paper_2303_13632_gb300.autograd import EriGeometry
from paper_2303_13632_gb300.workloads import ShellSet

POOL = 4096      # shells per angular momentum of the sweep (the benchmark's pool)
GPOOL = 2048     # the same for the classes with a g shell and the gradient workload


def ncart(L):
    return (L + 1) * (L + 2) // 2


def size(c):
    return ncart(c[0]) * ncart(c[1]) * ncart(c[2]) * ncart(c[3])


def class_id(c):
    if max(c) <= 3:
        return ((c[0] * 4 + c[1]) * 4 + c[2]) * 4 + c[3]
    return 256 + ((c[0] * 5 + c[1]) * 5 + c[2]) * 5 + c[3]


def all_classes(Ls):
    return sorted(((a, b, c, d) for a in Ls for b in Ls for c in Ls for d in Ls), key=class_id)


def listed():
    return [
        # 10,000 fresh [pp|pp] quartets in FP64: the smallest call, one class, one launch pair
        {"name": "class_pppp_fp64", "kind": "class", "cls": "pppp", "quartets": 10000, "pool": 0, "precision": "fp64", "bits": 0},
        # one high class, an odd count and a width that straddles words: a block of a bulk job
        {"name": "class_fdfd_12bit", "kind": "class", "cls": "fdfd", "quartets": 40001, "pool": 2048, "precision": "mixed", "bits": 12},
        # a geometry optimisation or dynamics step of a diatomic: many classes, few quartets each
        {"name": "step_diatomic_fp64", "kind": "step", "atoms": 2, "kmax": 6, "spread": 1.0},
        # every class in bulk, integrals delivered in FP64
        {"name": "sweep_fp64", "kind": "sweep", "eris": 1 << 19, "precision": "fp64", "bits": 0},
        # the headline workload: every class in bulk, 16-bit codes
        {"name": "sweep_16bit", "kind": "sweep", "eris": 1 << 24, "precision": "mixed", "bits": 16},
        # a share of a contracted molecule's unique quartets as one CUDA-graph launch
        {"name": "molecule_graph_16bit", "kind": "molecule", "atoms": 40, "shards": 6000, "kmax": 6, "spread": 1.0, "bits": 16, "form": "graph"},
        # the same kind of job from the single work queue
        {"name": "molecule_queue_16bit", "kind": "molecule", "atoms": 40, "shards": 12000, "kmax": 6, "spread": 1.0, "bits": 16, "form": "queue"},
        # forces and exponent gradients with FP32 parameters
        {"name": "gradient_mixed", "kind": "gradient", "quartets": 1024, "K": 3, "precision": "mixed"},
        # the same in FP64
        {"name": "gradient_fp64", "kind": "gradient", "quartets": 384, "K": 3, "precision": "fp64"},
        # the classes beyond f
        {"name": "gshell_16bit", "kind": "gshell", "eris": 1 << 20, "precision": "mixed", "bits": 16},
        # one SCF iteration over stored ERIs
        {"name": "fock_16bit", "kind": "fock", "atoms": 12, "spread": 1.0, "symmetric": True},
        # the chunked layout of a stored stream
        {"name": "chunks_ffff_12bit", "kind": "chunks", "quartets": 40000, "cls": "ffff", "bits": 12},
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["class", "class", "sweep", "step", "molecule", "gradient", "gshell", "fock", "chunks"])
    spread = round(rng.uniform(0.9, 1.6), 3)
    if kind == "class":
        c = "".join(rng.choice("spdf") for _ in range(4))
        fp64 = rng.random() < 0.4
        n = max(1, min(2_000_000, span(1 << 16, 1 << (23 if fp64 else 25)) // size(tuple("spdf".index(x) for x in c))))
        pool = 0 if n <= 10000 and rng.random() < 0.5 else 2048
        return {"kind": kind, "cls": c, "quartets": n, "pool": pool, "precision": "fp64" if fp64 else "mixed",
                "bits": 0 if fp64 else rng.choice([8, 12, 16, 20])}
    if kind == "sweep":
        fp64 = rng.random() < 0.4
        return {"kind": kind, "eris": span(1 << 14, 1 << (19 if fp64 else 23)), "precision": "fp64" if fp64 else "mixed",
                "bits": 0 if fp64 else rng.choice([8, 12, 16, 20])}
    if kind == "step":
        return {"kind": kind, "atoms": rng.choice([1, 2, 2]), "kmax": rng.randint(1, 6), "spread": spread}
    if kind == "molecule":
        return {"kind": kind, "atoms": rng.randint(20, 40), "shards": span(6000, 60000), "kmax": rng.randint(1, 6),
                "spread": spread, "bits": 16, "form": rng.choice(["graph", "queue", "classes"])}
    if kind == "gradient":
        fp64 = rng.random() < 0.5
        K = rng.randint(1, 3)
        return {"kind": kind, "quartets": span(32, (384 if fp64 else 1024) * (81 // K ** 4 if K < 3 else 1) // 4),
                "K": K, "precision": "fp64" if fp64 else "mixed"}
    if kind == "gshell":
        return {"kind": kind, "eris": span(1 << 15, 1 << 20), "precision": rng.choice(["fp64", "mixed"]),
                "bits": rng.choice([12, 16, 20])}
    if kind == "fock":
        return {"kind": kind, "atoms": rng.randint(3, 12), "spread": spread, "symmetric": rng.random() < 0.5}
    c = "".join(rng.choice("spdf") for _ in range(4))
    n = max(1, span(1 << 20, 1 << 28) // size(tuple("spdf".index(x) for x in c)))
    return {"kind": kind, "quartets": min(n, 16_000_000), "cls": c, "bits": rng.choice([7, 8, 12, 16, 20])}


# --------------------------------------------------------------------------------------------
# inputs: shells (centres, L, primitives), quartet lists


def classes_of(case):
    k = case["kind"]
    if k in ("class", "chunks"):
        return [tuple("spdf".index(x) for x in case["cls"])]
    if k == "sweep":
        return all_classes((0, 1, 2, 3))
    if k == "gshell":
        return [c for c in all_classes((0, 1, 2, 3, 4)) if 4 in c]
    return all_classes((1, 2))  # gradient


def shellset(centers, L, exps, coefs, nprim):
    nprim = np.asarray(nprim, dtype=np.int32)
    pofs = np.zeros(len(nprim), dtype=np.int64)
    pofs[1:] = np.cumsum(nprim)[:-1]
    return ShellSet(np.ascontiguousarray(centers, dtype=np.float64), np.asarray(L, dtype=np.int32), nprim, pofs,
                    np.ascontiguousarray(exps, dtype=np.float64), np.ascontiguousarray(coefs, dtype=np.float64))


def primitive_pool(rng, L, n):
    """n shells for each entry of L: centres uniform in [-3, 3]^3 bohr, exponents log-uniform in
    [0.1, 10], unit coefficients."""
    m = n * len(L)
    return shellset(rng.uniform(-3, 3, (m, 3)), np.repeat(L, n), np.exp(rng.uniform(np.log(0.1), np.log(10), m)),
                    np.ones(m), np.ones(m))


def contracted_pool(rng, L, n, K):
    m = n * len(L)
    a0 = np.exp(rng.uniform(np.log(0.05), np.log(50.0 / 3.0 ** (K - 1)), m))
    return shellset(rng.uniform(-3, 3, (m, 3)), np.repeat(L, n), (a0[:, None] * 3.0 ** np.arange(K)).ravel(),
                    rng.uniform(0.1, 1.0, m * K), np.full(m, K))


def molecule(rng, atoms, kmax, spread):
    """Atoms at least 1.8 bohr apart in a cubic box (spread 1: the density of 200 in 20 bohr), each
    with s, s, p, p, d and f shells of 1 to kmax even-tempered primitives between 0.05 and 50.  The
    number of primitives of each shell belongs to the basis and is the same for every seed."""
    degree = np.random.default_rng(17)
    box = 20.0 * spread * (atoms / 200.0) ** (1 / 3)
    at = []
    while len(at) < atoms:
        p = rng.uniform(0, box, 3)
        if all(np.linalg.norm(p - x) >= 1.8 for x in at):
            at.append(p)
    centers, L, exps, coefs, nprim = [], [], [], [], []
    for p in at:
        for l in (0, 0, 1, 1, 2, 3):
            K = int(degree.integers(1, kmax + 1))
            a0 = np.exp(rng.uniform(np.log(0.05), np.log(50.0 / 3.0 ** (K - 1))))
            centers.append(p)
            L.append(l)
            nprim.append(K)
            exps += list(a0 * 3.0 ** np.arange(K))
            coefs += list(rng.uniform(0.1, 1.0, K))
    return shellset(np.array(centers), L, exps, coefs, nprim)


def unique_quartets(n):
    """One quartet (i >= j | k >= l), ij >= kl, of each set of eight equal ones."""
    i, j = np.tril_indices(n)
    p, q = np.tril_indices(len(i))
    return np.stack([i[p], j[p], i[q], j[q]], axis=1).astype(np.int32)


def shard_quartets(n, shards):
    """Positions 0, shards, 2 shards, ... of the enumeration of unique quartets of n shells: pairs
    (i >= j) by i, then j; quartets by bra pair, then ket pair (not before the bra)."""
    i, j = np.tril_indices(n)
    P = len(i)
    t = np.arange(0, P * (P + 1) // 2, shards, dtype=np.int64)
    starts = np.concatenate([[0], np.cumsum(np.arange(P, 0, -1, dtype=np.int64))])
    r = np.searchsorted(starts, t, side="right") - 1
    s = r + t - starts[r]
    return np.stack([i[r], j[r], i[s], j[s]], axis=1).astype(np.int32)


def pool_of(case, seed):
    """(shells, angular momenta of the pool, shells per angular momentum) of a random pool."""
    rng = np.random.default_rng([seed, 1])
    if case["kind"] == "sweep":
        return primitive_pool(rng, (0, 1, 2, 3), POOL), (0, 1, 2, 3), POOL
    if case["kind"] == "gshell":
        return primitive_pool(rng, (0, 1, 2, 3, 4), GPOOL), (0, 1, 2, 3, 4), GPOOL
    if case["kind"] == "gradient":
        return contracted_pool(rng, (1, 2), GPOOL, case["K"]), (1, 2), GPOOL
    L = tuple(sorted(set(classes_of(case)[0])))
    return primitive_pool(rng, L, case["pool"]), L, case["pool"]


def counts_of(case):
    per = [max(1, round(case["eris"] / size(c))) if "eris" in case else case["quartets"] for c in classes_of(case)]
    return per


def pool_quartets(case, seed, Ls, n, device):
    """Random quartets of each class over the pool, class after class, [total, 4] int32."""
    g = torch.Generator(device=device).manual_seed(seed * 7919 + 3)
    parts = []
    for c, m in zip(classes_of(case), counts_of(case)):
        base = torch.tensor([Ls.index(x) * n for x in c], dtype=torch.int32, device=device)
        parts.append(torch.randint(0, n, (m, 4), generator=g, device=device, dtype=torch.int32) + base)
    return torch.cat(parts)


def inputs(case, seed, device):
    """(shells, quartets) of every kind with an explicit list."""
    if case["kind"] in ("step", "fock", "molecule"):
        s = molecule(np.random.default_rng([seed, 2]), case["atoms"], case.get("kmax", 1), case["spread"])
        return s, shard_quartets(s.n, case["shards"]) if "shards" in case else unique_quartets(s.n)
    if case["kind"] == "class" and case["pool"] == 0:
        m = 4 * case["quartets"]
        s = primitive_pool(np.random.default_rng([seed, 1]), np.zeros(m, dtype=np.int32), 1)
        s.L[:] = np.tile(classes_of(case)[0], case["quartets"])
        return s, np.arange(m, dtype=np.int32).reshape(-1, 4)
    s, Ls, n = pool_of(case, seed)
    return s, pool_quartets(case, seed, Ls, n, device)


# --------------------------------------------------------------------------------------------
# preparation and the timed call


def coded_outputs(plan, bits):
    nb, ns = api.eri_output_bytes(plan, bits)
    return (torch.zeros(nb // 4, dtype=torch.int32, device="cuda"),
            torch.zeros(ns // 4, dtype=torch.float32, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "chunks":
        c = classes_of(case)[0]
        words = (case["quartets"] * size(c) * case["bits"] + 31) // 32
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["dense"] = torch.randint(-2**31, 2**31 - 1, (words,), generator=g, device="cuda", dtype=torch.int32)
        fields = 512 // case["bits"]
        st["chunks"] = torch.zeros(case["quartets"] * -(-size(c) // fields) * 16, dtype=torch.int32, device="cuda")
        return st
    if kind == "molecule":
        s = molecule(np.random.default_rng([seed, 2]), case["atoms"], case["kmax"], case["spread"])
        st["plan"] = api.eri_plan_create(s, None, precision="mixed", mode="unique8", shard=(0, case["shards"]))
        st["packed"], st["scales"] = coded_outputs(st["plan"], case["bits"])
        return st
    s, q = inputs(case, seed, "cuda")
    if kind == "gradient":
        st["geo"] = EriGeometry(s, q, precision=case["precision"])
        # mixed arithmetic goes with FP32 parameters, FP64 with FP64 ones
        dt = torch.float32 if case["precision"] == "mixed" else torch.float64
        st["centers"] = torch.tensor(s.centers, dtype=dt, requires_grad=True)
        st["exps"] = torch.tensor(s.exps, dtype=dt, requires_grad=True)
        st["G"] = upstream(case, seed, st["geo"].n_out)
        return st
    precision = case.get("precision", "fp64" if kind == "step" else "mixed")
    st["plan"] = api.eri_plan_create(s, q, precision=precision)
    if kind == "step":
        st["shells"] = s
    bits = case.get("bits", 16 if kind == "fock" else 0)
    if bits:
        if kind == "sweep":
            api.eri_plan_calibrate_precision(st["plan"], bits, sample=4096)
        st["packed"], st["scales"] = coded_outputs(st["plan"], bits)
    else:
        st["out"] = torch.zeros(api.eri_output_bytes(st["plan"], 0)[0] // 8, dtype=torch.float64, device="cuda")
    if kind == "fock":
        api.eri_compute_compressed(st["plan"], 16, st["packed"], st["scales"], torch.cuda.current_stream())
        st["D"] = density(case, seed, api.eri_plan_num_basis_functions(st["plan"]))
        st["J"], st["K"] = torch.zeros_like(st["D"]), torch.zeros_like(st["D"])
    return st


def upstream(case, seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def density(case, seed, n):
    D = torch.from_numpy(np.random.default_rng([seed, 6]).normal(0, 0.3, (n, n))).cuda()
    return (0.5 * (D + D.T)).contiguous() if case["symmetric"] else D


def run(st):
    case, s = st["case"], torch.cuda.current_stream()
    kind = case["kind"]
    if kind == "chunks":
        api.eri_pack_paper512_stream(st["dense"], case["quartets"], size(classes_of(case)[0]), case["bits"], st["chunks"], s)
        return st["chunks"]
    if kind == "gradient":
        eris = st["geo"](st["centers"], st["exps"])
        dR, da = torch.autograd.grad((eris * st["G"]).sum(), (st["centers"], st["exps"]))
        return {"eris": eris.detach(), "dR": dR, "dalpha": da}
    if kind == "fock":
        api.eri_digest_jk(st["plan"], 16, st["packed"], st["scales"], st["D"], st["J"], st["K"], unique8=True,
                          symmetric=case["symmetric"], stream=s)
        return {"J": st["J"], "K": st["K"]}
    if kind == "step":
        api.eri_plan_update_shells(st["plan"], st["shells"], s)
    if "out" in st:
        api.eri_compute(st["plan"], st["out"], s)
        return st["out"]
    form = {"graph": api.eri_compute_compressed_batched, "queue": api.eri_compute_compressed_queue}.get(
        case.get("form"), api.eri_compute_compressed)
    form(st["plan"], case["bits"], st["packed"], st["scales"], s)
    return {"codes": st["packed"], "scales": st["scales"]}


# --------------------------------------------------------------------------------------------
# unavoidable work


def flops_of(c, extra=0):
    """Flops of one primitive quartet: roots and B, C values, the 2-D integrals (5 per entry and
    axis), the quadrature (3 per root and output)."""
    n = (sum(c) + extra) // 2 + 1
    e = extra  # derivatives raise every index by one more
    tab = (c[0] + 1 + e) * (c[1] + 1 + e) * (c[2] + 1 + e) * (c[3] + 1 + e)
    return 40 + 80 * n + 15 * n * tab + 3 * n * size(c)


def mean_class(kmax):
    """Mean over the unique quartets of a molecule: (flops of a primitive quartet, ERIs, primitive
    quartets)."""
    Ls = (0, 0, 1, 1, 2, 3)
    f = sum(flops_of((a, b, c, d)) for a in Ls for b in Ls for c in Ls for d in Ls) / len(Ls) ** 4
    return f, (sum(ncart(l) for l in Ls) / 6) ** 4, ((kmax + 1) / 2) ** 4


def work(case):
    kind = case["kind"]
    if kind == "chunks":
        c = classes_of(case)[0]
        b = case["quartets"] * (size(c) * case["bits"] / 8 + 64 * -(-size(c) // (512 // case["bits"])))
        return {"bytes": b, "flops": 0}
    if kind in ("step", "fock", "molecule"):
        n = 6 * case["atoms"]
        p = n * (n + 1) // 2
        nq = p * (p + 1) // 2
        f, e, prims = mean_class(case.get("kmax", 1))
        if kind == "molecule":
            nq /= case["shards"]
        if kind == "fock":
            return {"bytes": nq * (20 + 2 * e), "flops": nq * 26 * e}
        return {"bytes": nq * (16 + (8 if kind == "step" else 2) * e), "flops": nq * prims * f}
    K4 = case.get("K", 1) ** 4
    by = fl = 0.0
    for c, m in zip(classes_of(case), counts_of(case)):
        out = size(c) * (case["bits"] / 8 if case.get("bits") else 8)
        by += m * (16 + out)
        fl += m * K4 * flops_of(c)
        if kind == "gradient":
            by += m * out
            fl += m * K4 * (flops_of(c, 1) + 12 * size(c))
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------------------------
# the same results in 64 bits, from the definition: 1/r12 as a Gaussian transform, its parameter
# integrated by a 64-point Gauss-Legendre rule, the integrand a product of three one-dimensional
# integrals raised by the Gaussian recursions

X64, W64 = np.polynomial.legendre.leggauss(64)
CART = {L: [(x, y, L - x - y) for x in range(L, -1, -1) for y in range(L - x, -1, -1)] for L in range(5)}


def norm(a, L):
    df = math.prod(range(2 * L - 1, 0, -2)) if L > 0 else 1
    return (2 * a / math.pi) ** 0.75 * (4 * a) ** (L / 2) / math.sqrt(df)


def primitive_eris(c, R, a, cf):
    """[n, n_eri] ERIs of primitive quartets of class c: R four [n, 3] centres, a four [n]
    exponents, cf [n] products of coefficients and normalisations."""
    A, B, C, D = R
    p, q = a[0] + a[1], a[2] + a[3]
    AB, CD = A - B, C - D
    PA = -(a[1] / p)[:, None] * AB
    QC = -(a[3] / q)[:, None] * CD
    PQ = (A + PA) - (C + QC)
    rho = p * q / (p + q)
    T = rho * PQ.square().sum(1)
    cut = (100.0 / T.detach().clamp(min=1e-300)).sqrt().clamp(max=1.0)
    x, w = (torch.tensor(v, dtype=torch.float64, device=T.device) for v in (X64, W64))
    t2 = (0.5 * cut[:, None] * (x + 1)) ** 2
    pref = 2 * math.pi ** 2.5 / (p * q * (p + q).sqrt()) * cf * torch.exp(
        -(a[0] * a[1] / p) * AB.square().sum(1) - (a[2] * a[3] / q) * CD.square().sum(1))
    wz = pref[:, None] * 0.5 * cut[:, None] * w * torch.exp(-T[:, None] * t2)
    b00 = 0.5 * t2 / (p + q)[:, None]
    b10 = (1 - t2 * (q / (p + q))[:, None]) / (2 * p)[:, None]
    b01 = (1 - t2 * (p / (p + q))[:, None]) / (2 * q)[:, None]
    La, Lb, Lc, Ld = c
    axis = []
    for s in range(3):
        u = t2 * (q / (p + q) * PQ[:, s])[:, None]
        v = t2 * (p / (p + q) * PQ[:, s])[:, None]
        cA, cB = PA[:, s, None] - u, (PA + AB)[:, s, None] - u
        cC, cD = QC[:, s, None] + v, (QC + CD)[:, s, None] + v
        t = {(0, 0, 0, 0): wz if s == 2 else torch.ones_like(wz)}
        for i in range(La + 1):
            for j in range(Lb + 1):
                for k in range(Lc + 1):
                    for l in range(Ld + 1):
                        if l:
                            o, z, low = (i, j, k, l - 1), cD, [(i, (i - 1, j, k, l - 1), b00), (j, (i, j - 1, k, l - 1), b00), (k, (i, j, k - 1, l - 1), b01), (l - 1, (i, j, k, l - 2), b01)]
                        elif k:
                            o, z, low = (i, j, k - 1, 0), cC, [(i, (i - 1, j, k - 1, 0), b00), (j, (i, j - 1, k - 1, 0), b00), (k - 1, (i, j, k - 2, 0), b01)]
                        elif j:
                            o, z, low = (i, j - 1, 0, 0), cB, [(i, (i - 1, j - 1, 0, 0), b10), (j - 1, (i, j - 2, 0, 0), b10)]
                        elif i:
                            o, z, low = (i - 1, 0, 0, 0), cA, [(i - 1, (i - 2, 0, 0, 0), b10)]
                        else:
                            continue
                        r = z * t[o]
                        for n, e, b in low:
                            if n:
                                r = r + n * b * t[e]
                        t[(i, j, k, l)] = r
        axis.append(torch.stack([t[(i, j, k, l)] for i in range(La + 1) for j in range(Lb + 1) for k in range(Lc + 1) for l in range(Ld + 1)]))
    rows = [[((ca[s] * (Lb + 1) + cb[s]) * (Lc + 1) + cc[s]) * (Ld + 1) + cd[s] for ca in CART[La] for cb in CART[Lb]
             for cc in CART[Lc] for cd in CART[Ld]] for s in range(3)]
    rows = torch.tensor(rows, device=T.device)
    out = []
    for e in range(0, rows.shape[1], 1296):
        r = rows[:, e:e + 1296]
        out.append((axis[0][r[0]] * axis[1][r[1]] * axis[2][r[2]]).sum(-1))
    return torch.cat(out).T


def class_lists(s, q):
    """(class, rows of q of that class in the list's order) by ascending class id."""
    L = np.asarray(s.L)
    ls = torch.from_numpy(L.astype(np.int64)).to(q.device)[q.long()]
    g = (ls > 3).any(1)
    w4, w5 = (torch.tensor([b ** 3, b ** 2, b, 1], device=q.device) for b in (4, 5))
    ids = torch.where(g, 256 + (ls * w5).sum(1), (ls * w4).sum(1))
    for i in torch.unique(ids).tolist():
        c = (i >> 6, i >> 4 & 3, i >> 2 & 3, i & 3) if i < 256 else ((i - 256) // 125, (i - 256) // 25 % 5, (i - 256) // 5 % 5, (i - 256) % 5)
        yield c, q[ids == i]


def blocks(s, c, q, centers, exps, budget=3e8):
    """Chunks of quartets of one class: (first, last, a function giving their ERIs)."""
    dev = q.device
    nprim = torch.from_numpy(s.nprim.astype(np.int64)).to(dev)[q.long()]
    pofs = torch.from_numpy(s.pofs).to(dev)[q.long()]
    coefs = torch.from_numpy(s.coefs).to(dev)
    per = nprim.prod(1)
    tab = (c[0] + 1) * (c[1] + 1) * (c[2] + 1) * (c[3] + 1)
    ends = per.cumsum(0).cpu().numpy()
    room = max(1, int(budget / (64 * (3 * min(size(c), 1296) + 3 * tab))))
    first = 0
    while first < len(q):
        done = ends[first - 1] if first else 0
        last = max(first + 1, int(np.searchsorted(ends, done + room, side="right")))

        def eris(first=first, last=last):
            m = per[first:last]
            own = torch.repeat_interleave(torch.arange(last - first, device=dev), m)
            r = torch.arange(int(m.sum()), device=dev) - (m.cumsum(0) - m)[own]
            at = []
            for k in (3, 2, 1, 0):
                n = nprim[first:last, k][own]
                at.insert(0, pofs[first:last, k][own] + r % n)
                r = r // n
            ids = q[first:last].long()[own]
            R = [centers[ids[:, k]] for k in range(4)]
            a = [exps[at[k]] for k in range(4)]
            cf = math.prod(coefs[at[k]] * norm(a[k], c[k]) for k in range(4))
            v = primitive_eris(c, R, a, cf)
            return torch.zeros((last - first, v.shape[1]), dtype=v.dtype, device=dev).index_add(0, own, v)

        yield first, last, eris
        first = last


def exact(case, seed):
    kind = case["kind"]
    if kind == "chunks":  # bytes
        return None
    # left out where a plain evaluation would take too long
    if kind == "sweep" and case["eris"] > 1 << 21 or kind == "fock" and case["atoms"] > 6:
        return None
    if kind == "molecule" and work(case)["flops"] > 3e10:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    s, q = inputs(case, seed, dev)
    q = torch.as_tensor(q, device=dev)
    dt = torch.float32 if kind == "gradient" and case["precision"] == "mixed" else torch.float64
    centers, exps = (torch.tensor(v, dtype=dt, device=dev).double() for v in (s.centers, s.exps))
    if kind == "gradient":
        G = upstream(case, seed, sum(m * size(c) for c, m in zip(classes_of(case), counts_of(case))))
        grads = [torch.zeros_like(centers), torch.zeros_like(exps)]
        parts, pos = [], 0
        for c, qc in class_lists(s, q):
            for first, last, eris in blocks(s, c, qc, centers.requires_grad_(), exps.requires_grad_(), 2e8):
                v = eris().reshape(-1)
                for g, d in zip(grads, torch.autograd.grad((v * G[pos:pos + len(v)]).sum(), (centers, exps))):
                    g += d
                parts.append(v.detach())
                pos += len(v)
        return {"eris": torch.cat(parts), "dR": grads[0], "dalpha": grads[1]}
    parts, bits = [], case.get("bits", 0)
    full = fock_tensor(s, dev) if kind == "fock" else None
    for c, qc in class_lists(s, q):
        for first, last, eris in blocks(s, c, qc, centers, exps):
            v = eris()
            if kind == "fock":
                full["add"](c, qc[first:last].long(), v)
            else:
                parts.append(v.abs().amax(1) / (2 ** (bits - 1) - 1) if bits else v.reshape(-1))
    if kind == "fock":
        D = density(case, seed, full["n"]).to(dev)
        E = full["E"]
        return {"J": torch.einsum("mnls,ls->mn", E, D), "K": torch.einsum("mnls,ns->ml", E, D)}
    return {"codes": None, "scales": torch.cat(parts)} if bits else torch.cat(parts)


def fock_tensor(s, dev):
    """All ERIs of a small basis, filled from unique quartets through the eight permutations."""
    sizes = [ncart(int(l)) for l in s.L]
    first = torch.tensor(np.concatenate([[0], np.cumsum(sizes)[:-1]]), device=dev)
    n = sum(sizes)
    E = torch.zeros((n, n, n, n), dtype=torch.float64, device=dev)

    def add(c, q, v):
        d = [ncart(l) for l in c]
        v = v.reshape(-1, *d)
        o = [first[q[:, k]][:, None, None, None, None] + torch.arange(d[k], device=dev).reshape([-1 if x == k + 1 else 1 for x in range(5)])
             for k in range(4)]
        for x in ((0, 1, 2, 3), (1, 0, 2, 3), (0, 1, 3, 2), (1, 0, 3, 2), (2, 3, 0, 1), (3, 2, 0, 1), (2, 3, 1, 0), (3, 2, 1, 0)):
            E[o[x[0]], o[x[1]], o[x[2]], o[x[3]]] = v

    return {"E": E, "add": add, "n": n}

"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one pass through a public entry point: one evaluation of an FMM or treecode on
particles in device memory or in host memory, one direct sum, or one replay of a batch of uneven
instances.  Outputs are the potential and its gradient at every particle.  Particles follow the
two distributions this repository works with: a uniform cube with charges U[0, 1)/n, and a
Plummer sphere (a = 1, truncated at r = 20) of equal masses 1/n.
"""
from __future__ import annotations

import math

import torch

from paper_1010_1482_gb300 import gbfmm as G
from paper_1010_1482_gb300 import inputs

ORDERS = (4, 6, 8, 10)
LEAVES = (32, 64, 128)

# particle counts drawn for each kind of case (log-uniform, both ends included)
RANGES = {
    "fmm_uniform": (1_000, 5_000_000),
    "fmm_adaptive": (1_000, 5_000_000),
    "host": (1_000, 1_000_000),
    "treecode_uniform": (1_000, 250_000),
    "treecode_adaptive": (1_000, 100_000),
    "direct": (500, 40_000),
}


def listed():
    return [
        # the smallest configuration: one evaluation of a small system, launches and latency
        dict(name="uniform_4k_p4", kind="fmm_uniform", n=4096, p=4, leaf=64, eps2=0.0),
        # an ordinary ragged system with Plummer softening, a depth-4 tree of ~24 per leaf
        dict(name="uniform_100k_p8_soft", kind="fmm_uniform", n=100_003, p=8, leaf=64, eps2=1e-8),
        # the headline configuration: a million particles at the highest order
        dict(name="uniform_1m_p10", kind="fmm_uniform", n=1 << 20, p=10, leaf=64, eps2=0.0),
        # a large uniform system whose count falls between two depths (19 per leaf)
        dict(name="uniform_5m_p6", kind="fmm_uniform", n=5_000_000, p=6, leaf=64, eps2=0.0),
        # one evaluation through host buffers, copies both ways included (a served request)
        dict(name="host_300k_p8", kind="host", n=300_007, p=8, leaf=64, eps2=0.0),
        # a small clustered system on the adaptive tree: the latency of the whole chain
        dict(name="plummer_20k_p4", kind="fmm_adaptive", n=20_011, p=4, leaf=64, eps2=0.0),
        # an ordinary clustered system at the highest order
        dict(name="plummer_400k_p10", kind="fmm_adaptive", n=400_009, p=10, leaf=64, eps2=0.0),
        # the largest configuration: 16M clustered particles
        dict(name="plummer_16m_p8", kind="fmm_adaptive", n=1 << 24, p=8, leaf=64, eps2=0.0),
        # the paper's treecode on the uniform tree, at the order that meets 1e-4
        dict(name="treecode_uniform_130k_p6", kind="treecode_uniform", n=131_072, p=6, leaf=64, eps2=0.0),
        # the treecode on a clustered set
        dict(name="treecode_plummer_50k_p8", kind="treecode_adaptive", n=50_021, p=8, leaf=64, eps2=0.0),
        # many independent uneven systems at once, both trees, two orders
        dict(name="batch_96", kind="batch", count=96, n_lo=1_000, n_hi=200_000, leaf=64),
        # the all-pairs sum, the fastest method for small systems and the check of the others
        dict(name="direct_16k_soft", kind="direct", n=16_411, eps2=1e-4),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fmm_uniform"] * 4 + ["fmm_adaptive"] * 4 + ["host"] * 2 +
                      ["treecode_uniform", "treecode_adaptive", "direct", "batch"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(24, 96), n_lo=1_000, n_hi=_between(rng, 20_000, 200_000),
                    leaf=rng.choice((64, 128)))
    n = _between(rng, *RANGES[kind])
    if kind == "direct":
        return dict(kind=kind, n=n, eps2=rng.choice((0.0, 1e-4)))
    return dict(kind=kind, n=n, p=rng.choice(ORDERS), leaf=rng.choice(LEAVES), eps2=rng.choice((0.0, 0.0, 1e-8)))


# ---- inputs --------------------------------------------------------------------------------

def _uniform(n, gen):
    x = torch.rand((n, 4), generator=gen, device="cuda", dtype=torch.float32)
    x[:, 3] /= n
    return x


def _plummer(n, gen, rmax=inputs.PLUMMER_RMAX):
    u = torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float64)
    mmax = rmax ** 3 / (1.0 + rmax * rmax) ** 1.5
    r = 1.0 / torch.sqrt(((1.0 - u[:, 0]) * mmax) ** (-2.0 / 3.0) - 1.0)
    ct = 2.0 * u[:, 1] - 1.0
    st = torch.sqrt((1.0 - ct * ct).clamp_min(0.0))
    ph = 2.0 * math.pi * u[:, 2]
    x = torch.empty((n, 4), device="cuda", dtype=torch.float32)
    x[:, 0] = r * st * torch.cos(ph)
    x[:, 1] = r * st * torch.sin(ph)
    x[:, 2] = r * ct
    x[:, 3] = 1.0 / n
    return x


def _instances(case):
    """Sizes, distributions and orders of a batch's instances (the particles follow the seed)."""
    return inputs.batch_instances(case["count"], n_lo=case["n_lo"], n_hi=case["n_hi"])


def _particles(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "batch":
        return torch.cat([(_uniform if i["dist"] == "uniform" else _plummer)(i["n"], gen) for i in _instances(case)])
    return (_plummer if kind.endswith("adaptive") else _uniform)(case["n"], gen)


# ---- handles -------------------------------------------------------------------------------

_kept = None  # (parameters, handle): a program keeps its handle from one set of particles to the next


def _handle(**params):
    global _kept
    key = tuple(sorted(params.items()))
    if _kept is None or _kept[0] != key:
        _kept = (key, G.FMM(0, **params))
    return _kept[1]


class _Batch:
    def __init__(self, fmm, offsets, params, x, out):
        self.fmm, self.x, self.out = fmm, x, out
        self.batch = G.gbfmm_batch_create(fmm.ctx, offsets, params, x, out, lanes=64)

    def __del__(self):
        if getattr(self, "batch", None):
            G.gbfmm_batch_destroy(self.batch)


def prepare(case, seed):
    x = _particles(case, seed)
    kind = case["kind"]
    if kind == "batch":
        fmm = _handle()
        inst = _instances(case)
        offsets = [0]
        for i in inst:
            offsets.append(offsets[-1] + i["n"])
        params = [G.gbfmm_default_params(p=i["p"], leaf_size=case["leaf"],
                                         tree=G.TREE_UNIFORM if i["dist"] == "uniform" else G.TREE_ADAPTIVE)
                  for i in inst]
        out = torch.empty_like(x)
        return dict(kind=kind, batch=_Batch(fmm, offsets, params, x, out), out=out)
    if kind == "direct":
        return dict(kind=kind, fmm=_handle(), x=x, out=torch.empty_like(x), eps2=case["eps2"])
    fmm = _handle(p=case["p"], leaf_size=case["leaf"], eps2=case["eps2"],
                  tree=G.TREE_ADAPTIVE if kind.endswith("adaptive") else G.TREE_UNIFORM,
                  method=G.METHOD_TREECODE if kind.startswith("treecode") else G.METHOD_FMM)
    if kind == "host":
        h = x.cpu().pin_memory()
        return dict(kind=kind, fmm=fmm, x=h, out=torch.empty_like(h).pin_memory())
    return dict(kind=kind, fmm=fmm, x=x, out=torch.empty_like(x))


def run(state):
    kind, out = state["kind"], state["out"]
    if kind == "batch":
        G.gbfmm_batch_launch(state["batch"].fmm.ctx, state["batch"].batch)
    elif kind == "direct":
        G.gbfmm_direct(state["fmm"].ctx, state["x"], state["x"], out, state["eps2"])
    elif kind == "host":
        G.gbfmm_evaluate_host(state["fmm"].ctx, state["fmm"].params, state["x"], out)
    else:
        state["fmm"].evaluate(state["x"], out, check=False)
    return out


# ---- work ----------------------------------------------------------------------------------

PAIR = 20  # operations of one particle pair (Listing 1's 19 and the potential's sum)


def _uniform_counts(n, leaf):
    """Depth, particle pairs of the 27-neighbour sums, and M2L pairs per level of a filled tree."""
    depth = 0
    while n > leaf * 8 ** depth:
        depth += 1
    side = 2 ** depth
    near = (3 * side - 2) ** 3 * (n / side ** 3) ** 2 if depth else float(n) * n
    far = {l: (6 * 2 ** l - 8) ** 3 - (3 * 2 ** l - 2) ** 3 for l in range(2, depth + 1)}
    return depth, min(near, float(n) * n), far


def _flops(tree, method, n, p, leaf):
    ends = 20 * p * (p + 1) * n  # P2M and L2P
    if tree == "uniform":
        depth, near, far = _uniform_counts(n, leaf)
        if method == "treecode":
            return PAIR * near + sum(c * n / 8 ** l for l, c in far.items()) * 8 * p * p + ends / 4
        cells = sum(8 ** l for l in range(3, depth + 1))
        return PAIR * near + 2 * p ** 4 * (sum(far.values()) + 2 * cells) + (ends if depth >= 2 else 0)
    # Plummer spheres on the adaptive tree: about 10 leaves' worth of near particles each, 0.75
    # cells a particle at leaf size 12, and 170 M2L pairs a cell (rates of the 16M set)
    near, cells = 10.3 * leaf * float(n), 4.0 * n / leaf
    if method == "treecode":
        return PAIR * min(near, float(n) * n) + 170 * math.log(max(n / leaf, 8), 8) * n * 8 * p * p + ends / 4
    return PAIR * min(near, float(n) * n) + 2 * p ** 4 * (170 + 2) * cells + ends


def work(case):
    kind = case["kind"]
    if kind == "batch":
        inst = _instances(case)
        return dict(bytes=32 * sum(i["n"] for i in inst),
                    flops=sum(_flops("uniform" if i["dist"] == "uniform" else "adaptive", "fmm", i["n"], i["p"],
                                     case["leaf"]) for i in inst))
    n = case["n"]
    if kind == "direct":
        return dict(bytes=32 * n, flops=PAIR * float(n) * n)
    return dict(bytes=32 * n, flops=_flops("adaptive" if kind.endswith("adaptive") else "uniform",
                                           "treecode" if kind.startswith("treecode") else "fmm", n, case["p"],
                                           case["leaf"]))


# ---- correctness ---------------------------------------------------------------------------

def tolerance(case):
    # The all-pairs sum: up to 40,000 terms in 32 bits, 2.2e-6 (largest 9.5e-6) between two orders
    # of 16,411 sources.  FMM and treecode: the same with the particles in another order 2.4e-7
    # (largest 3.7e-6), and with the M2L's products formed on the FP32 cores instead 8.3e-7 (4.1e-6).
    if case["kind"] == "direct":
        return dict(rel=1.5e-5, max=1e-4)
    return dict(rel=4e-6, max=2e-5)


def _direct64(x, eps2):
    """Potential and gradient of every particle in 64 bits, all pairs."""
    n = x.shape[0]
    x = x.double()
    pos, q = x[:, :3].t().contiguous(), x[:, 3]
    out = torch.empty((n, 4), device="cuda", dtype=torch.float64)
    rows = max(1, min(n, 200_000_000 // n))
    for a in range(0, n, rows):
        b = min(n, a + rows)
        d = [pos[k][None, :] - pos[k][a:b, None] for k in range(3)]
        d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        zero = d2 == 0
        inv = torch.rsqrt(d2 + eps2)
        inv[zero] = 0.0
        w = inv * q
        out[a:b, 0] = w.sum(1)
        w *= inv
        w *= inv
        for k in range(3):
            d[k] *= w
            out[a:b, 1 + k] = d[k].sum(1)
    return out


def exact(case, seed):
    """The all-pairs sum: an evaluation differs from it by its order's truncation as well."""
    kind = case["kind"]
    if kind == "batch":
        inst = _instances(case)
        if sum(float(i["n"]) ** 2 for i in inst) > 1e11:
            return None
        x, out, at = _particles(case, seed), [], 0
        for i in inst:
            out.append(_direct64(x[at:at + i["n"]], 0.0))
            at += i["n"]
        return torch.cat(out)
    if float(case["n"]) ** 2 > 1e11:
        return None
    out = _direct64(_particles(case, seed), case["eps2"])
    return out.cpu() if kind == "host" else out

"""Performance cases of the density / entropy / training paths.

A case is a dict of plain values; ``prepare`` builds what a program has in hand
before the call (H on the GPU, the model set, the planned ``Solver``) and ``run``
is one pass through the public API.  The Hamiltonians are those of
``workloads/`` drawn with the GPU's generator: open cubic tight-binding
lattices and chains with dense noise, optionally long-range couplings, and
dense rotated spectra.  ``exact`` evaluates the definitions (Fermi function and
entropy of the eigenvalues) in FP64.
"""
from __future__ import annotations

import json
import math
import os

import numpy as np
import torch

import paper_2605_08523_gb300 as ft

TABLES = os.path.join(os.path.dirname(os.path.abspath(ft.__file__)), "tables")
MU0 = 1.0 / 3.0

# model sets by use: the printed table alone; the printed table with its
# trained entropy table and the 24-layer beta0 = 1000 one (lattices at
# kT >= 0.1); the printed, beta0 = 2250 and 3000 tables (wide Gershgorin
# intervals); the set of the ragged batches; the Max-SP2 table
SETS = {
    "printed": None,
    "lattice": ("entropy_b1500_L26", "b1000_L24"),
    "longrange": ("entropy_b1500_L26", "b2250_L27", "b3000_L34"),
    "ragged": ("entropy_b1500_L26", "b100_L32", "b200_L32", "b20_L32", "b50_L32", "b12000_L40", "b24000_L44",
               "b3000_L34", "b6000_L37", "b100_L18", "b200_L21", "b400_L24"),
    "max": ("max_b100_L12",),
}
FLAGS = {"": 0, "lanczos": ft.LANCZOS, "lanczos,min_layers": ft.LANCZOS | ft.MIN_LAYERS,
         "refine2": ft.REFINE2, "refine2_tc": ft.REFINE2 | ft.REFINE_TC}


def _lattice(name, dims, mode, want, kT, tables, flags="", longrange=0.0, mu=0.0):
    return dict(name=name, kind="lattice", nx=dims[0], ny=dims[1], nz=dims[2], mode=mode, want=want, kT=kT, mu=mu,
                tables=tables, flags=flags, longrange=longrange)


def _ragged(name, batch, nmin, nmax, mode, want, flags):
    return dict(name=name, kind="ragged", batch=batch, nmin=nmin, nmax=nmax, mode=mode, want=want, tables="ragged",
                flags=flags)


def listed():
    return [
        # one small molecule or chain: D and S of a single n = 256 matrix, where launches and latency count
        _lattice("chain_256", (256, 1, 1), "fp16x2", 3, 0.1, "printed"),
        # an SCF step of a small system: mu for a prescribed electron count by Newton updates, then D and S
        dict(name="mu_512", kind="mu", nx=8, ny=8, nz=8, mode="fp16x2", want=3, kT=0.1, mu=0.15, tables="printed",
             flags="", longrange=0.0, iterations=3),
        # density matrix alone (forces, populations) of a mid-size lattice in the 24-bit split mode
        _lattice("lattice_1024_bf16x3", (8, 8, 16), "bf16x3", 1, 0.1, "lattice"),
        # entropy alone (free-energy differences) of a chain of an odd order
        _lattice("chain_1501_entropy", (1501, 1, 1), "fp16x2", 2, 0.3, "lattice"),
        # D and S at a low temperature in the TF32 split mode
        _lattice("lattice_2048_tf32x3", (8, 16, 16), "tf32x3", 3, 0.05, "longrange"),
        # the lattice of the benchmark's sweep: n = 4096, D and S
        _lattice("lattice_4096", (16, 16, 16), "fp16x2", 3, 0.1, "lattice"),
        # the largest single matrix: n = 8192 with long-range couplings, two BF16X3 refinement layers
        _lattice("longrange_8192", (16, 16, 32), "fp16x2", 3, 0.1, "longrange", "refine2_tc", 0.05),
        # the last two layers in FP32 on the CUDA cores, odd order
        _lattice("refine_fp32_2197", (13, 13, 13), "fp16x2", 3, 0.1, "lattice", "refine2"),
        # Max-SP2 in FP32 mode with Lanczos bounds (the comparison of the table families)
        _lattice("max_fp32_1728", (12, 12, 12), "fp32", 3, 0.3, "max", "lanczos"),
        # 512 dense Hamiltonians of an ensemble, n in [64, 768], one call: D and S
        _ragged("ragged_512", 512, 64, 768, "fp16x2", 3, "lanczos,min_layers"),
        # 60 fragments with n in [16, 200], density alone, Gershgorin bounds
        _ragged("fragments_60", 60, 16, 200, "fp16x2", 1, ""),
        # fitting a table of the model set: 100 Levenberg-Marquardt iterations on 1e5 samples
        dict(name="train_L16", kind="train", L=16, beta0=100.0, nsamples=100_000, iterations=100, target=0),
    ]


def _dims_near(rng, n):
    """Three lattice edges, odd ones among them, whose product is close to n."""
    a = max(1, round(n ** (1 / 3) * rng.uniform(0.6, 1.1)))
    b = max(1, round(math.sqrt(n / a) * rng.uniform(0.7, 1.2)))
    return a, b, max(1, round(n / (a * b)))


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "chain", "mu", "ragged", "fp32", "train"])
    lo_hi = {"lattice": (64, 5500), "chain": (33, 3000), "mu": (64, 1500), "fp32": (64, 1800)}
    if kind == "train":
        return dict(kind="train", L=rng.choice([12, 14, 16, 18, 20, 24]), beta0=rng.choice([50.0, 100.0, 200.0]),
                    nsamples=int(math.exp(rng.uniform(math.log(5e3), math.log(1e5)))), iterations=rng.randint(5, 40),
                    target=0)
    if kind == "ragged":
        batch = int(math.exp(rng.uniform(math.log(8), math.log(300))))
        nmin, nmax = rng.randint(16, 100), rng.randint(120, 768)
        flags = rng.choice(["lanczos,min_layers", "lanczos", ""])
        return _unnamed(_ragged("", batch, nmin, nmax, rng.choice(["fp16x2", "fp16x2", "bf16x3"]), rng.choice([1, 3]),
                                flags))
    lo, hi = lo_hi[kind]
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    dims = (n, 1, 1) if kind == "chain" else _dims_near(rng, n)
    kT = round(rng.uniform(0.1, 0.3), 3)
    if kind == "mu":
        return dict(kind="mu", nx=dims[0], ny=dims[1], nz=dims[2], mode="fp16x2", want=rng.choice([1, 3]), kT=kT,
                    mu=round(rng.uniform(-0.2, 0.2), 3), tables="lattice", flags="", longrange=0.0,
                    iterations=rng.randint(1, 4))
    if kind == "fp32":
        tables, flags = rng.choice([("max", "lanczos"), ("lattice", "")])
        kT = 0.3 if tables == "max" else kT
        return _unnamed(_lattice("", dims, "fp32", rng.choice([1, 2, 3]), kT, tables, flags))
    mode = rng.choice(["fp16x2", "fp16x2", "fp16x2", "bf16x3", "tf32x3"])
    flags = rng.choice(["", "", "refine2_tc", "lanczos", "refine2"])
    lr = rng.choice([0.0, 0.05]) if kind == "lattice" else 0.0
    return _unnamed(_lattice("", dims, mode, rng.choice([1, 2, 3, 3]), kT, "longrange" if lr else "lattice", flags,
                             lr, round(rng.uniform(-0.3, 0.3), 3)))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def _hamiltonian(case, seed):
    """Open nx x ny x nz lattice: on-site U(-1, 1), hopping -1, symmetrised 0.01 N(0, 1) noise, a fraction
    `longrange` of the pairs with N(0, 0.05) couplings."""
    g = _generator(seed)
    dims = (case["nx"], case["ny"], case["nz"])
    n = dims[0] * dims[1] * dims[2]
    f64 = dict(dtype=torch.float64, device="cuda")
    H = torch.randn(n, n, generator=g, **f64)
    H = (H + H.T) * 0.005
    H.diagonal().add_(torch.rand(n, generator=g, **f64) * 2.0 - 1.0)
    idx = torch.arange(n, device="cuda").reshape(dims)
    for ax in range(3):
        if dims[ax] > 1:
            a = idx.narrow(ax, 0, dims[ax] - 1).reshape(-1)
            b = idx.narrow(ax, 1, dims[ax] - 1).reshape(-1)
            H[a, b] -= 1.0
            H[b, a] -= 1.0
    if case["longrange"] > 0.0:
        C = torch.randn(n, n, generator=g, **f64) * 0.05
        C = torch.where(torch.rand(n, n, generator=g, device="cuda") < case["longrange"], C, 0.0).triu(1)
        H += C + C.T
    return H.contiguous()


def _rotation(n, g):
    """A dense orthogonal n x n matrix: two cosine transforms with random signs and a permutation between."""
    k = torch.arange(n, dtype=torch.float64, device="cuda")
    C = torch.cos(math.pi / n * (k[None, :] + 0.5) * k[:, None]) * math.sqrt(2.0 / n)
    C[0] *= math.sqrt(0.5)
    s = torch.randint(0, 2, (2, n), generator=g, device="cuda").double() * 2.0 - 1.0
    p = torch.randperm(n, generator=g, device="cuda")
    return (C * s[0])[:, p] @ (C * s[1])


def _spectra(case, seed):
    """Per instance (Q, eigenvalues, mu, kT): eigenvalues U(-10, 10) eV, mu U(-5, 5), kT U(0.02, 0.5)."""
    g = _generator(seed)
    r = np.random.default_rng(seed)
    # the orders belong to the case, the matrices to the seed
    ns = np.random.default_rng(case["batch"]).integers(case["nmin"], case["nmax"] + 1, case["batch"])
    out = []
    for n in ns.tolist():
        lam = torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * 20.0 - 10.0
        out.append((_rotation(n, g), lam, float(r.uniform(-5.0, 5.0)), float(r.uniform(0.02, 0.5))))
    return out


def _model_set(name):
    if SETS[name] is None:
        return ft.ModelSet()
    return ft.ModelSet.from_json([os.path.join(TABLES, t + ".json") for t in SETS[name]])


def prepare(case, seed):
    if case["kind"] == "train":
        return dict(case=case, seed=int(seed) + 1)
    if case["kind"] == "ragged":
        inst = _spectra(case, seed)
        H = torch.cat([((Q * lam) @ Q.T).add_(((Q * lam) @ Q.T).T).mul_(0.5).reshape(-1) for Q, lam, _, _ in inst])
        ns, mus, kTs = [Q.shape[0] for Q, _, _, _ in inst], [i[2] for i in inst], [i[3] for i in inst]
    else:
        H = _hamiltonian(case, seed)
        ns, mus, kTs = [H.shape[0]], [case["mu"]], [case["kT"]]
        H = H.reshape(-1)
    s = ft.Solver(ns, mus, kTs, _model_set(case["tables"]), mode=case["mode"], want=case["want"],
                  flags=FLAGS[case["flags"]])
    return dict(case=case, H=H, solver=s, mus=mus, kTs=kTs)


def _outputs(s):
    out = {}
    if s.want & 1:
        out.update(D=s.D, trace=s.trace)
    if s.want & 2:
        out["S"] = s.S
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        theta, report = ft.ftsp2_train_coeffs(case["target"], case["beta0"], MU0, case["L"],
                                              nsamples=case["nsamples"], seed=state["seed"],
                                              iterations=case["iterations"])
        return dict(theta=theta, max_err=report["max_err"])
    s = state["solver"]
    if case["kind"] == "mu":
        # the electron count is prescribed; mu starts from the previous step's value
        s.set_mu_kT(state["mus"], state["kTs"])
        steps = s.run_mu(state["H"], [s.ns[0] / 2.0], iterations=case["iterations"])
        return dict(_outputs(s), steps=steps, mu=s.mus())
    s.run(state["H"])
    return _outputs(s)


# ---------------------------------------------------------------------------
# work and exact results
# ---------------------------------------------------------------------------
def _layers(case):
    """(density, entropy) layers of the case's table: the smallest beta0 of a single system's set that a solve
    takes at these temperatures; ragged batches count their typical 21-layer table."""
    if case["kind"] == "ragged":
        return (21 if "min_layers" in case["flags"] else 34,) * 2
    name = {"lattice": "b1000_L24", "longrange": "b2250_L27", "max": "max_b100_L12"}.get(case["tables"],
                                                                                        "entropy_b1500_L26")
    with open(os.path.join(TABLES, name + ".json")) as f:
        L = json.load(f).get("L")
    return (L or int(name.split("_L")[1]),) * 2


def work(case):
    if case["kind"] == "train":
        # per evaluation the Jacobian's columns and the symmetric Gram matrix of 4L + 1 columns
        m, ns, evals = 4 * case["L"] + 1, case["nsamples"], case["iterations"] + 1
        return dict(bytes=8.0 * ns, flops=float(evals) * ns * (m * (m + 1) + 16.0 * case["L"]))
    if case["kind"] == "ragged":
        ns = np.random.default_rng(case["batch"]).integers(case["nmin"], case["nmax"] + 1, case["batch"]).tolist()
    else:
        ns = [case["nx"] * case["ny"] * case["nz"]]
    Ld, Le = _layers(case)
    n2, n3 = float(sum(n * n for n in ns)), float(sum(n ** 3 for n in ns))
    want, solves = case["want"], case.get("iterations", 0) + 1
    layers = (Ld if want & 1 else 0) + (Le if want & 2 else 0)
    # one symmetric square (n^3 operations) per layer and chain; H read and D written once
    flops = n3 * (layers + (solves - 1) * Ld)
    return dict(bytes=8.0 * n2 + (4.0 * n2 if want & 1 else 0.0), flops=flops)


def _fermi(t):
    return torch.where(t > 0, torch.exp(-t.abs()) / (1 + torch.exp(-t.abs())), 1 / (1 + torch.exp(-t.abs())))


def _entropy(t):
    e = torch.exp(-t.abs())
    return torch.log1p(e) + t.abs() * e / (1 + e)


def _exact_of(Q, eps, mu, kT, want):
    f = _fermi((eps - mu) / kT)
    D = (Q * f) @ Q.T if want & 1 else None
    return D, torch.stack([f.sum(), (f * f).sum()]), _entropy((eps - mu) / kT).sum()


def exact(case, seed):
    if case["kind"] == "train":
        return None
    want = case["want"]
    if case["kind"] == "ragged":
        got = [_exact_of(Q, lam, mu, kT, want) for Q, lam, mu, kT in _spectra(case, seed)]
    else:
        eps, Q = torch.linalg.eigh(_hamiltonian(case, seed))
        mu, kT, n = case["mu"], case["kT"], eps.numel()
        steps = 0
        for _ in range(case.get("iterations", 0)):
            f = _fermi((eps - mu) / kT)
            off = n / 2.0 - float(f.sum())
            if abs(off) > 1e-6:
                mu += off / (float((f - f * f).sum()) / kT)
                steps += 1
        got = [_exact_of(Q, eps, mu, kT, want)]
    out = {}
    if want & 1:
        out["D"] = torch.cat([D.reshape(-1) for D, _, _ in got])
        out["trace"] = torch.stack([t for _, t, _ in got])
    if want & 2:
        out["S"] = torch.stack([S for _, _, S in got])
    if case["kind"] == "mu":
        out.update(steps=None, mu=np.array([mu]))
    return out

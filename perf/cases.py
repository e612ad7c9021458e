"""The work that a program built on this library has it do, as cases that can be timed.

The library applies the two-site Hamiltonian (``Plan.sigma``), finds its lowest
state (``Plan.davidson``), truncates it and moves to the next bond
(``Plan.decimate`` and ``Plan.set_bond``), and offers the block products behind
all of these on the caller's own buffers (``grouped_gemm``).  Each case is one
of these calls on a seeded problem of the shape that the benchmark and the tests
use: K orbitals, D states per bond, the sector split of ``synthetic_inputs``.

``kind``       the call: sigma, hdiag, davidson, move, gemm
``precision``  the plan's (or the product's) arithmetic: x3, x6, bf16 are bf16
               pieces on the tensor cores, fp64 the FP64 units (the default of
               ``Plan``), fp64tc FP64-accurate products on the tensor cores
"""
from __future__ import annotations

import functools
import math
import os
import random
import tempfile

import numpy as np
import torch

import paper_2311_02854_gb300 as lib
import synthetic_inputs as si

PRECISION = {"fp64": lib.DMRG_FP64, "x3": lib.DMRG_BF16X3, "bf16": lib.DMRG_BF16, "x6": lib.DMRG_BF16X6,
             "fp64tc": lib.DMRG_FP64_TC}
DAVIDSON_ITERS = 8


def _chain(name, kind, precision, K, D, bond, width=0.0, N=None, twoS=0, nvec=1):
    """A problem on a chain of K orbitals: N electrons (K where not given), width 0 the proportional sector split."""
    return {"name": name, "kind": kind, "precision": precision, "K": K, "N": K if N is None else N, "twoS": twoS, "D": D,
            "bond": bond, "width": width, "nvec": nvec}


def _gemm(name, precision, blocks, dim, depth, segments):
    return {"name": name, "kind": "gemm", "precision": precision, "blocks": blocks, "dim": dim, "depth": depth,
            "segments": segments}


def listed():
    return [
        # The smallest plan of the workloads (blocks up to 9 states): what a call costs when there is hardly any work in it,
        # as at the bonds near the ends of every chain.
        _chain("sigma_x3_k8_d64", "sigma", "x3", 8, 64, 4),
        # The mixed sigma where one output tile still sums several products: the parity size of the tests.
        _chain("sigma_x3_k14_d600", "sigma", "x3", 14, 600, 7, 1.0),
        # Four vectors in one call, as block Davidson for several states asks for them.
        _chain("sigma_x3_k24_d500_4vec", "sigma", "x3", 24, 500, 12, 1.45, nvec=4),
        # The mixed sigma of a production sweep (the middle bond of the benchmark's K = 36 workload): most of a run's time.
        _chain("sigma_x3_k36_d1000", "sigma", "x3", 36, 1000, 18, 1.45),
        # The default precision on a small system, as a user meets the library first; odd electron number.
        _chain("sigma_fp64_k10_d100", "sigma", "fp64", 10, 100, 5, N=9, twoS=1),
        # The default precision at the size of the parity tests.
        _chain("sigma_fp64_k14_d600", "sigma", "fp64", 14, 600, 7, 1.0),
        # FP64 accuracy on the tensor cores: the residuals of the corrected Davidson, final energies.
        _chain("sigma_fp64tc_k24_d500", "sigma", "fp64tc", 24, 500, 12, 1.45),
        # The diagonal of H that every Davidson call forms before its first step.
        _chain("hdiag_x3_k24_d500", "hdiag", "x3", 24, 500, 12, 1.45),
        # A whole eigensolver call (a fixed number of steps from a guess): sigma, orthogonalisation, Ritz steps.
        _chain("davidson_x3_k14_d600", "davidson", "x3", 14, 600, 7, 1.0),
        # There and back over one bond: density matrices, eigenvectors, renormalised operators, the next bond's lists.
        _chain("move_fp64tc_k14_d300", "move", "fp64tc", 14, 300, 7, 1.0),
        # Block products on the caller's buffers, blocks up to the sector size of the K = 73 workload.
        _gemm("gemm_x3_440", "x3", 48, 440, 440, 6),
        _gemm("gemm_fp64tc_152", "fp64tc", 40, 152, 152, 12),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "sigma", "sigma", "hdiag", "davidson", "move", "gemm", "gemm"])
    if kind == "gemm":
        precision = rng.choice(["x3", "x3", "fp64tc", "fp64"])
        big = {"x3": 440, "fp64tc": 256, "fp64": 152}[precision]
        case = _gemm("", precision, _spread(rng, 2, 48), _spread(rng, 7, big), _spread(rng, 7, big), rng.randint(1, 8))
    else:
        if kind == "move":
            precision = rng.choice(["fp64tc", "fp64"])
        else:
            precision = rng.choice(["x3", "x3", "x3", "x6", "bf16", "fp64", "fp64tc"])
        # the FP64 engines take what their rates let them do within the largest listed case
        K, D = {"fp64": (12, 400), "fp64tc": (20, 500)}.get(precision, (32, 900))
        if kind in ("move", "davidson"):
            K, D = min(K, 16), min(D, 300 if kind == "move" else 600)
        K = rng.randint(7, K)
        D = _spread(rng, 30, D)
        N = rng.randint(max(4, K - 3), K + 3)
        bond = rng.randint(3, K - 4) if kind == "move" else rng.randint(2, K - 2)
        width = rng.choice([0.0, 1.0, 1.2, 1.45])
        if D > 200:
            width = max(width, 1.0)
        nvec = rng.choice([1, 1, 2, 3]) if kind == "sigma" else 1
        case = _chain("", kind, precision, K, D, bond, width, N, N % 2, nvec)
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# Problems on a chain
# ---------------------------------------------------------------------------

def _plan(case, seed):
    """The plan of a chain problem at its bond: integrals and matrix product state from the seed."""
    K, N, twoS, k, w = case["K"], case["N"], case["twoS"], case["bond"], case["width"]
    h, chol = si.make_integrals(K, 4 * K, seed=2 * seed)
    bonds = si.bond_sectors(K, N, twoS, case["D"], "gaussian" if w else "proportional", w or None, w or None)
    mps = si.random_mps(K, N, twoS, bonds, center=k, seed=2 * seed + 1)
    with tempfile.TemporaryDirectory() as folder:
        path = os.path.join(folder, "mps.bin")
        si.write_mps(path, mps)
        plan = lib.Plan(h, chol, K, N, twoS, case["D"], path, precision=PRECISION[case["precision"]],
                        n_roots=case["nvec"])
    plan.set_bond(k)
    return plan


def _vectors(n, nvec, seed):
    """nvec normalised vectors of n standard-normal entries: a wavefunction with all its sectors filled."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((nvec, n), dtype=torch.float64, device="cuda", generator=gen)
    return x / x.norm(dim=1, keepdim=True)


# ---------------------------------------------------------------------------
# Block products on the caller's buffers
# ---------------------------------------------------------------------------

def _blocks(case):
    """Ragged output blocks of a few segments each, operands in both orders, and the lengths of a, b and c."""
    rng = random.Random("%s %d %d %d %d" % (case["precision"], case["blocks"], case["dim"], case["depth"],
                                            case["segments"]))
    blocks, a, b, c = [], 0, 0, 0
    for _ in range(case["blocks"]):
        m = rng.randint(max(1, case["dim"] // 3), case["dim"])
        n = rng.randint(max(1, case["dim"] // 3), case["dim"])
        segs = []
        for _ in range(case["segments"]):
            k = rng.randint(max(1, case["depth"] // 3), case["depth"])
            a_tr, b_tr = rng.randint(0, 1), rng.randint(0, 1)
            # leading dimensions as the tensor-core engine wants them
            lda, ldb = -(-(m if a_tr else k) // 8) * 8, -(-(k if b_tr else n) // 8) * 8
            segs.append((k, a, lda, a_tr, b, ldb, b_tr, rng.choice([1.0, -1.0])))
            a += (k if a_tr else m) * lda
            b += (n if b_tr else k) * ldb
        blocks.append((m, n, c, segs))
        c += m * n
    return blocks, a, b, c


def _operands(case, seed):
    blocks, na, nb, nc = _blocks(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(na, dtype=torch.float64, device="cuda", generator=gen)
    b = torch.randn(nb, dtype=torch.float64, device="cuda", generator=gen)
    return blocks, a, b, nc


# ---------------------------------------------------------------------------
# What is measured
# ---------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "gemm":
        blocks, a, b, nc = _operands(case, seed)
        return {"kind": "gemm", "precision": PRECISION[case["precision"]], "blocks": blocks, "a": a, "b": b,
                "c": torch.empty(nc, dtype=torch.float64, device="cuda")}
    plan = _plan(case, seed)
    state = {"kind": case["kind"], "plan": plan, "bond": case["bond"], "D": case["D"], "nvec": case["nvec"]}
    state["psi"] = _vectors(plan.dim, case["nvec"], seed)
    state["out"] = torch.empty_like(state["psi"])
    if case["kind"] == "move":
        # room for the state at the next bond and back here, whatever the truncation keeps of each sector
        state["ahead"], state["back"], state["out"] = (
            torch.zeros(4 * plan.dim + 65536, dtype=torch.float64, device="cuda") for _ in range(3))
        state["psi"] = state["psi"].reshape(-1).clone()
    return state


def _move(state):
    """Truncate the state to D and move one bond to the right, then back: what a sweep does between two eigensolver calls."""
    plan, k, psi, out = state["plan"], state["bond"], state["psi"], state["out"]
    weights = []
    for at, forward, ahead in ((k, True, state["ahead"]), (k + 1, False, state["back"])):
        w, dim = plan.decimate(psi, 1, state["D"], forward, next_psi=ahead, next_cap=ahead.numel())
        plan.set_bond(at + 1 if forward else at - 1)
        ahead[dim:].zero_()
        psi = ahead[:dim]
        weights.append(w)
    plan.sigma(psi, out)  # with the operators that the move renormalised
    out[dim:].zero_()
    state["psi"] = state["back"][:dim].clone()
    return {"discarded": np.array(weights), "psi": state["back"], "sigma": out}


def run(state):
    if state["kind"] == "gemm":
        lib.grouped_gemm(state["precision"], state["blocks"], state["a"], state["b"], state["c"])
        return state["c"]
    plan, psi, out = state["plan"], state["psi"], state["out"]
    if state["kind"] == "sigma":
        plan.sigma(psi, out, nvec=state["nvec"])
        return out
    if state["kind"] == "hdiag":
        plan.hdiag(out)
        return out
    if state["kind"] == "davidson":
        out.copy_(psi)
        energy, _, _ = plan.davidson(out, 1, tol=1e-10, max_iter=DAVIDSON_ITERS)
        return {"energy": energy, "psi": out}
    return _move(state)


@functools.lru_cache(maxsize=64)
def _counts(key):
    """Length of the wavefunction, operations of one sigma and bytes of the operators it reads, as the planner counts them."""
    plan = _plan(dict(key), 0)
    stats = plan.stats()
    got = plan.dim, stats["sigma_flops"], stats["store_bytes"] + stats["interm_bytes"], stats["interm_flops"]
    plan.close()
    return got


def work(case):
    if case["kind"] == "gemm":
        blocks, a, b, c = _blocks(case)
        return {"bytes": 8.0 * (a + b + c),
                "flops": sum(2.0 * m * n * sum(s[0] for s in segs) for m, n, _, segs in blocks)}
    dim, flops, operators, between = _counts(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    nvec = case["nvec"]
    if case["kind"] == "sigma":
        return {"bytes": operators + 16.0 * nvec * dim, "flops": nvec * flops}
    if case["kind"] == "hdiag":
        return {"bytes": 8.0 * dim, "flops": 2.0 * dim}
    if case["kind"] == "davidson":
        # per step: one sigma, its operators, the vector read and the result written
        return {"bytes": DAVIDSON_ITERS * (operators + 16.0 * dim), "flops": DAVIDSON_ITERS * flops}
    # two bonds' intermediates, the operators read and written, the last sigma
    return {"bytes": 4.0 * operators + 64.0 * dim, "flops": flops + 2.0 * between}


def exact(case, seed):
    """The block products in 64-bit arithmetic of torch; the chain problems need the method itself."""
    if case["kind"] != "gemm":
        return None
    blocks, a, b, nc = _operands(case, seed)
    c = torch.empty(nc, dtype=torch.float64, device="cuda")
    for m, n, off, segs in blocks:
        total = torch.zeros((m, n), dtype=torch.float64, device="cuda")
        for k, ao, lda, a_tr, bo, ldb, b_tr, alpha in segs:
            x = a[ao:ao + (k if a_tr else m) * lda].view(-1, lda)
            y = b[bo:bo + (n if b_tr else k) * ldb].view(-1, ldb)
            total += alpha * ((x[:, :m].t() if a_tr else x[:, :k]) @ (y[:, :k].t() if b_tr else y[:, :n]))
        c[off:off + m * n] = total.reshape(-1)
    return c

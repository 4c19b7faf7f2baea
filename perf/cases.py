"""Performance cases of the FCIQMC engine: what a program asks of it through its
public entry points (paper_1811_11679_gb300.hande), over the range of sizes,
systems, key widths and options that the repository's workloads and tests name.

Paths
  run            one report block of a production run: `cycles` iterations, their
                 estimator records and the walker list (the restart snapshot).
                 The state is an equilibrated run (grown to its target, the shift
                 varying), so every pass sees about the same population.
  batch          the same for many independent replicas advanced together.
  gradients      forward and backward of the learned proposal on a sample batch.
  probabilities  forward of the learned proposal (its masked softmax rows).
  gemm           the BF16 tensor-core product behind the learned proposal.
  estimate       projected-energy sums of a list the program holds on the device.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1811_11679_gb300 import hande, inputs

RECORD = ("iter", "nw_pre", "n0", "num_hi", "num_lo", "nw_post", "ndet", "natt", "nspawn", "shift", "num", "tau")


def listed():
    run = {"path": "run", "cycles": 20, "key_words": 1, "core": 0, "table": False}
    return [
        # the tutorial's 1D Hubbard ring: integer walkers on 4900 determinants; an
        # iteration is a chain of tiny kernels, latency is all there is
        dict(run, name="hubbard ring 8, 1e4", system="hubbard", norb=8, nalpha=4, nbeta=4, U=4.0, walkers=1e4,
             tau=0.01, real=False, initiator=False, cutoff=0.1, init=500.0),
        # half-filled 2D Hubbard cluster with a deterministic space (18 sites, U/t = 1.3)
        dict(run, name="hubbard 2d 18, 1e6", system="hubbard2d", norb=18, nalpha=9, nbeta=9, U=1.3, walkers=1e6,
             tau=0.002, real=True, initiator=True, cutoff=0.01, init=100.0, core=10000),
        # electron gas, uniform generator, 128-bit keys: the ordinary initiator calculation
        dict(run, name="ueg 14e/38, 1e6", system="ueg", norb=38, nalpha=7, nbeta=7, rs=1.0, key_words=2, walkers=1e6,
             tau=0.002, real=True, initiator=True, cutoff=0.1, init=5e4),
        # the larger basis of the replica workload: 512-bit keys
        dict(run, name="ueg 14e/66, 3e5", system="ueg", norb=66, nalpha=7, nbeta=7, rs=1.0, key_words=8, walkers=3e5,
             tau=0.002, real=True, initiator=True, cutoff=0.1, init=2e4),
        # electron gas drawn from a proposal table (what the learned proposal runs on)
        dict(run, name="ueg 14e/38 table, 2e5", system="ueg", norb=38, nalpha=7, nbeta=7, rs=1.0, key_words=2,
             walkers=2e5, tau=0.002, real=True, initiator=True, cutoff=0.1, init=2e4, table=True),
        # a small molecule calculation: odd electron number, modest walker number
        dict(run, name="molecule 15e/28, 1e5", system="molecule", norb=28, nalpha=8, nbeta=7, walkers=1e5, tau=0.01,
             real=True, initiator=True, cutoff=0.1, init=1e4, core=1000),
        # the headline workload: 1e7 walkers, heat-bath, semi-stochastic core of 1e4
        dict(run, name="molecule 15e/28, 1e7", system="molecule", norb=28, nalpha=8, nbeta=7, walkers=1e7, tau=0.01,
             real=True, initiator=True, cutoff=0.1, init=1e5, core=10000),
        # error bars from independent small runs: both key widths, uneven sizes
        {"name": "32 ueg replicas, 2e3-2e4", "path": "batch", "cycles": 10, "replicas": 32, "lo": 2e3, "hi": 2e4},
        # a training step's gradients at the default batch of the 38-orbital basis
        {"name": "gradients 38, 4096", "path": "gradients", "norb": 38, "width": 256, "batch": 4096, "count": 4096},
        # network output of a batch of rows at the largest basis the tests use
        {"name": "probabilities 246, 4096", "path": "probabilities", "norb": 246, "width": 256, "batch": 4096,
         "count": 4000},
        # the first layer of the 246-orbital table refresh
        {"name": "gemm 121088x256x512", "path": "gemm", "m": 121088, "n": 256, "k": 512},
        # the estimator of a caller-owned list inside a latency-critical loop: the smallest call
        {"name": "estimate ueg 3e4", "path": "estimate", "system": "ueg", "norb": 38, "nalpha": 7, "nbeta": 7,
         "rs": 1.0, "key_words": 2, "ndet": 30011},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    what = rng.choice(["hubbard", "hubbard2d", "ueg", "ueg", "ueg", "molecule", "molecule", "molecule", "batch",
                       "gradients", "probabilities", "gemm", "gemm", "estimate"])
    run = {"path": "run", "cycles": rng.randint(12, 20), "key_words": 1, "core": 0, "table": False, "system": what,
           "cutoff": round(rng.uniform(0.02, 0.2), 3)}
    if what == "hubbard":
        norb = rng.choice([6, 8, 10, 12])
        walkers = _log(rng, 3e3, 1e5)
        return dict(run, norb=norb, nalpha=norb // 2, nbeta=norb // 2 - rng.randint(0, 1), U=round(rng.uniform(2, 6), 2),
                    walkers=walkers, tau=0.01 * 8 / max(norb, 8), real=rng.random() < 0.4, initiator=False, init=500.0)
    if what == "hubbard2d":
        half = rng.choice([2, 3, 3, 4])
        norb = 2 * half * half
        return dict(run, norb=norb, nalpha=norb // 2, nbeta=norb // 2, U=round(rng.uniform(1, 4), 2),
                    walkers=_log(rng, 2e4, 1e6), tau=0.002 * min(1.0, 18 / norb), real=True, initiator=True, init=100.0,
                    core=rng.choice([0, 300, rng.randint(1000, 10000)]))
    if what == "ueg":
        norb = rng.choice([19, 25, 32, 33, 38, 45, 57, 64, 66])
        words = 1 if norb <= 32 else (2 if norb <= 64 else 8)
        walkers = _log(rng, 2e4, 1.5e6 if words < 8 else 4e5)
        return dict(run, norb=norb, nalpha=7, nbeta=7 - rng.randint(0, 1), rs=rng.choice([0.5, 1.0, 2.0, 5.0]),
                    key_words=words, walkers=walkers, tau=0.002, real=True, initiator=True,
                    init=min(0.3 * walkers, 2e4), table=rng.random() < 0.3, core=rng.choice([0, 0, 500]))
    if what == "molecule":
        walkers = _log(rng, 2e4, 8e6)
        return dict(run, norb=rng.choice([20, 23, 24, 27, 28]), nalpha=8, nbeta=rng.choice([6, 7, 7, 8]),
                    walkers=walkers, tau=0.01, real=True, initiator=True, init=min(0.1 * walkers, 1e5),
                    core=rng.choice([0, int(_log(rng, 100, 10000))]))
    if what == "batch":
        lo = _log(rng, 1e3, 5e3)
        return {"path": "batch", "cycles": rng.randint(5, 10), "replicas": rng.randint(5, 32), "lo": lo,
                "hi": lo * rng.uniform(2, 10)}
    if what == "gradients":
        batch = 128 * rng.randint(4, 64)
        return {"path": "gradients", "norb": rng.choice([19, 33, 38, 66, 129]), "width": 64 * rng.randint(2, 8),
                "batch": batch, "count": rng.randint(batch // 2, batch)}
    if what == "probabilities":
        batch = 128 * rng.randint(1, 64)
        return {"path": "probabilities", "norb": rng.choice([19, 38, 66, 123, 246]), "width": 64 * rng.randint(2, 8),
                "batch": batch, "count": rng.randint(batch // 2, batch)}
    if what == "gemm":
        return {"path": "gemm", "m": int(_log(rng, 100, 130000)), "n": int(_log(rng, 30, 520)),
                "k": int(_log(rng, 40, 1100))}
    norb = rng.choice([19, 38, 64, 66])
    return {"path": "estimate", "system": "ueg", "norb": norb, "nalpha": 7, "nbeta": 7, "rs": 1.0,
            "key_words": 1 if norb <= 32 else (2 if norb <= 64 else 8), "ndet": int(_log(rng, 1e3, 1e6))}


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=8)
def _molecule(norb, nalpha, nbeta):
    return inputs.molecule_system(norb, nalpha, nbeta)


def _system(c):
    if c["system"] == "hubbard":
        return inputs.hubbard_system(c["norb"], c["nalpha"], c["nbeta"], 1.0, c["U"])
    if c["system"] == "hubbard2d":
        h = int(round(math.sqrt(c["norb"] / 2)))
        return inputs.hubbard_lattice_system([[h, h], [h, -h]], c["nalpha"], c["nbeta"], 1.0, c["U"])
    if c["system"] == "molecule":
        return _molecule(c["norb"], c["nalpha"], c["nbeta"])
    return dict(inputs.ueg_system(c["nalpha"] + c["nbeta"], c["norb"], c["rs"], c["key_words"]), nalpha=c["nalpha"],
                nbeta=c["nbeta"])


@functools.lru_cache(maxsize=8)
def _momentum(norb):
    """The `norb` plane waves of lowest |n|^2, and for every row (I, J, same spin) of the
    proposal table the orbital B that goes with each A (-1: none), on the GPU."""
    r = range(-8, 9)
    pts = sorted((x * x + y * y + z * z, x, y, z) for x in r for y in r for z in r)[:norb]
    n = torch.tensor([p[1:] for p in pts], dtype=torch.int64, device="cuda")
    side = 33
    look = torch.full((side ** 3,), -1, dtype=torch.int64, device="cuda")
    code = lambda v: ((v[..., 0] + 16) * side + v[..., 1] + 16) * side + v[..., 2] + 16
    look[code(n)] = torch.arange(norb, device="cuda")
    b = n[:, None, None] + n[None, :, None] - n[None, None, :]
    B = torch.where(b.abs().amax(-1) <= 16, look[code(b.clamp(-16, 16))], -1)
    return n, B


def _drawable(norb):
    _, B = _momentum(norb)
    A = torch.arange(norb, device="cuda")
    ok = torch.stack([B >= 0, (B >= 0) & (B != A)], dim=2)        # [I, J, same, A]
    return ok.reshape(2 * norb * norb, norb)


def _table(norb):
    """Integer proposal weights proportional to |H| of each draw (what training aims at)."""
    n, B = _momentum(norb)
    d = (n[:, None, :] - n[None, :, :]).pow(2).sum(-1).double()
    v = torch.where(d > 0, 1.0 / d.clamp(min=1), 0.0)             # v[I, A]
    direct = v[:, None, :].expand(norb, norb, norb)
    exch = torch.gather(v[:, None, :].expand(norb, norb, norb), 2, B.clamp(min=0))
    h = torch.stack([direct, (direct - exch).abs()], dim=2).reshape(2 * norb * norb, norb)
    ok = _drawable(norb)
    h = torch.where(ok, h + 1e-3, 0.0)
    q = torch.floor(h / h.sum(1, keepdim=True).clamp(min=1e-30) * 2.0 ** 24).clamp(min=1, max=2.0 ** 24)
    return torch.where(ok, q, 0.0).cpu().numpy().astype(np.uint32)


def _grow(advance, records, target, limit=1500, settle=240):
    """Iterations until the population has passed its target, then `settle` more."""
    done = 0
    while done < limit:
        advance(60)
        done += 60
        if records()["nw_post"][-1] > target * hande.ONE_WALKER:
            break
    advance(settle)
    records()


def _prepare_run(c, seed):
    w = float(c["walkers"])
    q = inputs.qmc_params(tau=c["tau"], target_population=w, initiator=int(c["initiator"]),
                          real_amplitudes=int(c["real"]), spawn_cutoff=c["cutoff"], init_pop=c["init"],
                          semi_stoch_size=c["core"], semi_stoch_start=480 if c["core"] else 0, seed=1000 + seed,
                          excit_gen=int(c["table"]), state_capacity=int(1.6 * w) + 200_000,
                          spawn_capacity=int(4 * w) + 400_000)
    h = hande.Hande(_system(c), q)
    if c["table"]:
        h.set_proposal(_table(c["norb"]))
    _grow(h.iterate, h.estimators, w)
    if c["core"] and h.iterations < 540:       # past the iteration that chooses the deterministic space
        h.iterate(540 - h.iterations)
        h.estimators()
    return {"h": h, "cycles": c["cycles"], "buffers": _buffers(h, int(w * LIST[c["system"]]) + 80_000)}


def _buffers(h, capacity):
    """Page-locked list buffers, kept for the whole run as a restart writer keeps them
    (entries past the list's length stay as they were)."""
    out = h.host_buffers(capacity)
    for a in out:
        a[...] = 0
    return out


def _prepare_batch(c, seed):
    rng = np.random.Generator(np.random.Philox(100 + seed))
    systems, qmcs = [], []
    for r in range(c["replicas"]):
        norb = (38, 66)[r % 2]
        target = float(np.exp(np.log(c["lo"]) + (np.log(c["hi"]) - np.log(c["lo"])) * (r + rng.uniform()) / c["replicas"]))
        systems.append(inputs.ueg_system(14, norb, (0.5, 1.0, 2.0, 5.0)[(r // 2) % 4]))
        qmcs.append(inputs.qmc_params(tau=0.002, target_population=target, initiator=1, real_amplitudes=1,
                                      spawn_cutoff=0.1, init_pop=0.5 * target, seed=1000 + seed, replica=r,
                                      state_capacity=int(1.5 * target) + (1 << 16),
                                      spawn_capacity=int(3 * target) + (1 << 17)))
    b = hande.HandeBatch(systems, qmcs)
    b.iterate(400)
    b.synchronize()
    for v in b.replicas:
        v.estimators()
    # one set of buffers per key width, a fixed share of it for each replica
    share = int(1.2 * c["hi"]) + 2000
    whole = {W: _buffers(next(v for v in b.replicas if v.W == W), share * sum(v.W == W for v in b.replicas))
             for W in (2, 8)}
    used, buffers = {2: 0, 8: 0}, []
    for v in b.replicas:
        o = used[v.W]
        used[v.W] += share
        buffers.append(tuple(a[o:o + share] for a in whole[v.W]))
    return {"b": b, "cycles": c["cycles"], "buffers": buffers, "whole": whole}


def _network(c, seed):
    """Seeded parameters in the order of hande.Hande.learn_params, and a sample batch."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    M, H = c["norb"], c["width"]
    u = lambda *s, lim=1.0: (torch.rand(*s, generator=g, device="cuda", dtype=torch.float64) * 2 - 1) * lim
    din = 2 * M + 1
    p = [u(H, din, lim=math.sqrt(6 / din)), u(H, lim=0.05), u(H, H, lim=math.sqrt(6 / H)), u(H, lim=0.05),
         u(M, H, lim=math.sqrt(6 / H)), u(M, lim=0.05)]
    p = [t.float() for t in p]
    ok = _drawable(M)
    rows = torch.randint(0, 2 * M * M, (c["count"],), generator=g, device="cuda")
    rows = torch.where(ok[rows].any(1), rows, torch.zeros_like(rows))
    score = torch.rand((c["count"], M), generator=g, device="cuda")
    targets = torch.where(ok[rows], score, -1.0).argmax(1)
    weights = torch.rand(c["count"], generator=g, device="cuda").pow(-0.4).clamp(max=20.0)   # a few large |H| / p
    return p, ok, rows, targets, weights


def _prepare_learner(c, seed):
    p, _, rows, targets, weights = _network(c, seed)
    q = inputs.qmc_params(target_population=100.0, init_pop=10.0, initiator=1, real_amplitudes=1, excit_gen=1,
                          state_capacity=4096, spawn_capacity=8192, seed=1000 + seed)
    h = hande.Hande(inputs.ueg_system(14, c["norb"], 1.0), q)
    h.learn_proposal(width=c["width"], batch=c["batch"], period=0, seed=seed)
    h.learn_params(torch.cat([t.reshape(-1) for t in p]).cpu().numpy())
    return {"h": h, "rows": rows.to(torch.int32).cpu().numpy(), "targets": targets.to(torch.int32).cpu().numpy(),
            "weights": weights.float().cpu().numpy()}


def _operands(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ld = (c["k"] + 7) // 8 * 8
    a = torch.randn((c["m"], ld), generator=g, device="cuda").relu().to(torch.bfloat16)   # activations
    b = (torch.randn((c["n"], ld), generator=g, device="cuda") * math.sqrt(2 / c["k"])).to(torch.bfloat16)
    return a[:, :c["k"]], b[:, :c["k"]]


def _prepare_gemm(c, seed):
    a, b = _operands(c, seed)
    return {"a": a, "b": b, "out": torch.empty((c["m"], c["n"]), dtype=torch.float32, device="cuda"),
            "status": torch.zeros(1, dtype=torch.int32, device="cuda")}


def _prepare_estimate(c, seed):
    h = hande.Hande(_system(c), inputs.qmc_params(target_population=100.0, init_pop=10.0, state_capacity=4096,
                                                  spawn_capacity=8192, seed=1000 + seed))
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, W, norb = c["ndet"], c["key_words"], c["norb"]
    occ = torch.zeros((n, 2 * norb), dtype=torch.bool, device="cuda")
    for spin, nel in ((0, c["nalpha"]), (1, c["nbeta"])):
        # the lowest orbitals with up to two of them excited: most determinants connect to the reference
        score = torch.arange(norb, device="cuda").float().expand(n, norb).clone()
        moves = torch.randint(0, 3, (n, 1), generator=g, device="cuda")
        for k in range(2):
            hole = torch.randint(0, nel, (n, 1), generator=g, device="cuda")
            part = torch.randint(nel, norb, (n, 1), generator=g, device="cuda")
            use = moves > k
            score.scatter_(1, hole, torch.where(use, 1e6, score.gather(1, hole)))
            score.scatter_(1, part, torch.where(use, -1.0, score.gather(1, part)))
        pick = score.argsort(dim=1, stable=True)[:, :nel]
        occ.scatter_(1, 2 * pick + spin, True)
    occ[0] = False                                                # the reference itself
    occ[0, torch.arange(c["nalpha"], device="cuda") * 2] = True
    occ[0, torch.arange(c["nbeta"], device="cuda") * 2 + 1] = True
    bits = torch.nn.functional.pad(occ, (0, 64 * W - 2 * norb)).reshape(n, W, 64).to(torch.int64)
    keys = (bits << torch.arange(64, device="cuda")).sum(2)
    pops = torch.randn(n, generator=g, device="cuda", dtype=torch.float64).mul(3 * 2.0 ** 32).round().to(torch.int64)
    return {"h": h, "keys": keys.contiguous(), "pops": pops, "out": torch.zeros(4, dtype=torch.int64, device="cuda")}


def prepare(case, seed):
    p = case["path"]
    if p == "run":
        s = _prepare_run(case, seed)
    elif p == "batch":
        s = _prepare_batch(case, seed)
    elif p in ("gradients", "probabilities"):
        s = _prepare_learner(case, seed)
    elif p == "gemm":
        s = _prepare_gemm(case, seed)
    else:
        s = _prepare_estimate(case, seed)
    s["path"] = p
    return s


# ------------------------------------------------------------------ one pass
def _records(r):
    return {k: (r[k].view(np.int64) if r[k].dtype == np.uint64 else r[k]) for k in RECORD}


def _list(buffers):
    return {k: a.view(np.int64) if a.dtype == np.uint64 else a for k, a in zip(("keys", "pops", "hdiag", "core"), buffers)}


def run(state):
    p = state["path"]
    if p == "run":
        h = state["h"]
        h.iterate(state["cycles"])
        rec = _records(h.estimators())
        h.walkers(out=state["buffers"])
        return {"records": rec, "list": _list(state["buffers"])}
    if p == "batch":
        b = state["b"]
        b.iterate(state["cycles"])
        rec = [_records(v.estimators()) for v in b.replicas]
        for v, buf in zip(b.replicas, state["buffers"]):
            v.walkers(out=buf)
        return {"records": {k: np.concatenate([r[k] for r in rec]) for k in RECORD},
                "lists": {str(W): _list(a) for W, a in state["whole"].items()}}
    if p == "gradients":
        loss, grads = state["h"].learn_gradients(state["rows"], state["targets"], state["weights"])
        return {"loss": loss, "grads": grads}
    if p == "probabilities":
        return {"p": state["h"].learn_probabilities(state["rows"])}
    if p == "gemm":
        return {"d": hande.gemm_bf16(state["a"], state["b"], out=state["out"], status=state["status"])}
    h, out = state["h"], state["out"]
    h.estimate_noalloc(state["keys"].data_ptr(), state["pops"].data_ptr(), len(state["pops"]), out.data_ptr())
    return {"sums": out}


# ------------------------------------------------------------------ work and exact values
# determinants per walker, spawns per walker and final walkers per target walker of
# the equilibrated runs (measured; they set the bytes an iteration has to move)
SHAPE = {"hubbard": (0.145, 0.11, 2.5), "hubbard2d": (0.5, 0.7, 2.2), "ueg": (0.6, 0.25, 1.03),
         "molecule": (0.19, 0.11, 1.22)}


def _run_bytes(system, words, walkers, cycles):
    dets, spawns, grown = SHAPE[system]
    n = walkers * grown
    # the list read and written once (key, population, diagonal, flag), each spawn
    # (key, amount, initiator bit) written and read once
    return cycles * n * (2 * dets * (8 * words + 17) + 2 * spawns * (8 * words + 9))


def work(case):
    p = case["path"]
    if p == "run":
        # one Philox4x64-10 block (20 wide products) per attempt
        n = case["walkers"] * SHAPE[case["system"]][2] * case["cycles"]
        return {"bytes": _run_bytes(case["system"], case["key_words"], case["walkers"], case["cycles"]), "flops": 20 * n}
    if p == "batch":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        n = case["replicas"] * mean
        return {"bytes": _run_bytes("ueg", 2, n / 2, case["cycles"]) + _run_bytes("ueg", 8, n / 2, case["cycles"]),
                "flops": 20 * n * case["cycles"]}
    if p in ("gradients", "probabilities"):
        M, H, n = case["norb"], case["width"], case["count"]
        par = H * (2 * M + 1) + H + H * H + H + M * H + M
        mac = n * (H * H + M * H)                                 # the first layer is a gather of three columns
        if p == "gradients":
            return {"bytes": 12 * n + 8 * par, "flops": 6 * mac}
        return {"bytes": 4 * n + 4 * par + 4 * n * M, "flops": 2 * mac}
    if p == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 2 * (m + n) * k + 4 * m * n, "flops": 2 * m * n * k}
    return {"bytes": case["ndet"] * 8 * (case["key_words"] + 1), "flops": 0}


# room for the list, per target walker
LIST = {"hubbard": 1.0, "hubbard2d": 2.0, "ueg": 1.0, "molecule": 0.36}


def exact(case, seed):
    """64-bit values of the dense paths; the Monte Carlo runs have none (their lists are
    whole numbers drawn at random)."""
    p = case["path"]
    if p == "gemm":
        a, b = _operands(case, seed)
        return {"d": torch.cat([x.double() @ b.double().T for x in a.split(16384)])}
    if p not in ("gradients", "probabilities"):
        return None
    par, ok, rows, targets, weights = _network(case, seed)
    M = case["norb"]
    par = [t.double().requires_grad_(True) for t in par]
    W1, b1, W2, b2, W3, b3 = par
    I, J, same = (rows >> 1) // M, (rows >> 1) % M, (rows & 1).double()
    x = torch.zeros((len(rows), 2 * M + 1), dtype=torch.float64, device="cuda")
    x.scatter_(1, I[:, None], 1.0)
    x.scatter_(1, M + J[:, None], 1.0)
    x[:, 2 * M] = same
    z = torch.relu(torch.relu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    logp = torch.log_softmax(z.masked_fill(~ok[rows], -math.inf), dim=1)
    if p == "probabilities":
        return {"p": logp.detach().exp().cpu().numpy()}
    c = weights.double() / weights.double().sum()
    loss = -(c * logp.gather(1, targets[:, None])[:, 0]).sum()
    grads = torch.autograd.grad(loss, par)
    return {"loss": float(loss.detach()), "grads": torch.cat([g.reshape(-1) for g in grads]).cpu().numpy()}

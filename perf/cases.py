"""What this library's users have it do, as cases that can be timed and compared.

Every case goes through the public binding (``paper_2402_03920_gb300.qisg``):

* ``sweep``: Monte Carlo sweeps with parallel tempering of one handle, and the
  read-out that follows them (measurement sums, energies, permutation, and
  the configurations where a program of that size would write them), in
  every packing and option that is used in earnest;
* ``uneven``: many instances of uneven size advanced together by the batch
  kernel, and their results;
* ``tau``: the imaginary-time observables of a handle's configurations;
* ``transfer``: one product of the exact-diagonalisation transfer matrix.

Sizes are those of ``workloads.py``, the benchmark and the tests.  A handle is
created and thermalised for a few sweeps in ``prepare``; each pass continues
its run, as a simulation does.  Whole numbers must be the same; the two
floating results (SF of ``tau``, the vector of ``transfer``) have tolerances.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2402_03920_gb300 import qisg, workloads

_LAYOUT = {"auto": qisg.QISG_LAYOUT_AUTO, "lanes": qisg.QISG_LAYOUT_LANES, "samples": qisg.QISG_LAYOUT_SAMPLES,
           "sites": qisg.QISG_LAYOUT_SITES}


def _sweep(L, L_tau, slots, replicas, samples, sweeps, layout="auto", word_bits=0, measure_every=10, pt_every=1,
           per_sample=False, persistent=False, antiperiodic=False, equal=False, spins=False):
    """A ``sweep`` case.  ``equal``: the paper's single coupling k_tau = k,
    else k_tau from Gamma = 1."""
    return {"kind": "sweep", "L": L, "L_tau": L_tau, "slots": slots, "replicas": replicas, "samples": samples,
            "sweeps": sweeps, "layout": layout, "word_bits": word_bits, "measure_every": measure_every,
            "pt_every": pt_every, "per_sample": per_sample, "persistent": persistent, "antiperiodic": antiperiodic,
            "equal": equal, "spins": spins}


def listed():
    P = workloads.PRODUCTION
    B = workloads.BATCHED
    S = workloads.PLAIN_SMALL
    return [
        # the smallest run: one sample of 64 kB of spins, ten sweeps and
        # everything read back (interactive use, tests, equilibration checks)
        dict(_sweep(S.L, S.L_tau, S.n_slots, S.n_replicas, S.n_samples, 10, "lanes", S.word_bits, spins=True),
             name="plain_small"),
        # the production lattice in the per-instance form: one launch per
        # sample and half sweep
        dict(_sweep(P.L, P.L_tau, P.n_slots, P.n_replicas, P.n_samples, 10, "lanes", P.word_bits, per_sample=True),
             name="per_instance"),
        # the benchmark's step: ten sweeps of the production batch, one
        # measurement, the sums read back
        dict(_sweep(P.L, P.L_tau, P.n_slots, P.n_replicas, P.n_samples, 10), name="production_step"),
        # a block of measurements of the same batch, after which the
        # configurations are written out
        dict(_sweep(P.L, P.L_tau, P.n_slots, P.n_replicas, P.n_samples, 2000, spins=True), name="production_block"),
        # ragged: planes that do not fill a block, a second replica quad half
        # empty, a partly filled word, an antiperiodic boundary
        dict(_sweep(12, 90, 11, 6, 27, 200, "samples", 32, antiperiodic=True, spins=True), name="ragged"),
        # the HBM-sized batch with 32-bit words
        dict(_sweep(B.L, B.L_tau, B.n_slots, B.n_replicas, B.n_samples, 20, "samples", 32, measure_every=20),
             name="batched_1024"),
        # the same lattice with 64 samples per word (the default word of large batches)
        dict(_sweep(B.L, B.L_tau, B.n_slots, B.n_replicas, 256, 20, measure_every=20), name="batched_w64"),
        # the batch as one cooperative launch per run of sweeps
        dict(_sweep(B.L, B.L_tau, B.n_slots, B.n_replicas, 256, 20, "samples", 32, measure_every=20, persistent=True),
             name="persistent"),
        # the paper's own update rule at its performance lattice
        dict(_sweep(16, 8192, 16, 4, 16, 10, "sites", 32, equal=True), name="daemon_rule"),
        # 512 instances of uneven size in one batch (the serving loop's kernel)
        {"name": "uneven_batch", "kind": "uneven", "instances": 512, "sweeps": 20, "mix": 2024},
        # the analysis quantities of the production batch's configurations
        {"name": "tau_production", "kind": "tau", "L": P.L, "L_tau": P.L_tau, "slots": P.n_slots,
         "replicas": P.n_replicas, "samples": P.n_samples, "layout": "auto", "word_bits": 0},
        # the largest product one GPU holds
        {"name": "transfer_L5", "kind": "transfer", "L": 5, "parity": 1, "k": 0.3, "gamma": 1.0},
    ]


def _log_int(rng, lo, hi, step=1):
    """An integer multiple of step in [lo, hi], uniform over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + step)))
    return max(lo, min(hi, int(v / step) * step))


def _updates(c):
    return float(c["L"] ** 2 * c["L_tau"] * c["slots"] * c["replicas"] * c["samples"])


def draw(rng):
    kind = rng.choice(["lanes", "samples", "samples", "samples", "sites", "uneven", "tau", "transfer"])
    if kind == "transfer":
        return {"kind": "transfer", "L": rng.choice([3, 4, 4, 5, 5, 5]), "parity": rng.choice([1, -1]),
                "k": round(rng.uniform(0.2, 0.5), 4), "gamma": round(rng.uniform(0.8, 1.2), 4)}
    if kind == "uneven":
        return {"kind": "uneven", "instances": _log_int(rng, 4, 400), "sweeps": rng.randint(3, 20),
                "mix": rng.randrange(1 << 20)}
    while True:   # no dearer than the largest listed case
        if kind == "tau":
            c = {"kind": "tau", "L": 2 * rng.randint(2, 12), "L_tau": _log_int(rng, 16, 512, 2),
                 "slots": rng.randint(4, 16), "replicas": rng.randint(2, 6), "samples": _log_int(rng, 1, 32),
                 "layout": rng.choice(["auto", "samples"]), "word_bits": rng.choice([0, 64])}
            if _updates(c) <= 1.4e8:
                return c
            continue
        if kind == "lanes":
            slots = rng.randint(4, 16)
            c = _sweep(2 * rng.randint(3, 12), _log_int(rng, 32, 1024, 2), slots, rng.randint(1, min(6, 2 * (64 // slots))),
                       _log_int(rng, 1, 32), 10 * rng.randint(1, 3), "lanes", 64, per_sample=rng.random() < 0.5,
                       antiperiodic=rng.random() < 0.3)
        elif kind == "sites":
            c = _sweep(2 * rng.randint(3, 12), _log_int(rng, 128, 8192, 64), rng.randint(4, 16), rng.randint(2, 6),
                       _log_int(rng, 1, 16), 10, "sites", 32, antiperiodic=rng.random() < 0.3, equal=True)
        else:
            words = rng.choice([32, 32, 64])
            me = rng.choice([5, 10, 10, 20])
            c = _sweep(2 * rng.randint(3, 12), _log_int(rng, 32, 2048, 2), rng.randint(4, 32), rng.randint(2, 6),
                       _log_int(rng, 8, 512), me * rng.randint(1, 4), "samples", words, measure_every=me,
                       antiperiodic=rng.random() < 0.3, equal=rng.random() < 0.2,
                       persistent=words == 32 and rng.random() < 0.2)
        limit = {"lanes": 1.3e10, "sites": 2.2e10, "samples": 3e11}[kind]
        if _updates(c) * c["sweeps"] <= limit:
            return dict(c, spins=_updates(c) < 2e7)   # small states are read back whole


def _ladder(c):
    if c["equal"]:
        return qisg.ladder_equal(0.2, 0.5, c["slots"])
    return qisg.ladder_linear(0.2, 0.5, c["slots"], 1.0)


def _tau_spins(case, seed):
    """Configurations with the imaginary-time correlation of the thermalised
    ones: each site's line a Markov chain along tau, int8 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["samples"], case["replicas"], case["slots"], case["L_tau"], case["L"] ** 2)
    p = torch.linspace(0.35, 0.08, case["slots"], device="cuda").view(1, 1, -1, 1, 1)
    flips = torch.rand(shape, generator=g, device="cuda", dtype=torch.float32) < p
    return (1 - 2 * (flips.cumsum(3, dtype=torch.int32) & 1)).to(torch.int8)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        inst = qisg.Instance(qisg.Config(
            case["L"], case["L_tau"], _ladder(case), case["replicas"], case["samples"], seed + 1,
            word_bits=case["word_bits"], pt_every=case["pt_every"], measure_every=case["measure_every"],
            layout=_LAYOUT[case["layout"]], per_sample_launch=int(case["per_sample"]),
            tau_antiperiodic=int(case["antiperiodic"])))
        if case["persistent"]:
            inst.set_persistent(True)
        inst.sweep(2 * case["measure_every"])
        inst.sync()
        return {"case": case, "inst": inst}
    if kind == "uneven":
        specs = workloads.uneven_batch(case["instances"], case["mix"])
        lads = [qisg.ladder_linear(s.k_lo, s.k_hi, s.n_slots, s.gamma) for s in specs]
        room = sum(qisg.Batch.instance_bytes(s.L, s.L_tau, ld, s.n_replicas) + 256 for s, ld in zip(specs, lads))
        batch = qisg.Batch(case["instances"], room + (1 << 20))
        slots = [batch.admit(s.L, s.L_tau, ld, s.n_replicas, (seed + 1) * 100003 + s.seed) for s, ld in zip(specs, lads)]
        batch.run(2)
        batch.sync()
        return {"case": case, "batch": batch, "slots": slots}
    if kind == "tau":
        inst = qisg.Instance(qisg.Config(
            case["L"], case["L_tau"], qisg.ladder_linear(0.2, 0.5, case["slots"], 1.0), case["replicas"],
            case["samples"], seed + 1, word_bits=case["word_bits"], layout=_LAYOUT[case["layout"]]))
        walker_at = workloads.random_permutations(case["samples"] * case["replicas"], case["slots"], seed)
        inst.set_state(_tau_spins(case, seed).cpu().numpy(), walker_at, 1000)
        return {"case": case, "inst": inst}
    n = 1 << (case["L"] ** 2 - 1)
    x, J, k_tau = _transfer_inputs(case, seed)
    return {"case": case, "x": x, "y": torch.empty(n, dtype=torch.float64, device="cuda"), "J": J, "k_tau": k_tau}


def _transfer_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(1 << (case["L"] ** 2 - 1), generator=g, device="cuda", dtype=torch.float64)
    J = np.random.default_rng(seed).choice(np.array([-1, 1], dtype=np.int8), size=(case["L"] ** 2, 2))
    return x / x.norm(), J, -0.5 * math.log(math.tanh(case["k"] * case["gamma"]))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweep":
        inst = state["inst"]
        inst.sweep(case["sweeps"])
        sumA, sumB, sumq, sumq2, n_meas = inst.measurements()
        A, B = inst.energies()
        out = {"sumA": sumA, "sumB": sumB, "sumq": sumq, "sumq2": sumq2, "n_meas": n_meas, "A": A, "B": B,
               "walker_at": inst.permutation()}
        if case["spins"]:
            out["S"] = inst.spins()
        return out
    if kind == "uneven":
        batch = state["batch"]
        batch.run(case["sweeps"])
        res = [batch.results(s) for s in state["slots"]]
        return {"A": np.concatenate([r[0].ravel() for r in res]), "B": np.concatenate([r[1].ravel() for r in res]),
                "walker_at": np.concatenate([r[2].ravel() for r in res])}
    if kind == "tau":
        S1, S2, S4, SF = state["inst"].tau_observables()
        return {"S1": S1, "S2": S2, "S4": S4, "SF": SF}
    qisg.transfer_matvec(state["x"].data_ptr(), state["y"].data_ptr(), case["L"], case["k"], state["k_tau"], state["J"],
                         case["parity"])
    return state["y"]


def work(case):
    """Bytes: the state read once and written once, and the results.  Flops
    of the sweeps: integer operations on 32-bit words, about 52 per word of
    32 spins with a quarter Philox call per word (SAMPLES), a quarter Philox
    call and a comparison per spin (LANES), three Philox calls and twelve
    look-ups per word (SITES)."""
    kind = case["kind"]
    if kind == "sweep":
        n = _updates(case)
        chains = case["samples"] * case["replicas"] * case["slots"]
        out = chains * 36.0 + (n if case["spins"] else 0.0)
        per = {"lanes": 14.0, "sites": 9.0}.get(case["layout"], 1.64)
        return {"bytes": 2 * n / 8 + out, "flops": per * n * case["sweeps"]}
    if kind == "uneven":
        specs = workloads.uneven_batch(case["instances"], case["mix"])
        n = float(sum(s.L ** 2 * s.L_tau * s.n_slots * s.n_replicas for s in specs))
        return {"bytes": 2 * n / 8, "flops": 14.0 * n * case["sweeps"]}
    if kind == "tau":
        # per pair of time slices: two exclusive-ors and counts per row and
        # column and the squared moduli from their folded sums
        cfg = float(case["samples"] * case["replicas"] * case["slots"])
        pairs = cfg * case["L_tau"] * (case["L_tau"] // 2 + 1)
        return {"bytes": cfg * (case["L"] ** 2 * case["L_tau"] / 8 + 32.0 * case["L_tau"]),
                "flops": pairs * 6.0 * case["L"]}
    n = float(1 << (case["L"] ** 2 - 1))
    return {"bytes": 16 * n, "flops": n * (2 * (case["L"] ** 2 - 1) + 4)}


def tolerance(case):
    """Whole numbers are the same.  Doubles: about four times the distance
    from ``exact`` that was measured (SF 4.2e-16, the product 1.1e-15)."""
    if case["kind"] == "tau":
        return {"rel": 2e-15}
    if case["kind"] == "transfer":
        return {"rel": 5e-15}
    return "exact"


def _tau_exact(case, seed):
    """SF by slot from the definition, in FP64 on the GPU."""
    S = _tau_spins(case, seed)
    a, r, w, T, P = S.shape
    L = case["L"]
    walker_at = torch.from_numpy(
        workloads.random_permutations(a * r, w, seed).astype(np.int64)).cuda().view(a * r, w)
    S = S.view(a * r, w, T, L, L)   # [.., tau, x2, x1]
    S = torch.gather(S, 1, walker_at.view(a * r, w, 1, 1, 1).expand_as(S)).reshape(a * r * w, T, L, L)
    th = 2 * math.pi * torch.arange(L, device="cuda", dtype=torch.float64) / L
    cs, sn = torch.cos(th), torch.sin(th)
    t1 = torch.arange(T, device="cuda")
    t2 = (t1.view(-1, 1) + t1.view(1, -1)) % T   # [t1][lag]
    SF = torch.empty(a * r * w, T, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // (T * T * L))
    for lo in range(0, a * r * w, step):
        s = S[lo:lo + step].double()
        tot = 0.0
        for perm in ((3, 1), (2, 1)):   # sums over x2 at fixed x1, then over x1 at fixed x2
            v = s.movedim(perm[0], 1)                       # [cfg][kept][tau][summed]
            G = v @ v.transpose(-1, -2)                     # [cfg][kept][t1][t2]
            re = torch.einsum("cxij,x->cij", G, cs)
            im = torch.einsum("cxij,x->cij", G, sn)
            tot = tot + re * re + im * im
        SF[lo:lo + step] = torch.gather(tot, 2, t2.expand(tot.shape[0], T, T)).sum(1)
    return SF.view(a, r, w, T).cpu()


def _transfer_exact(case, seed):
    """The product round by round, in FP64 on the GPU."""
    x, J, k_tau = _transfer_inputs(case, seed)
    L, nb = case["L"], case["L"] ** 2 - 1
    n = torch.arange(1 << nb, device="cuda")
    spin = [1 - 2 * ((n >> j) & 1) for j in range(nb + 1)]   # the top site is +1 in this half
    E = torch.zeros_like(n)
    for x2 in range(L):
        for x1 in range(L):
            i = x1 + L * x2
            E += int(J[i][0]) * spin[i] * spin[(x1 + 1) % L + L * x2]
            E += int(J[i][1]) * spin[i] * spin[x1 + L * ((x2 + 1) % L)]
    w = torch.exp(0.5 * case["k"] * E.double())
    jP = math.exp(k_tau) / (math.exp(k_tau) + math.exp(-k_tau))
    jM = math.exp(-k_tau) / (math.exp(k_tau) + math.exp(-k_tau))
    v = x * w
    for j in range(nb):
        p = v.view(-1, 2, 1 << j)
        v = (jP * p + jM * p.flip(1)).reshape(-1)
    v = jP * v + case["parity"] * jM * v.flip(0)
    return (v * w).cpu()


def exact(case, seed):
    if case["kind"] == "tau":
        return {"S1": None, "S2": None, "S4": None, "SF": _tau_exact(case, seed)}
    if case["kind"] == "transfer":
        return _transfer_exact(case, seed)
    return None

"""What a user of this solver has it do, as cases that can be timed.

Every case goes through the package's public entry points.  Sizes come from the
repository's own workloads (`paper_2504_00987_gb300/workloads.py`, `bench.py`,
`README.md`) and tests; `draw` spreads more cases over the same ranges.

Kinds of case:
  run         blocking Memetic-Tabu run, results on the host     (mts_run)
  launch      asynchronous Memetic-Tabu launch                   (mts_launch)
  resume      a run in two checkpointed slices                   (mts_resume)
  batch       uneven instances in one autotuned graph launch     (Batch)
  serve       a burst of requests through the solve service      (Server)
  tabu        one tabu search per start sequence                 (tabu_run)
  energy      E of a batch of sequences, optionally all C_k      (energy_batch)
  skew_dev    deviation from skew symmetry of a batch            (skew_deviation_batch)
"""
import math
import random
import time

import numpy as np
import torch

import paper_2504_00987_gb300 as labs

DEV = "cuda"


def listed():
    return [
        # The smallest solve: one N = 24 instance to 2,000 generations, results on the host.
        {"name": "run_n24_one", "kind": "run", "N": 24, "K": 100, "replicas": 1, "generations": 2000,
         "variant": 0, "worst": False},
        # The headline workload: 1,024 replicas x 10^5 tabu steps of a one-word sequence.
        {"name": "launch_n64_r1024", "kind": "launch", "N": 64, "K": 100, "replicas": 1024, "steps": 100_000,
         "variant": 0, "worst": False},
        # The N = 92..120 sweep at its largest N, 16 replicas on every SM (a tenth of its step budget).
        {"name": "launch_n120_r2432", "kind": "launch", "N": 120, "K": 100, "replicas": 2432, "steps": 100_000,
         "variant": 0, "worst": False},
        # Search restricted to skew-symmetric sequences, odd N, replace-worst population.
        {"name": "launch_n101_skew", "kind": "launch", "N": 101, "K": 100, "replicas": 1216, "steps": 10_000,
         "variant": labs.VARIANT_SKEW, "worst": True},
        # A long run kept as checkpoints: one slice from scratch, one continued from its records.
        {"name": "resume_n92_r608", "kind": "resume", "N": 92, "K": 100, "replicas": 608, "generations": 100},
        # 512 instances of uneven N, K and budget (10 N^2 steps) in one captured launch.
        {"name": "batch_uneven_512", "kind": "batch", "count": 512, "n_lo": 40, "n_hi": 127, "steps_per_n2": 10},
        # As many requests at once as the Poisson stream keeps in flight, N = 32..160, step caps and targets.
        {"name": "serve_burst_64", "kind": "serve", "count": 64, "n_lo": 32, "n_hi": 160, "steps": 20_000},
        # Local search from given starts at long N (default search length), a ragged number of them.
        {"name": "tabu_n201_b5000", "kind": "tabu", "N": 201, "B": 5000, "variant": 0},
        # Energies of one population: a call that is all latency.
        {"name": "energy_n64_b100", "kind": "energy", "N": 64, "B": 100, "with_C": False},
        # Energies of a large sample.
        {"name": "energy_n120_b1m", "kind": "energy", "N": 120, "B": 1_000_000, "with_C": False},
        # Energies and every correlation, odd N and a ragged number of sequences.
        {"name": "corr_n127_b300007", "kind": "energy", "N": 127, "B": 300_007, "with_C": True},
        # d(S) of 100,000 random sequences.
        {"name": "skew_dev_n120_b100k", "kind": "skew_dev", "N": 120, "B": 100_000},
    ]


def _log_int(rng, lo, hi):
    """An integer in lo..hi, uniform over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["run", "launch", "launch", "launch", "resume", "batch", "serve", "tabu", "tabu",
                       "energy", "energy", "skew_dev"])
    variant = rng.choice([0, 0, 0, labs.VARIANT_FIX_FIRST_SPIN, labs.VARIANT_UNIFORM_CROSSOVER, labs.VARIANT_SKEW])
    worst = rng.random() < 0.25
    N = _log_int(rng, 20, 256)
    if variant & labs.VARIANT_SKEW:
        N = min(N | 1, 255)
    if kind == "run":
        return {"kind": kind, "N": N, "K": rng.randint(20, 200), "replicas": _log_int(rng, 1, 64),
                "generations": _log_int(rng, 20, 400), "variant": variant, "worst": worst}
    if kind == "launch":
        replicas = _log_int(rng, 1, 2432)
        # a replica's steps: at most 10^5, fewer for long sequences
        steps = _log_int(rng, 1000, min(100_000, 100_000 * 64 // N))
        return {"kind": kind, "N": N, "K": rng.randint(20, 200), "replicas": replicas, "steps": steps,
                "variant": variant, "worst": worst}
    if kind == "resume":
        return {"kind": kind, "N": N, "K": rng.randint(20, 200), "replicas": _log_int(rng, 1, 2432),
                "generations": _log_int(rng, 10, 100)}
    if kind == "batch":
        lo = rng.randint(32, 120)
        return {"kind": kind, "count": _log_int(rng, 16, 512), "n_lo": lo, "n_hi": rng.randint(lo, 160),
                "steps_per_n2": rng.randint(1, 5)}
    if kind == "serve":
        lo = rng.randint(32, 120)
        return {"kind": kind, "count": _log_int(rng, 1, 128), "n_lo": lo, "n_hi": rng.randint(lo, 160),
                "steps": _log_int(rng, 1000, 20_000)}
    if kind == "tabu":
        return {"kind": kind, "N": N, "B": _log_int(rng, 8, 20_000), "variant": variant & ~labs.VARIANT_UNIFORM_CROSSOVER}
    if kind == "energy":
        with_C = rng.random() < 0.5
        return {"kind": kind, "N": rng.randint(16, 256), "B": _log_int(rng, 50, 200_000 if with_C else 1_000_000),
                "with_C": with_C}
    return {"kind": "skew_dev", "N": rng.randint(16, 160), "B": _log_int(rng, 50, 60_000)}


# ------------------------------------------------------------------ inputs


def _sequences(N, B, seed):
    """B uniformly random packed sequences on the GPU, bits >= N zero."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    W = (N + 63) // 64
    s = torch.randint(-(1 << 63), (1 << 63) - 1, (B, W), dtype=torch.int64, device=DEV, generator=g)
    tail = N - 64 * (W - 1)
    if tail < 64:
        s[:, W - 1] &= (1 << tail) - 1
    return s


def _params(case, **budget):
    policy = labs.REPLACE_WORST if case.get("worst") else labs.REPLACE_RANDOM
    return labs.make_params(case["N"], case["K"], replace_policy=policy, variant=case.get("variant", 0), **budget)


def _uneven(case, seed):
    """Instances as in the uneven batch: N and K uniform, budgets proportional to N^2."""
    rng = random.Random(seed)
    out = []
    for i in range(case["count"]):
        n = rng.randint(case["n_lo"], case["n_hi"])
        out.append(labs.make_instance(n, rng.randint(50, 200), seed=seed, instance=i,
                                      max_steps=case["steps_per_n2"] * n * n))
    return out


def _requests(case, seed):
    """Requests as in the Poisson stream: half run to a step cap, half stop early at a target
    (merit factor 5, which random restarts reach within a few searches)."""
    rng = random.Random(seed)
    out = []
    for i in range(case["count"]):
        n = rng.randint(case["n_lo"], case["n_hi"])
        target = int(n * n / 10) if rng.random() < 0.5 else -1
        out.append(labs.make_instance(n, 100, seed=seed, instance=i, max_steps=case["steps"], target_E=target))
    return out


def prepare(case, seed):
    k = case["kind"]
    st = {"case": case, "seed": seed}
    if k == "run":
        st["params"] = _params(case, max_generations=case["generations"])
    elif k == "launch":
        st["params"] = _params(case, max_steps=case["steps"])
        st["out"] = torch.zeros((case["replicas"], 8), dtype=torch.int64, device=DEV)
    elif k == "resume":
        st["slices"] = [_params(case, max_generations=g * case["generations"]) for g in (1, 2)]
        st["state"] = torch.zeros(case["replicas"] * labs.mts_state_bytes(case["N"], case["K"]), dtype=torch.uint8,
                                  device=DEV)
        st["out"] = torch.zeros((case["replicas"], 8), dtype=torch.int64, device=DEV)
    elif k == "batch":
        st["batch"] = labs.Batch(_uneven(case, seed))
    elif k == "serve":
        st["requests"] = _requests(case, seed)
        st["server"] = labs.Server(max_slots=256, max_N=160, max_K=100, quantum_steps=2000)
    else:
        st["seqs"] = _sequences(case["N"], case["B"], seed)
    return st


# ------------------------------------------------------------------ one pass


def _columns(results):
    """Host results (a list of dicts) as arrays; `seconds` is a time, not a result."""
    words = max(len(r["seq"]) for r in results)
    out = {key: np.array([r[key] for r in results]) for key in
           ("E", "F", "status", "generations", "steps", "flip_evals", "instance")}
    out["seq"] = np.array([r["seq"] + [0] * (words - len(r["seq"])) for r in results], dtype=np.uint64).view(np.int64)
    return out


def run(state):
    case, seed = state["case"], state["seed"]
    k = case["kind"]
    if k == "run":
        return _columns(labs.mts_run(state["params"], seed, 0, case["replicas"]))
    if k == "launch":
        return labs.mts_launch(state["params"], seed, 0, case["replicas"], out=state["out"])
    if k == "resume":
        for i, p in enumerate(state["slices"]):
            labs.mts_resume(p, seed, 0, case["replicas"], state["state"], resume=i > 0, out=state["out"])
        return state["out"], state["state"]
    if k == "batch":
        state["batch"].launch()
        return _columns(state["batch"].results())
    if k == "serve":
        srv = state["server"]
        tickets = [srv.submit(r) for r in state["requests"]]
        done = {}
        while len(done) < len(tickets):
            for t in tickets:
                if t not in done:
                    r = srv.poll(t)
                    if r is not None:
                        done[t] = r
            time.sleep(0.0002)
        return _columns([done[t] for t in tickets])
    if k == "tabu":
        r = labs.tabu_run(state["seqs"], case["N"], seed, variant=case["variant"])
        return r["best"], r["bestE"], r["steps"]
    if k == "energy":
        return labs.energy_batch(state["seqs"], case["N"], with_C=case["with_C"])
    return labs.skew_deviation_batch(state["seqs"], case["N"])


# ------------------------------------------------------------------ work of one pass


def _search_ops(moves, steps):
    """A tabu step cannot do without bringing each move's energy up to date (four terms), the
    tabu and the aspiration test and its place in the minimum: seven integer operations a move."""
    return 7.0 * moves * steps


def work(case):
    k = case["kind"]
    if k in ("run", "launch", "resume"):
        N, R = case["N"], case["replicas"]
        moves = (N + 1) // 2 if case.get("variant", 0) & labs.VARIANT_SKEW else N
        per = case["steps"] if k == "launch" else case["generations"] * moves * (2 if k == "resume" else 1)
        moved = 64 * R
        if k == "resume":  # results and records of two slices, the records read once in between
            moved = 2 * 64 * R + 3 * R * labs.mts_state_bytes(N, case["K"])
        return {"bytes": float(moved), "flops": _search_ops(moves, per) * R}
    if k == "batch":
        n = [x for x in range(case["n_lo"], case["n_hi"] + 1)]
        mean = sum(_search_ops(x, case["steps_per_n2"] * x * x) for x in n) / len(n)
        return {"bytes": 128.0 * case["count"], "flops": mean * case["count"]}
    if k == "serve":  # the capped half runs its whole budget
        n = (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": 128.0 * case["count"], "flops": _search_ops(n, case["steps"]) * case["count"] / 2}
    N, B = case["N"], case["B"]
    row = 8.0 * ((N + 63) // 64)
    if k == "tabu":
        moves = (N + 1) // 2 if case["variant"] & labs.VARIANT_SKEW else N
        return {"bytes": B * (2 * row + 12), "flops": _search_ops(moves, moves) * B}
    if k == "energy":
        # a shift, an exclusive or and a popcount for every 32 products, a multiply-add for each C_k
        return {"bytes": B * (row + 4 + (4.0 * (N - 1) if case["with_C"] else 0)),
                "flops": B * (3.0 * N * (N - 1) / 64 + 2 * (N - 1))}
    # every rotation, and for even N every deletion in it: one changed pair each
    return {"bytes": B * (row + 4), "flops": B * (float(N) * N if N % 2 == 0 else 3.0 * N * N / 64)}


# ------------------------------------------------------------------ 64-bit values


def _bits(seqs, N):
    j = torch.arange(N, device=seqs.device)
    return (seqs[:, j // 64] >> (j % 64)) & 1


def _exact_energy(seqs, N, with_C):
    E, C = [], []
    for part in seqs.split(200_000):
        s = (2 * _bits(part, N) - 1).to(torch.float32)  # sums of at most 256 products of +-1: exact
        c = torch.stack([(s[:, : N - k] * s[:, k:]).sum(1) for k in range(1, N)], dim=1).to(torch.int64)
        E.append((c * c).sum(1))
        if with_C:
            C.append(c)
    return (torch.cat(E), torch.cat(C)) if with_C else torch.cat(E)


def _exact_skew_dev(seqs, N):
    """Mismatches with skew symmetry of every rotation (odd N), and of every rotation with one
    element deleted (even N); the least of them."""
    b = _bits(seqs, N).to(torch.uint8).t().contiguous()  # (N, B)
    L = N if N % 2 else N - 1
    c = (L - 1) // 2
    odd = (torch.arange(1, c + 1, device=b.device) % 2).to(torch.uint8)[:, None]
    best = torch.full((b.shape[1],), N, dtype=torch.int64, device=b.device)
    for r in range(N):
        u = torch.roll(b, -r, 0)
        for d in range(N) if N % 2 == 0 else [None]:
            t = u if d is None else torch.cat([u[:d], u[d + 1:]])
            bad = (t[c + 1:] ^ t[:c].flip(0) ^ odd).sum(0, dtype=torch.int64)
            best = torch.minimum(best, bad)
    return best


def exact(case, seed):
    # A search's outputs are the records of a random walk: no formula gives them.
    if case["kind"] == "energy":
        return _exact_energy(_sequences(case["N"], case["B"], seed), case["N"], case["with_C"])
    if case["kind"] == "skew_dev" and (case["N"] ** 3) * case["B"] < 2e11:
        return _exact_skew_dev(_sequences(case["N"], case["B"], seed), case["N"])
    return None

"""The work that users of this package have it do, as cases that can be timed and compared.

A case names a synthetic problem (the generator's keys of `workloads.CONFIGS`) and a way of stepping it:

    run    the solver continues from a checkpoint for `rounds` rounds with one call of `run`
    round  the same with one call of `round` per round, for a program that looks at every round's block
    host   the same with `round_host`: the state lives in pinned host memory
    fit    a whole fit: a new handle, `rounds` rounds from beta = 0, the objective and the totals, close
    draw   one candidate draw by `sample_static`, which needs no handle

A checkpoint is the state after `done` rounds of the same problem: far enough into the run that coefficients already
chosen move again beside those never touched, not so far that nothing moves any more.
"""
from __future__ import annotations

import dataclasses
import math

import torch

from paper_1312_5766_b200 import binding, workloads as wl

ETA = 1e-6
DENSE_KINDS = ("dense_iid", "dense_grouped")


def _case(name, call, kind, n_rows, n_cols, n_candidates, n_keep, rounds, done=0, n_true=None, lam_frac=0.02, rho=0.1,
          nnz_col=0, schedulers=1, schedule="priority", loss="squared"):
    c = dict(call=call, kind=kind, n_rows=n_rows, n_cols=n_cols, n_candidates=n_candidates, n_keep=n_keep, rounds=rounds,
             done=done, n_true=n_true or max(1, n_cols // 100), lam_frac=lam_frac, rho=rho, nnz_col=nnz_col,
             schedulers=schedulers, schedule=schedule, loss=loss)
    return dict(c, name=name) if name else c


def _config(name, label, call, rounds, done=0, **kw):
    """A case on one of the benchmark configurations."""
    c = wl.CONFIGS[name]
    return _case(label, call, c["kind"], c["n_rows"], c["n_cols"], c["n_candidates"], c["n_keep"], rounds, done,
                 n_true=c["n_true"], lam_frac=c["lam_frac"], rho=c["rho"], nnz_col=c.get("nnz_col", 0), **kw)


def listed():
    return [
        # the draw alone, for a program with no handle of its own, at the size of the middle dense configuration
        _case("draw_100k", "draw", "dense_iid", 0, 100_000, 2_048, 1, 1),
        # a small problem stepped round by round, each round's block looked at
        _config("c1", "round_small_dense", "round", 8, done=200),
        # a small problem from start to end: one point of a comparison of schedules, or of a path over lambda
        _config("c1", "fit_small_dense", "fit", 1_000),
        # the ordinary dense problem, continued
        _config("c2", "run_dense", "run", 100, done=400),
        # ... with its state in host memory
        _config("c2", "host_dense", "host", 8, done=400),
        # the largest dense problem: groups of correlated columns
        _config("c3", "run_large_dense_grouped", "run", 100, done=400),
        # few samples and very many covariates, as in genome-wide association (463 x 508,999, correlated neighbours): with so
        # few rows every pair of columns correlates a little and the filter turns most candidates away
        _case("run_few_rows", "run", "dense_grouped", 463, 508_999, 1_024, 240, 50, done=200, n_true=5_000, lam_frac=0.05),
        # logistic loss, sizes that divide by nothing
        _case("run_logistic_ragged", "run", "dense_iid", 3_001, 50_021, 1_001, 121, 100, done=300, n_true=500, loss="logistic"),
        # the middle sparse problem: uniform rows, hardly a conflict
        _config("c4", "run_sparse", "run", 100, done=800),
        # ... by four scheduler threads taking turns
        _config("c4", "run_sparse_4_schedulers", "run", 128, done=768, schedulers=4),
        # the uniform schedule without priorities (the static scheduler of the comparisons) on a small sparse problem
        _case("run_small_sparse_static", "run", "csc_uniform", 5_000, 100_003, 819, 102, 100, done=200, n_true=500, lam_frac=0.01,
              nnz_col=50, schedule="static"),
        # the largest sparse problem: rows by Zipf's law, most candidates turned away
        _config("c5", "run_large_sparse_zipf", "run", 600, done=300),
    ]


def _log_int(rng, lo, hi):
    """A whole number between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["run", "run", "run", "run", "round", "host", "fit", "draw"])
    if call == "draw":
        n_cols = _log_int(rng, 5_000, 2_000_000)
        return _case(None, "draw", "dense_iid", 0, n_cols, _log_int(rng, 64, min(4_096, n_cols // 4)), 1, 1)
    kind = rng.choice(["dense_iid", "dense_grouped", "csc_uniform", "csc_zipf"])
    rounds = {"run": rng.randint(40, 120), "round": rng.randint(4, 12), "host": rng.randint(4, 12),
              "fit": rng.randint(50, 300)}[call]
    done = 0 if call == "fit" else rng.randint(100, 400)
    schedule = rng.choice(["priority", "priority", "priority", "abs", "dynamic", "static"])
    loss = "squared" if call == "host" else rng.choice(["squared", "squared", "logistic"])
    schedulers = rng.choice([1, 1, 2, 4]) if call == "run" else 1
    if kind in DENSE_KINDS:
        n_rows = _log_int(rng, 300, 20_000)
        n_cols = _log_int(rng, 5_000, min(500_000, 2_000_000_000 // n_rows))
        n_keep = _log_int(rng, 16, 512)
        nnz_col, rho = 0, 0.1
    else:
        nnz_col = rng.randint(10, 60)
        n_rows = _log_int(rng, 3_000, 1_000_000)
        n_cols = _log_int(rng, 20_000, 100_000_000 // nnz_col)
        n_keep = _log_int(rng, 32, 2_048)
        rho = 0.1 if kind == "csc_uniform" else 0.05
    most = min(_max_candidates(kind), n_cols // schedulers // 4)
    n_keep = min(n_keep, most)
    n_candidates = min(most, int(n_keep * rng.uniform(2.0, 9.0)))
    return _case(None, call, kind, n_rows, n_cols, max(n_candidates, n_keep), n_keep, rounds, done,
                 n_true=max(10, n_cols // 200), lam_frac=rng.choice([0.01, 0.02, 0.05]), rho=rho, nnz_col=nnz_col,
                 schedulers=schedulers, schedule=schedule, loss=loss)


def _max_candidates(kind):
    return 4_096 if kind in DENSE_KINDS else 16_384


SCHEDULES = {"priority": 0, "abs": binding.FLAG_ABS_WEIGHT, "dynamic": binding.FLAG_DYNAMIC_DEPS,
             "static": binding.FLAG_UNIFORM_DRAW}


def _flags(case):
    return SCHEDULES[case["schedule"]] | (binding.FLAG_LOGISTIC if case["loss"] == "logistic" else 0)


class _State:
    """What a program holds between calls: the problem on the device, the solver's handle, a checkpoint."""


def prepare(case, seed):
    s = _State()
    s.case, s.seed = case, seed
    if case["call"] == "draw":
        # priorities of a run under way: a third never updated (c_init), a third at rest, a third with small changes
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        n = case["n_cols"]
        which = torch.randint(0, 3, (n,), generator=g, device="cuda")
        change = torch.randn(n, generator=g, device="cuda").abs() * 1e-2
        s.delta = torch.where(which == 0, torch.full_like(change, 1e4), torch.where(which == 1, torch.zeros_like(change), change))
        s.cand = torch.empty(case["n_candidates"], dtype=torch.int32, device="cuda")
        return s
    keys = ["kind", "n_rows", "n_cols", "n_true", "lam_frac", "n_candidates", "n_keep", "rho"]
    cfg = {k: case[k] for k in keys}
    if case["kind"] in DENSE_KINDS:
        cfg["group"] = 20
    else:
        cfg["nnz_col"] = case["nnz_col"]
    s.problem = wl.make_problem(cfg, seed=seed, device="cuda", eta=ETA)
    if case["kind"] in DENSE_KINDS and case["n_rows"] % 4:            # dense columns start at multiples of 16 bytes
        s.problem = dataclasses.replace(s.problem, values=torch.nn.functional.pad(s.problem.values, (0, -case["n_rows"] % 4)))
    if case["loss"] == "logistic":
        s.problem = wl.to_logistic(s.problem, case["lam_frac"])
    if case["call"] == "fit":
        return s
    s.solver = binding.StradsLasso.from_problem(s.problem, flags=_flags(case), n_schedulers=case["schedulers"])
    s.solver.run(case["done"])
    live = [s.solver.beta, s.solver.resid, s.solver.delta]
    if case["loss"] == "logistic":
        live.append(s.solver.margin())
    if case["call"] == "host":
        s.live = [t.cpu().pin_memory() for t in live]
        s.block = [torch.zeros(case["n_keep"], dtype=torch.int32).pin_memory(), torch.zeros(case["n_keep"]).pin_memory(),
                   torch.zeros(4, dtype=torch.int32).pin_memory()]
    else:
        s.live = live
    s.checkpoint = [t.clone() for t in s.live]
    return s


def run(s):
    case = s.case
    if case["call"] == "draw":
        return binding.sample_static(s.delta, ETA, s.seed, 3, case["n_candidates"], out=s.cand)
    if case["call"] == "fit":
        solver = binding.StradsLasso.from_problem(s.problem, flags=_flags(case))
        solver.run(case["rounds"])
        out = {"objective": solver.objective(), "kept": solver.totals()["kept"], "beta": solver.beta, "resid": solver.resid,
               "delta": solver.delta}
        solver.close()
        return out
    for now, then in zip(s.live, s.checkpoint):
        now.copy_(then)
    s.solver.set_round(case["done"])
    if case["call"] == "run":
        s.solver.run(case["rounds"])
        return s.live
    if case["call"] == "host":
        for _ in range(case["rounds"]):
            s.solver.round_host(*s.live, *s.block)
        return s.live + s.block
    for _ in range(case["rounds"]):
        block = s.solver.round()
    return s.live + list(block)


def work(case):
    """Per round: the priorities, the columns of the candidates looked at (stored values; sparse ones with their rows), the
    residual read and written, the state of the coefficients updated; and the inner products of the pairs of kept columns.
    Where the filter turns most candidates away it looks at all of them."""
    J, N, K = case["n_cols"], case["n_rows"], case["n_candidates"]
    if case["call"] == "draw":
        return {"bytes": 4.0 * J + 4.0 * K, "flops": 0.0}
    dense = case["kind"] in DENSE_KINDS
    column = 4.0 * N if dense else 8.0 * case["nnz_col"]
    rejects = N < 1_000 if dense else case["kind"] == "csc_zipf"
    looked_at = K if rejects else case["n_keep"]
    owned = J / case["schedulers"]
    per_round = (0.0 if case["schedule"] == "static" else 4.0 * owned) + column * looked_at + 8.0 * N + 16.0 * case["n_keep"]
    flops = (float(N) * looked_at * (looked_at - 1) if dense else 0.0) + column / 2 * looked_at
    total = {"bytes": per_round * case["rounds"], "flops": flops * case["rounds"]}
    if case["call"] == "fit":
        total["bytes"] += column * J + 12.0 * J
    if case["call"] == "host":
        total["bytes"] += 2 * 4.0 * (2 * J + N) * case["rounds"]
    return total


def tolerance(case):
    # whole numbers (candidates, kept lists, counts) are the same; the state is binary32, from sums in binary64
    return "exact" if case["call"] == "draw" else {"rel": 1e-5}

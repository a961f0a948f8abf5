"""CSC rounds by squads of CTAs (csrc/squads.cu: several schedulers, or the static schedule) against the same rounds one by one, bit for
bit, at the sizes where they can go wrong.  Single rounds are checked against the oracle in test_gpu_schedulers.py and test_gpu_engine.py."""
import pytest
import torch

from paper_1312_5766_b200 import workloads as wl

pytestmark = pytest.mark.gpu

UNIFORM, NO_FILTER, ABS, DYNAMIC, LOGISTIC = 1, 2, 32, 64, 128
CASES = {
    # the static schedule: windows that do; that do not; kept lists without a filter; more kept than a draw ahead takes
    "static": dict(kind="csc_uniform", n_rows=3000, n_cols=9001, n_candidates=900, n_keep=130, rho=0.1, nnz_col=33, flags=UNIFORM),
    "static_on_demand": dict(kind="csc_zipf", n_rows=5000, n_cols=20000, n_candidates=1500, n_keep=300, rho=0.05, nnz_col=20, flags=UNIFORM),
    "random": dict(kind="csc_uniform", n_rows=3000, n_cols=9001, n_candidates=200, n_keep=130, rho=0.1, nnz_col=33, flags=UNIFORM | NO_FILTER),
    "static_logistic": dict(kind="csc_uniform", n_rows=3000, n_cols=9001, n_candidates=300, n_keep=60, rho=0.1, nnz_col=33, flags=UNIFORM | LOGISTIC),
    "static_no_draw_ahead": dict(kind="csc_uniform", n_rows=60000, n_cols=12000, n_candidates=5000, n_keep=4200, rho=0.1, nnz_col=8, flags=UNIFORM),
    # few coefficients: the lists of several blocks under way share most of them; all of them in every list
    "static_few": dict(kind="csc_uniform", n_rows=2000, n_cols=150, n_candidates=100, n_keep=90, rho=0.2, nnz_col=12, flags=UNIFORM),
    "static_all": dict(kind="csc_uniform", n_rows=2000, n_cols=150, n_candidates=150, n_keep=150, rho=0.2, nnz_col=12, flags=UNIFORM),
    # schedulers: shares that divide unevenly, down to all of a share; buckets that overflow; dependencies dropped; the printed weight
    "two": dict(kind="csc_uniform", n_rows=3000, n_cols=9001, n_candidates=900, n_keep=130, rho=0.1, nnz_col=33, S=2),
    "three": dict(kind="csc_uniform", n_rows=1500, n_cols=9001, n_candidates=900, n_keep=130, rho=0.1, nnz_col=40, S=3, flags=ABS),
    "share": dict(kind="csc_uniform", n_rows=3000, n_cols=1003, n_candidates=200, n_keep=150, rho=0.1, nnz_col=13, S=5),
    "dynamic": dict(kind="csc_zipf", n_rows=5000, n_cols=20000, n_candidates=1500, n_keep=200, rho=0.05, nnz_col=20, S=4, flags=DYNAMIC),
    "logistic": dict(kind="csc_uniform", n_rows=3000, n_cols=9001, n_candidates=300, n_keep=60, rho=0.1, nnz_col=33, S=4, flags=LOGISTIC),
    "no_filter": dict(kind="csc_uniform", n_rows=3000, n_cols=9001, n_candidates=300, n_keep=60, rho=0.1, nnz_col=33, S=4, flags=NO_FILTER),
    # a warp's kept columns: more entries than it holds in shared memory, at once and each; more of them than it has lanes
    "held": dict(kind="csc_uniform", n_rows=200000, n_cols=20000, n_candidates=2000, n_keep=1900, rho=0.3, nnz_col=150, S=8),
    "long": dict(kind="csc_uniform", n_rows=50000, n_cols=3000, n_candidates=300, n_keep=200, rho=0.3, nnz_col=600, S=7),
    "many_kept": dict(kind="csc_uniform", n_rows=500000, n_cols=131500, n_candidates=16000, n_keep=15000, rho=0.4, nnz_col=4, S=8),
    "most_kept": dict(kind="csc_uniform", n_rows=500000, n_cols=100500, n_candidates=12500, n_keep=11900, rho=0.4, nnz_col=4, S=8),
    # the walk over all candidates by few CTAs: more candidates and entries than a CTA holds
    "on_demand_turns": dict(kind="csc_zipf", n_rows=30000, n_cols=140000, n_candidates=16384, n_keep=400, rho=0.05, nnz_col=21, S=8),
    "on_demand_entries": dict(kind="csc_zipf", n_rows=30000, n_cols=40000, n_candidates=9500, n_keep=700, rho=0.05, nnz_col=63, S=4),
}


def _solver(b, p, case):
    return b.StradsLasso.from_problem(p, device="cuda", flags=case.get("flags", 0), n_schedulers=case.get("S", 1))


def _problem(case, seed):
    cfg = {k: v for k, v in case.items() if k not in ("flags", "S")}
    p = wl.make_problem(dict(cfg, n_true=30, lam_frac=0.02), seed=seed)
    return wl.to_logistic(p, 0.02) if case.get("flags", 0) & LOGISTIC else p


def _same(a, b):
    for x, y in ((a.beta, b.beta), (a.resid, b.resid), (a.delta, b.delta)):
        assert torch.equal(x, y)
    assert a.totals() == b.totals() and a.get_round() == b.get_round()


@pytest.mark.parametrize("name", list(CASES))
def test_runs_equal_rounds(name):
    from paper_1312_5766_b200 import binding as b
    case = CASES[name]
    p = _problem(case, 3)
    a, one = _solver(b, p, case), _solver(b, p, case)
    calls = [3, 21, 1, 70, 8]                              # squads without a round, launches one behind the other, lists in place and not
    for n in calls:
        a.run(n)
    for _ in range(sum(calls)):
        one.round()
    _same(a, one)
    a.round(); a.run(19)                                   # lists drawn ahead are forgotten
    one.run(13)
    for _ in range(7):
        one.round()
    _same(a, one)
    again = _solver(b, p, case)                            # resumed from the middle of a cycle
    for x, y in ((again.beta, a.beta), (again.resid, a.resid), (again.delta, a.delta)):
        x.copy_(y)
    if case.get("flags", 0) & LOGISTIC:
        again.margin().copy_(a.margin())
    again.set_round(a.get_round())
    again.run(17); a.run(9); a.run(8)
    assert all(torch.equal(x, y) for x, y in ((again.beta, a.beta), (again.resid, a.resid), (again.delta, a.delta)))
    assert a.status()[0] == 0 and one.status()[0] == 0


@pytest.mark.parametrize("name", ["static", "three"])
def test_a_squad_gives_up_and_the_handle_recovers(name):
    """The barrier of the squad on turn gives up; the others wait for its turn to pass, in vain, within the same limit."""
    from paper_1312_5766_b200 import binding as b
    case = CASES[name]
    p = _problem(case, 4)
    ref, s = _solver(b, p, case), _solver(b, p, case)
    saved = [t.clone() for t in (s.beta, s.resid, s.delta)]
    s.set_wait_limit(4096)
    s.inject_stall(b.STALL_WALK_BARRIER)
    s.run(24)
    assert s.status()[0] == -6 and s.status()[1] & 4
    s.run(24)                                              # nothing runs, and the launch ends
    assert s.status()[0] == -6
    for t, c in zip((s.beta, s.resid, s.delta), saved):
        t.copy_(c)
    s.recover()
    s.set_round(0)
    s.set_wait_limit(0)
    s.run(50); ref.run(50)
    assert all(torch.equal(x, y) for x, y in ((s.beta, ref.beta), (s.resid, ref.resid), (s.delta, ref.delta)))
    assert s.status()[0] == 0

"""Whole rounds in one launch (csrc/engine.cu) at the sizes where it can go wrong: every round teacher-forced against the
oracle, then the same rounds through strads_run (candidates drawn one round ahead) against strads_round bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from helpers import oracle_matrix
from paper_1312_5766_b200 import workloads as wl
from test_gpu_parity import HALF_ULP32, RTOL_DBETA, _assert_kept_matches

pytestmark = pytest.mark.gpu

CASES = {
    # dense: one row group and tile; just past a tile of rows, of columns and of K; several pieces of the walk; P' = P = J
    "one_tile": dict(kind="dense_iid", n_rows=24, n_cols=600, n_true=5, n_candidates=64, n_keep=64, rho=0.5),
    "tile_edges": dict(kind="dense_iid", n_rows=65, n_cols=900, n_true=5, n_candidates=129, n_keep=40, rho=0.3),
    "two_windows": dict(kind="dense_iid", n_rows=257, n_cols=3000, n_true=9, n_candidates=1000, n_keep=120, rho=0.15),
    "walk_in_pieces": dict(kind="dense_grouped", n_rows=401, n_cols=6000, n_true=9, n_candidates=2500, n_keep=300, rho=0.1),
    "longest_columns": dict(kind="dense_iid", n_rows=2048, n_cols=1500, n_true=9, n_candidates=700, n_keep=100, rho=0.06),
    "everything": dict(kind="dense_iid", n_rows=100, n_cols=300, n_true=5, n_candidates=300, n_keep=300, rho=0.2),
    # CSC: buckets that hold; that overflow now and then; columns longer than a warp's two turns; P too large to draw ahead
    "buckets": dict(kind="csc_uniform", n_rows=3000, n_cols=9000, n_true=50, n_candidates=900, n_keep=130, rho=0.1, nnz_col=33),
    "full_buckets": dict(kind="csc_uniform", n_rows=1500, n_cols=9000, n_true=50, n_candidates=900, n_keep=130, rho=0.1, nnz_col=40),
    "long_columns": dict(kind="csc_uniform", n_rows=20000, n_cols=2000, n_true=20, n_candidates=300, n_keep=60, rho=0.1, nnz_col=150),
    "no_draw_ahead": dict(kind="csc_uniform", n_rows=60000, n_cols=12000, n_true=50, n_candidates=5000, n_keep=4200, rho=0.1, nnz_col=8),
    "on_demand": dict(kind="csc_zipf", n_rows=20000, n_cols=50000, n_true=50, n_candidates=3000, n_keep=500, rho=0.05, nnz_col=21),
    # walks on demand that stop at P in a batch, and among the last survivors; with columns longer than the table of rows takes;
    # with more entries than a CTA holds; with few survivors from the start
    "demand_stops_early": dict(kind="csc_zipf", n_rows=20000, n_cols=50000, n_true=50, n_candidates=3001, n_keep=9, rho=0.05, nnz_col=21),
    "demand_stops_late": dict(kind="csc_zipf", n_rows=20000, n_cols=50000, n_true=50, n_candidates=2999, n_keep=33, rho=0.05, nnz_col=21),
    "demand_long_columns": dict(kind="csc_zipf", n_rows=4000, n_cols=9000, n_true=50, n_candidates=1500, n_keep=300, rho=0.05, nnz_col=90),
    "demand_many_entries": dict(kind="csc_zipf", n_rows=30000, n_cols=40000, n_true=50, n_candidates=9500, n_keep=900, rho=0.05, nnz_col=63),
    "demand_few": dict(kind="csc_zipf", n_rows=3000, n_cols=2000, n_true=50, n_candidates=70, n_keep=60, rho=0.05, nnz_col=30),
}


@pytest.mark.parametrize("name", list(CASES))
def test_rounds(name):
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(CASES[name], lam_frac=0.02, group=20), seed=3)
    if p.layout == wl.DENSE and p.n_rows % 4:
        pad = torch.full((p.n_cols, (p.n_rows + 3) // 4 * 4), float("nan"))        # nothing may leak in from the padding
        pad[:, : p.n_rows] = p.values
        p.values = pad
    X = oracle_matrix(p)
    n2, beta, resid, delta = oracle.init(X, p.y.numpy(), 1e4)
    lam, eta, rho = float(np.float32(p.lam)), float(np.float32(p.eta)), float(np.float32(p.rho))
    s, ahead = (b.StradsLasso.from_problem(p, device="cuda") for _ in range(2))
    n = 14
    for t in range(n):
        beta[:] = s.beta.cpu().numpy(); resid[:] = s.resid.cpu().numpy(); delta[:] = s.delta.cpu().numpy()
        cand, kept, dbeta, counts = (x.cpu().numpy() for x in s.round())
        nk = int(counts[2])
        assert np.array_equal(cand, oracle.sample(delta, eta, p.seed, t, p.n_candidates)), t
        _assert_kept_matches(X, n2, cand, p.n_keep, rho, kept[:nk], int(counts[1]))
        assert np.all(kept[nk:] == -1)
        want = oracle.update(X, n2, lam, kept[:nk], beta, resid, delta)
        assert np.all(np.abs(dbeta[:nk] - want) <= RTOL_DBETA * np.abs(want) + HALF_ULP32 * np.abs(beta[kept[:nk]])), t
    s.run(40)
    for k in (1, 33, 20):                                   # launches of different lengths, lists in place and not
        ahead.run(k)
    for _ in range(n + 40 - 54):
        ahead.round()
    for x, y in ((s.beta, ahead.beta), (s.resid, ahead.resid), (s.delta, ahead.delta)):
        assert torch.equal(x, y)
    assert s.totals() == ahead.totals() and s.status()[0] == 0


def test_products_that_cluster_at_rho():
    """Columns of +-1 over a few rows: a third of all pairs correlate at exactly rho, more than any list of open pairs holds."""
    from paper_1312_5766_b200 import binding as b
    N, J, P = 20, 2000, 60
    g = torch.Generator().manual_seed(2)
    x = (torch.randint(0, 2, (J, N), generator=g) * 2 - 1).float()
    y = torch.randn(N, generator=g)
    X = oracle.Matrix.dense(x.numpy())
    n2 = oracle.colnorm2(X)
    rho = float(np.float32(0.2))                            # products are even integers: |corr| = 0.2 exactly is |product| = 4
    s = b.StradsLasso(wl.DENSE, N, J, x.cuda(), y.cuda(), 0.1, 1e-6, rho, J, P, seed=1)
    for _ in range(3):
        cand, kept, _, counts = (v.cpu().numpy() for v in s.round())
        _assert_kept_matches(X, n2, cand, P, rho, kept[: int(counts[2])], int(counts[1]))
    assert s.status() == (0, 8)                             # informational: pairs decided one by one


# one tile of all pairs and more; rows that end inside a group of four and of 32, with columns padded by NaN
@pytest.mark.parametrize("N,J,product", [(70, 1900, 4), (33, 1601, 3), (97, 2177, 5)])
def test_all_pairs_exactly(N, J, product):
    """Columns of +-1 over a few rows: more pairs correlate at exactly rho than any list of open pairs holds."""
    from paper_1312_5766_b200 import binding as b
    P = 60
    g = torch.Generator().manual_seed(2)
    x = torch.full((J, (N + 3) // 4 * 4), float("nan"))
    x[:, :N] = (torch.randint(0, 2, (J, N), generator=g) * 2 - 1).float()
    y = torch.randn(N, generator=g)
    X = oracle.Matrix.dense(x.numpy(), n_rows=N)
    n2 = oracle.colnorm2(X)
    rho = float(np.float32(product / N))                    # products are whole numbers of N's parity
    s = b.StradsLasso(wl.DENSE, N, J, x.cuda(), y.cuda(), 0.1, 1e-6, rho, J, P, seed=1)
    for _ in range(3):
        cand, kept, _, counts = (v.cpu().numpy() for v in s.round())
        _assert_kept_matches(X, n2, cand, P, rho, kept[: int(counts[2])], int(counts[1]))
    assert s.status() == (0, 8)                             # informational: pairs decided one by one


def test_tied_keys():
    """Infinite priorities: thousands of race times of exactly 0, far more than the draw's boundary holds."""
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(kind="csc_uniform", n_rows=3000, n_cols=60000, n_true=20, lam_frac=0.02, n_candidates=700, n_keep=100,
                             rho=0.1, nnz_col=10), seed=4)
    s = b.StradsLasso.from_problem(p, device="cuda")
    s.delta[500:40000] = float("inf")
    for t in range(3):
        delta = s.delta.cpu().numpy().astype(np.float64)
        cand = s.round()[0].cpu().numpy()
        assert np.array_equal(cand, oracle.sample(delta, float(np.float32(p.eta)), p.seed, t, p.n_candidates))
    s.run(5)
    delta = s.delta.cpu().numpy().astype(np.float64)
    assert np.array_equal(s.round()[0].cpu().numpy(), oracle.sample(delta, float(np.float32(p.eta)), p.seed, 8, p.n_candidates))


# rows in the buckets on average 6.4 of 16 (every other round overflows one) and 10 (every attempt does)
@pytest.mark.parametrize("nnz_col", [25, 40])
def test_round_index_set_back_while_the_buckets_rest(nnz_col):
    """After an overflow the row buckets rest for a number of rounds; going back to an earlier round in that time changes nothing."""
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(CASES["full_buckets"], lam_frac=0.02, nnz_col=nnz_col), seed=5)
    s, fresh = (b.StradsLasso.from_problem(p, device="cuda") for _ in range(2))
    s.run(3)
    start = [t.clone() for t in (s.beta, s.resid, s.delta)]
    want = [[t.clone() for t in s.round()] for _ in range(12)]
    end = [t.clone() for t in (s.beta, s.resid, s.delta)]
    for first in (1, 2, 5, 12):                             # rounds gone before the next return
        for t, c in zip((s.beta, s.resid, s.delta), start):
            t.copy_(c)
        s.set_round(3)
        for i in range(first):
            for x, y in zip(s.round(), want[i]):
                assert torch.equal(x, y), (first, i)
    for x, y in zip((s.beta, s.resid, s.delta), end):
        assert torch.equal(x, y)
    fresh.run(15)
    for x, y in zip((fresh.beta, fresh.resid, fresh.delta), end):
        assert torch.equal(x, y)


MENDED = {
    # the untouched coefficients run out: the cutoff carried over is far too low for the draw of the next round
    "dense": dict(kind="dense_iid", n_rows=64, n_cols=1201, n_true=9, n_candidates=300, n_keep=90, rho=0.37),
    "csc": dict(kind="csc_uniform", n_rows=5000, n_cols=3003, n_true=9, n_candidates=500, n_keep=130, rho=0.1, nnz_col=20),
    "few": dict(kind="csc_uniform", n_rows=5000, n_cols=603, n_true=9, n_candidates=40, n_keep=30, rho=0.1, nnz_col=20),
}


@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("name", list(MENDED))
def test_launches_that_end_in_a_mended_draw(name, tied):
    """The draw for the round behind a launch's last one selected anew (too few keys below the cutoff, or -- tied -- more equal
    keys than there is room for): the next launch finds histogram and cursors as it expects them."""
    from paper_1312_5766_b200 import binding as b
    cfg = dict(MENDED[name], lam_frac=0.02)
    if tied:
        cfg.update(n_cols=30_000)
    p = wl.make_problem(cfg, seed=6)
    s, ahead = (b.StradsLasso.from_problem(p, device="cuda") for _ in range(2))
    eta, n = float(np.float32(p.eta)), 24
    if tied:
        for h in (s, ahead):
            h.delta[2_000:25_000] = float("inf")
            h.set_round(0)
    for t in range(n):
        delta = s.delta.cpu().numpy().astype(np.float64)
        assert np.array_equal(s.round()[0].cpu().numpy(), oracle.sample(delta, eta, p.seed, t, p.n_candidates)), t
        ahead.run(1)                                        # a launch per round, each with the draw of the next
        for x, y in ((s.beta, ahead.beta), (s.resid, ahead.resid), (s.delta, ahead.delta)):
            assert torch.equal(x, y), t
    ahead.run(7)
    for _ in range(7):
        s.round()
    for x, y in ((s.beta, ahead.beta), (s.resid, ahead.resid), (s.delta, ahead.delta)):
        assert torch.equal(x, y)
    assert (s.status()[1] & 1) == (1 if tied else 0)        # ties: the boundary was cut further


def _csc(lengths, n_rows, value, seed):
    """Columns of these lengths, rows uniform; value(generator, n): their entries."""
    g = torch.Generator().manual_seed(seed)
    ptr = torch.cat([torch.zeros(1, dtype=torch.int64), torch.cumsum(lengths, 0)])
    rows = torch.cat([torch.randperm(n_rows, generator=g)[:n].sort().values for n in lengths.tolist()]).to(torch.int32)
    return value(g, int(ptr[-1])), rows, ptr, torch.randn(n_rows, generator=g)


# products that are zero again and again (values of +-1, one in eight of the stored ones 0), by buckets and by the walk over all candidates;
# columns of 4 to 400 entries: more than the table of rows takes, and other than the mean says of the last survivors; windows with more
# candidates than a warp has places for, each with few of them and with more than it can list
@pytest.mark.parametrize("name,n_rows,n_candidates,n_keep,rho", [("cancel", 3000, 900, 130, 0.1), ("cancel", 700, 800, 300, 0.2), ("uneven", 700, 1500, 300, 0.1),
                                                                 ("uneven", 60000, 1700, 1000, 0.02), ("cancel", 20000, 2000, 1300, 0.1), ("many_met", 70000, 2000, 1300, 0.3)])
def test_rounds_on_unusual_columns(name, n_rows, n_candidates, n_keep, rho):
    from paper_1312_5766_b200 import binding as b
    J = 8000
    if name == "many_met":
        lengths, value = torch.full((J,), 150, dtype=torch.int64), lambda g, n: torch.randn(n, generator=g)
    elif name == "cancel":
        lengths = torch.full((J,), 33, dtype=torch.int64)
        value = lambda g, n: ((torch.randint(0, 2, (n,), generator=g) * 2 - 1) * (torch.randint(0, 8, (n,), generator=g) > 0)).float()
    else:
        lengths = (400.0 * (torch.arange(J) + 1.0) ** -0.5).long()[torch.randperm(J, generator=torch.Generator().manual_seed(1))]
        value = lambda g, n: torch.randn(n, generator=g)
    values, rows, ptr, y = _csc(lengths, n_rows, value, 7)
    X = oracle.Matrix.csc(n_rows, J, values.numpy(), rows.numpy(), ptr.numpy())
    n2 = oracle.colnorm2(X)
    args = (wl.CSC, n_rows, J, values.cuda(), y.cuda(), 0.05, 1e-6, rho, n_candidates, n_keep)
    kw = dict(seed=2, row_idx=rows.cuda(), col_ptr=ptr.cuda())
    s, ahead = b.StradsLasso(*args, **kw), b.StradsLasso(*args, **kw)
    for t in range(10):
        delta = s.delta.cpu().numpy().astype(np.float64)
        cand, kept, _, counts = (x.cpu().numpy() for x in s.round())
        assert np.array_equal(cand, oracle.sample(delta, float(np.float32(1e-6)), 2, t, n_candidates)), t
        _assert_kept_matches(X, n2, cand, n_keep, float(np.float32(rho)), kept[: int(counts[2])], int(counts[1]))
    ahead.run(10)
    four, one = (b.StradsLasso(*args, n_schedulers=4, **kw) for _ in range(2))
    four.run(10)
    for _ in range(10):
        one.round()
    for u, v in ((s, ahead), (four, one)):
        assert all(torch.equal(x, y) for x, y in ((u.beta, v.beta), (u.resid, v.resid), (u.delta, v.delta)))
        assert u.status()[0] == 0 and v.status()[0] == 0

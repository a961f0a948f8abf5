"""The whole candidate list in one screen whose last CTA walks (csrc/gram_dense_tc.cu, no candidate window): open pairs decided
by the CTAs that found them, by the recheck kernel behind, and by the 3xTF32 kernel when even the list overflows."""
import numpy as np
import pytest
import torch

import oracle
from helpers import oracle_matrix
from paper_1312_5766_b200 import workloads as wl
from test_gpu_parity import _assert_kept_matches

pytestmark = pytest.mark.gpu


# one tile and one K split short of two; a few dozen open pairs per round; more than one CTA keeps; P' = P
@pytest.mark.parametrize("n_rows,n_candidates,n_keep,rho", [(2052, 128, 128, 0.07), (3000, 200, 100, 0.06), (2500, 700, 320, 0.05), (2048 + 64, 129, 60, 0.07)])
def test_open_pairs(n_rows, n_candidates, n_keep, rho):
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(kind="dense_iid", n_rows=n_rows, n_cols=2500, n_true=20, lam_frac=0.02, n_candidates=n_candidates, n_keep=n_keep, rho=rho), seed=8)
    X = oracle_matrix(p)
    n2 = oracle.colnorm2(X)
    s, ahead = (b.StradsLasso.from_problem(p, device="cuda") for _ in range(2))
    for _ in range(8):
        cand, kept, _, counts = (v.cpu().numpy() for v in s.round())
        _assert_kept_matches(X, n2, cand, n_keep, float(np.float32(rho)), kept[: int(counts[2])], int(counts[1]))
    ahead.run(8)
    for x, y in ((s.beta, ahead.beta), (s.resid, ahead.resid), (s.delta, ahead.delta)):
        assert torch.equal(x, y)
    assert s.status()[0] == 0


# long columns: a few turns of every CTA; more pairs than the CTAs decide themselves; the shortest; rows that end inside a
# group of four, just behind and just before whole trips
@pytest.mark.parametrize("n_rows,rho", [(20_004, 0.024), (20_004, 0.012), (4096, 0.05), (4097, 0.05), (5119, 0.045), (5123, 0.045)])
def test_open_pairs_of_long_columns(n_rows, rho):
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(kind="dense_iid", n_rows=n_rows, n_cols=700, n_true=20, lam_frac=0.02, n_candidates=161, n_keep=90, rho=rho), seed=9)
    if n_rows % 4:
        pad = torch.full((p.n_cols, (n_rows + 3) // 4 * 4), float("nan"))          # nothing may leak in from the padding
        pad[:, :n_rows] = p.values
        p.values = pad
    X = oracle_matrix(p)
    n2 = oracle.colnorm2(X)
    s, ahead = (b.StradsLasso.from_problem(p, device="cuda") for _ in range(2))
    for _ in range(4):
        cand, kept, _, counts = (v.cpu().numpy() for v in s.round())
        _assert_kept_matches(X, n2, cand, 90, float(np.float32(rho)), kept[: int(counts[2])], int(counts[1]))
    ahead.run(4)
    for x, y in ((s.beta, ahead.beta), (s.resid, ahead.resid), (s.delta, ahead.delta)):
        assert torch.equal(x, y)
    assert s.status()[0] == 0


@pytest.mark.parametrize("n_candidates,bits", [(300, 0), (1600, 8)])
def test_products_that_cluster_at_rho(n_candidates, bits):
    """Columns of +-1 over a few rows: a third of all pairs correlate at exactly rho.  Two schedulers: not whole rounds in one launch."""
    from paper_1312_5766_b200 import binding as b
    N, J, P = 20, 3400, 60
    P = max(P, n_candidates // 2)                           # no window
    g = torch.Generator().manual_seed(2)
    x = (torch.randint(0, 2, (J, N), generator=g) * 2 - 1).float()
    X = oracle.Matrix.dense(x.numpy())
    n2 = oracle.colnorm2(X)
    rho = float(np.float32(0.2))                            # products are even integers: |corr| = 0.2 exactly is |product| = 4
    s = b.StradsLasso(wl.DENSE, N, J, x.cuda(), torch.randn(N, generator=g).cuda(), 0.1, 1e-6, rho, n_candidates, P, seed=1, n_schedulers=2)
    for _ in range(3):
        cand, kept, _, counts = (v.cpu().numpy() for v in s.round())
        _assert_kept_matches(X, n2, cand, P, rho, kept[: int(counts[2])], int(counts[1]))
    assert s.status() == (0, bits)                          # informational: pairs decided by the fallback

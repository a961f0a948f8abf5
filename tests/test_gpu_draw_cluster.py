"""Draws of rounds made launch by launch (csrc/draw_cluster.cu up to 2^19 coefficients, csrc/sampler.cu beyond) against ranking all keys: with the
cutoff of the draw before good, far too low, far too high or absent, and with times that tie."""
import numpy as np
import pytest
import torch

import oracle
from paper_1312_5766_b200 import workloads as wl

pytestmark = pytest.mark.gpu


# all there are; a list longer than a share leaves over; keys that end inside a group of four; the largest list; both sides of the line;
# schedulers that own two of four coefficients, one, and one in more than four
@pytest.mark.parametrize("J,n_cand,S,weight", [(37, 37, 1, "square"), (8191, 4096, 1, "square"), (50_021, 1001, 1, "abs"), (99_998, 16384, 1, "square"),
                                               (2 ** 19, 2048, 1, "square"), (2 ** 19 + 1, 2048, 1, "square"), (9002, 3000, 2, "square"),
                                               (9001, 3000, 3, "square"), (100_003, 819, 4, "square"), (65, 13, 5, "square")])
def test_draws(J, n_cand, S, weight):
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(kind="csc_uniform", n_rows=200, n_cols=J, n_true=1, lam_frac=0.1, nnz_col=2, n_candidates=n_cand, n_keep=1, rho=0.1), seed=6)
    s = b.StradsLasso.from_problem(p, device="cuda", n_schedulers=S, flags=b.FLAG_ABS_WEIGHT if weight == "abs" else 0)
    rng = np.random.default_rng(4)
    base = np.abs(rng.normal(size=J)).astype(np.float32)
    ties = np.where(rng.random(J) < 0.9, np.inf, base).astype(np.float32)              # times of exactly 0, more than a boundary holds
    steps = [None, None, base * np.float32(1e-3), base, np.where(rng.random(J) < 0.99, 0, base).astype(np.float32), ties, base, None]
    eta = float(np.float32(p.eta))
    for t, delta in enumerate(steps):
        if delta is not None:
            s.delta.copy_(torch.from_numpy(delta))
        for i in range(S):                                 # every scheduler's draw
            s.set_round(t * S + i)
            got, d = s.sample().cpu().numpy(), s.delta.cpu().numpy().astype(np.float64)
            if S > 1:
                want = oracle.sample_part(d, eta, p.seed, t * S + i, S, i, n_cand)
            else:
                want = oracle.sample(d, eta, p.seed, t, n_cand, weight=weight)
            assert np.array_equal(got, want), (t, i)
    assert s.status()[0] == 0

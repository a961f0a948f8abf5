"""Handles one after another, and several at a time from several threads: the streams, events and captured sequences that
a destroyed handle leaves to the next one must not leak anything of it."""
import threading

import pytest
import torch

from paper_1312_5766_b200 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = {"window": dict(kind="dense_iid", n_rows=1200, n_cols=3000, n_true=30, lam_frac=0.05, n_candidates=512, n_keep=48, rho=0.1),
          "no_window": dict(kind="dense_iid", n_rows=1000, n_cols=2000, n_true=30, lam_frac=0.05, n_candidates=200, n_keep=48, rho=0.1)}


def _fit(b, p, rounds, **kw):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        s = b.StradsLasso.from_problem(p, device="cuda", stream=stream, **kw)
        for n in rounds:
            s.run(n)
        out = (s.beta.clone(), s.resid.clone(), s.delta.clone())
        stream.synchronize()
        s.close()
    return out


@pytest.mark.parametrize("kw", [dict(), dict(n_schedulers=4)])
def test_handles_in_turn_and_side_by_side(kw):
    from paper_1312_5766_b200 import binding as b
    problems = [wl.make_problem(SHAPES[name], seed=seed, device="cuda") for name in SHAPES for seed in (1, 2)]
    rounds = (23, 23, 23, 70)                              # every length of captured sequence, left-overs launched one by one first
    b.load().strads_release_cached()
    want = []
    for p in problems:
        s = b.StradsLasso.from_problem(p, device="cuda", **kw)
        for _ in range(sum(rounds)):
            s.round()
        want.append((s.beta.clone(), s.resid.clone(), s.delta.clone()))
        s.close()
    for order in ([0, 1, 2, 3], [1, 0, 3, 2, 0, 2]):       # same shape again, and shapes that take turns
        for i in order:
            for x, y in zip(_fit(b, problems[i], rounds, **kw), want[i]):
                assert torch.equal(x, y), i
    torch.cuda.synchronize()
    got, failed = {}, []

    def work(i):
        try:
            torch.cuda.set_device(0)
            got[i] = [_fit(b, problems[i % 4], rounds, **kw) for _ in range(2)]
        except Exception as e:                             # pragma: no cover
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for i, outs in got.items():
        for out in outs:
            for x, y in zip(out, want[i % 4]):
                assert torch.equal(x, y), i
    assert b.load().strads_release_cached() == 0

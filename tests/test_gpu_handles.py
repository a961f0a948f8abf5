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


# (more rows: columns too long for rounds in one launch)
@pytest.mark.parametrize("kw,more_rows", [(dict(), 0), (dict(), 1200), (dict(n_schedulers=4), 0)])
def test_handles_in_turn_and_side_by_side(kw, more_rows):
    from paper_1312_5766_b200 import binding as b
    problems = [wl.make_problem(dict(SHAPES[name], n_rows=SHAPES[name]["n_rows"] + more_rows), seed=seed, device="cuda") for name in SHAPES for seed in (1, 2)]
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


def test_dense_rounds_in_one_launch_beyond_the_first_line():
    """1,200 rows, rho = 0.1 (N rho^2 = 12): with room for its buffers rounds go in one launch, without it by the launch chain; the
    same blocks, and the same state up to the order of the dense products (each good to 2^-44 of its terms, then rounded to binary32)."""
    import ctypes as C
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(SHAPES["window"], seed=7, device="cuda")
    s = b.StradsLasso.from_problem(p, device="cuda")
    lib, cfg = b.load(), b.Config()
    C.memmove(C.byref(cfg), C.byref(s._cfg), C.sizeof(cfg))
    need = C.c_size_t(0)
    assert lib.strads_workspace_bytes(C.byref(cfg), C.byref(need)) == 0 and need.value + (12 << 20) < s.workspace.numel()
    ws = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    beta, resid, delta = torch.zeros_like(s.beta), torch.empty_like(s.resid), torch.empty_like(s.delta)
    cfg.workspace, cfg.workspace_bytes = ws.data_ptr(), need.value
    cfg.beta, cfg.resid, cfg.delta = beta.data_ptr(), resid.data_ptr(), delta.data_ptr()
    h = C.c_void_p(None)
    assert lib.strads_lasso_init(C.byref(cfg), C.byref(h)) == 0
    cand, kept = torch.empty(p.n_candidates, dtype=torch.int32, device="cuda"), torch.empty(p.n_keep, dtype=torch.int32, device="cuda")
    out = b.RoundOut()
    out.cand, out.kept = cand.data_ptr(), kept.data_ptr()
    for t in range(200):
        assert lib.strads_round(h, C.byref(out)) == 0
        mine = s.round()
        assert torch.equal(mine[0], cand) and torch.equal(mine[1], kept), t
    for x, y in ((s.beta, beta), (s.resid, resid), (s.delta, delta)):
        assert float((x - y).norm()) <= 1e-5 * float(x.norm())
    assert lib.strads_destroy(h) == 0


def test_a_workspace_sized_for_another_rho():
    """Sized with rho = 0.1 (no buffers for rounds in one launch), used with rho = 0.05, which would have them: other kernels, same rounds."""
    import ctypes as C
    from paper_1312_5766_b200 import binding as b
    p = wl.make_problem(dict(SHAPES["no_window"], rho=0.05), seed=6, device="cuda")
    s = b.StradsLasso.from_problem(p, device="cuda")
    lib, cfg = b.load(), b.Config()
    C.memmove(C.byref(cfg), C.byref(s._cfg), C.sizeof(cfg))
    need = C.c_size_t(0)
    cfg.rho = 0.1
    assert lib.strads_workspace_bytes(C.byref(cfg), C.byref(need)) == 0 and need.value < s.workspace.numel()
    cfg.rho = p.rho
    ws = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    beta, resid, delta = torch.zeros_like(s.beta), torch.empty_like(s.resid), torch.empty_like(s.delta)
    cfg.workspace, cfg.workspace_bytes = ws.data_ptr(), need.value
    cfg.beta, cfg.resid, cfg.delta = beta.data_ptr(), resid.data_ptr(), delta.data_ptr()
    h = C.c_void_p(None)
    assert lib.strads_lasso_init(C.byref(cfg), C.byref(h)) == 0
    kept = torch.empty(2, p.n_keep, dtype=torch.int32, device="cuda")
    for _ in range(6):
        out = b.RoundOut()
        out.kept = kept[1].data_ptr()
        assert lib.strads_round(h, C.byref(out)) == 0
        kept[0].copy_(s.round()[1])
        assert torch.equal(kept[0], kept[1])
    assert lib.strads_run(h, 20) == 0
    s.run(20)
    torch.cuda.synchronize()
    for x, y in ((s.beta, beta), (s.resid, resid), (s.delta, delta)):
        assert float((x - y).norm()) <= 1e-5 * float(x.norm())          # dense products in another order
    assert lib.strads_destroy(h) == 0
    cfg.workspace_bytes = need.value - 256
    assert lib.strads_lasso_init(C.byref(cfg), C.byref(h)) == -3

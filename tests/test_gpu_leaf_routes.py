"""The routes of the leaves that few calls take: the bounded waits of the strips, which
have to report that they ran out, and many tall problems side by side, whose strips do
not all run at once (one launch per tile anti-diagonal for all problems instead).
"""
import pytest
import torch

import workloads as WL

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2608_06291_gb300 as P


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()


def test_strips_report_a_wait_that_ran_out(monkeypatch):
    W, A, B = WL.small_problem(300, 200, 4)
    W, f = W.cuda(), P.bakron_prepare(A.cuda(), B.cuda(), 0.01)
    want = P.bakron_solve(W, f, 4)
    monkeypatch.setenv("BAKRON_SPIN_CYCLES", "0")
    with pytest.raises(P.BakronError) as e:
        P.bakron_solve(W, f, 4)
    assert e.value.status == 4
    monkeypatch.delenv("BAKRON_SPIN_CYCLES")
    for a, b in zip(P.bakron_solve(W, f, 4), want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("H,m,n,block", [(32, 200, 640, ""), (32, 180, 130, "5"), (20, 300, 300, "")])
def test_more_strips_than_run_at_once(H, m, n, block, monkeypatch):
    """7 strips of 32 problems, 10 of 20: more CTAs than the GPU holds."""
    if block:
        monkeypatch.setenv("BAKRON_LEAF_BLOCK", block)
    _, A, _ = WL.small_problem(8, n, 11)
    Ws, fs = [], []
    for h in range(H):
        W, _, B = WL.small_problem(m, n, 300 + h)
        Ws.append(W.cuda())
        fs.append(P.bakron_prepare(A.cuda(), B.cuda(), 0.01))
    outs = P.bakron_solve_batched(Ws, fs, 4, streams=H)
    for W, f, o in zip(Ws, fs, outs):
        for a, b in zip(P.bakron_solve(W, f, 4), o):
            assert torch.equal(a, b)

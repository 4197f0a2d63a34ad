"""Blocks of leaves as one launch of strips (clusters of up to eight 32-row strips
that hand each other their last G): more strips than a cluster, strips that start
late or end early in a block, blocks of 1 to 16 anti-diagonals, one column or one
row of tiles, groups, and several problems in one launch.  The oracle decides, as
in test_gpu_parity.py: codes equal free-running, or every code certified where a
decision inside the 1e-4 tie band went the other way.
"""
import numpy as np
import pytest
import torch

import workloads as WL
from tests.test_gpu_parity import _assert_parity_or_certified_tie, _lib, _solve_small  # noqa: F401

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2608_06291_gb300 as P


@pytest.mark.parametrize("block", ["1", "7", "16"])
@pytest.mark.parametrize("m,n,group", [(20, 900, 0), (900, 20, 0), (290, 610, 0), (610, 300, 30), (545, 96, 32)])
def test_strips_match_oracle(m, n, group, block, monkeypatch):
    monkeypatch.setenv("BAKRON_LEAF_BLOCK", block)
    _assert_parity_or_certified_tie(_solve_small(m, n, 31 * m + n, bits=4, group=group))


@pytest.mark.parametrize("H,m,n", [(5, 300, 200), (32, 40, 96)])
def test_strips_of_several_problems_are_the_single_ones(H, m, n):
    fs, Ws = [], []
    for h in range(H):
        W, A, B = WL.small_problem(m, n, 900 + 7 * h)
        fs.append(P.bakron_prepare(A.cuda(), B.cuda(), 0.01))
        Ws.append(W.cuda())
    outs = P.bakron_solve_batched(Ws, fs, 4)
    for W, f, o in zip(Ws, fs, outs):
        for a, b in zip(P.bakron_solve(W, f, 4), o):
            assert torch.equal(a, b)


def test_strips_bounded_wait(monkeypatch):
    """No time for the strips' waits: the call ends with an error, not a hang, and
    the next solve is right."""
    W, A, B = WL.small_problem(300, 200, 4)
    f = P.bakron_prepare(A.cuda(), B.cuda(), 0.01)
    want = P.bakron_solve(W.cuda(), f, 4)[0]
    monkeypatch.setenv("BAKRON_SPIN_CYCLES", "0")
    try:
        P.bakron_solve(W.cuda(), f, 4)
    except P.BakronError as e:
        assert e.status == 4
    monkeypatch.delenv("BAKRON_SPIN_CYCLES")
    assert np.array_equal(P.bakron_solve(W.cuda(), f, 4)[0].cpu().numpy(), want.cpu().numpy())

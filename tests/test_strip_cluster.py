"""The clusters of k_strips: a CTA's shared memory may be touched from outside only
once a cluster barrier has shown that every CTA of the cluster has begun, and the
claim counter keeps solves on several streams apart.
"""
import os
import re

import pytest
import torch

import workloads as WL

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_06291_gb300", "csrc")


def _body(source, head):
    """The text of the function that `head` starts, up to its closing brace."""
    at = source.index(head)
    depth = 0
    for i in range(source.index("{", at), len(source)):
        depth += {"{": 1, "}": -1}.get(source[i], 0)
        if depth == 0:
            return source[at:i]
    raise AssertionError(head)


def test_no_remote_access_before_the_cluster_barrier():
    with open(os.path.join(CSRC, "solve.cu")) as f:
        body = re.sub(r"//[^\n]*", "", _body(f.read(), "void strip_body("))
    before, after = body.split("barrier.cluster.arrive", 1)
    assert "peer_u32" not in before and "shared::cluster" not in before
    assert "peer_u32" in after
    # and none after the last one
    assert "peer_u32" not in body.rsplit("barrier.cluster.wait", 1)[1]


@pytest.mark.gpu
def test_solves_on_two_streams_are_the_single_ones():
    """Several strips' launches of two solves in flight together, each with its own
    workspace: the codes and grids of each alone."""
    import paper_2608_06291_gb300 as P
    P.build()
    jobs = []
    for seed, (m, n) in ((1, (900, 610)), (2, (545, 1200))):
        W, A, B = WL.small_problem(m, n, seed)
        W, f = W.cuda(), P.bakron_prepare(A.cuda(), B.cuda(), 0.01)
        jobs.append((W, f, P.alloc_workspace(m, n), P.bakron_solve(W, f, 4)))
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()
    got = []
    for _ in range(8):
        for s, (W, f, ws, _) in zip(streams, jobs):
            got.append(P.bakron_solve(W, f, 4, workspace=ws, sync=False, stream=s))
    torch.cuda.synchronize()
    for (_, _, ws, _) in jobs:
        assert P.bakron_read_status(ws) == 0
    for i, g in enumerate(got):
        for a, b in zip(g, jobs[i % 2][3]):
            assert torch.equal(a, b)

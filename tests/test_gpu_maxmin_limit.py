"""Max-min on both sides of the size up to which one cluster orders the points
(6,144 points in each CTA's shared memory; a launch a point above it), bit-exact
against the oracle."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu

LIMIT = 98304


def test_around_the_cluster_limit():
    xy = {n: synth.jittered_grid(n, 5) for n in (LIMIT, LIMIT + 1)}
    with ThreadPoolExecutor(2) as pool:  # the oracle is quadratic: the two beside each other
        ref = {n: pool.submit(oracle.order, xy[n], "maxmin") for n in xy}
        ctx = tlr.Context(0)
        got = {n: tlr.tlr_order(ctx, torch.from_numpy(xy[n]).cuda(), "maxmin").cpu().numpy() for n in xy}
        ctx.close()
        for n in xy:
            assert np.array_equal(got[n], ref[n].result()[0]), n

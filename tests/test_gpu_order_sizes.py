"""The cluster orderings at the edges of their warps, CTAs, node sizes and
upper sizes: bit-exact against the oracle, with ties (a lattice, coincident
points, equal codes), coordinates far from the unit square, and xy_out."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 31, 32, 33, 255, 512, 513, 1000, 2047, 2048, 2049, 4095, 4097, 16384, 16385, 33000]


@pytest.fixture(scope="module")
def ctx():
    c = tlr.Context(0)
    yield c
    c.close()


def points(n, kind):
    if kind == "grid":
        return synth.jittered_grid(n, 11)
    g = np.random.default_rng(n)
    if kind == "lattice":
        side = int(np.ceil(np.sqrt(n)))
        i = np.arange(n)
        return np.concatenate([(i % side) / side, (i // side) / side])
    if kind == "far":
        return np.concatenate([1e3 * g.standard_normal(n), -50.0 + 1e-7 * g.standard_normal(n)])
    xy = g.uniform(size=(2, max(1, n // 4)))  # "same": every point about four times
    return xy[:, g.integers(0, xy.shape[1], n)].reshape(-1).copy()


@pytest.mark.parametrize("kind", ["grid", "lattice", "far", "same"])
@pytest.mark.parametrize("method", ["random", "morton", "hilbert", "kdtree", "maxmin"])
def test_orders(ctx, method, kind):
    for n in SIZES:
        if method == "maxmin" and n > 4097:
            continue  # the oracle is quadratic
        xy = points(n, kind)
        d = torch.from_numpy(xy).cuda()
        out = torch.empty_like(d)
        p = tlr.tlr_order(ctx, d, method, xy_out=out).cpu().numpy()
        ref, _ = oracle.order(xy, method)
        assert np.array_equal(p, ref), n
        assert np.array_equal(out.cpu().numpy(), oracle.permute_xy(xy, ref))
        quant = torch.empty_like(d)
        tlr.tlr_order(ctx, d, method, flags=tlr.TLR_ORDER_QUANTIZE, xy_out=quant)
        q = np.rint(np.clip(oracle.permute_xy(xy, ref), 0, 1) * 65535.0) / 65535.0
        assert np.array_equal(quant.cpu().numpy(), q)


@pytest.mark.parametrize("method", ["morton", "hilbert", "kdtree"])
@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1])
def test_around_the_cluster_limit(ctx, method, n):
    xy = synth.jittered_grid(n, 5)
    p = tlr.tlr_order(ctx, torch.from_numpy(xy).cuda(), method).cpu().numpy()
    assert np.array_equal(p, oracle.order(xy, method)[0])

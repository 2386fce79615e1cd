"""The interpolation table of the covariance over its whole range: smoothness,
range, distances from the smallest tabulated one up to sqrt(2), exact powers of
two, points nearer than the table begins, and coincident points, against the
oracle's K_nu at the tiles' bound (1e-12 relative, tests/test_gpu_matern.py)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [0.3, 0.5, 0.81, 1.0, 1.19, 1.5, 2.5])
@pytest.mark.parametrize("beta", [0.01, 0.03, 0.3, 5.0])
def test_table_against_oracle(nu, beta):
    ctx = tlr.Context(0)
    theta = (1.7, beta, nu)
    g = np.random.default_rng(7)
    d = np.concatenate([2.0 ** g.uniform(-24, 0.5, 300), 2.0 ** np.arange(-24, 1.0), [0.0, 1e-9]])
    n = d.size + 1
    xy = np.zeros(2 * n)
    xy[1:n] = d  # on a line: the distances to point 0 are d exactly
    nb = 400
    tiles = tlr.tlr_generate(ctx, torch.from_numpy(xy).cuda(), nb, theta).reshape(-1, nb, nb)
    got = tiles[0, 0, 1:n].cpu().numpy()
    ref = oracle.matern(d, theta)
    assert np.all(np.abs(got - ref) <= 1e-12 * ref)
    ctx.close()

"""tlr_solve on right-hand sides that a product with an explicit inverse of a
32 x 32 diagonal block answers worse than substitution does."""
import numpy as np
import pytest
import torch

import paper_2402_09356_gb300 as tlr
from test_gpu_smooth_tiles import WIDE, covariance, factor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tlr.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("case", [(512, 1 / 100, 2.5, 0.1, 1), (512, 1 / 100, 2.5, 0.1, 3), (800, 1 / 140, 2.5, 0.3, 1)])
def test_smooth_field(ctx, case):
    """z = L w of a smooth field, whose y = w is far smaller than |L^-1| |z|.
    Substitution in blocks of 32: an entry takes up to 32 terms of its own block,
    one subtraction for each block before it and a few roundings of their sums, so
    |L y - z| <= (32 + m / 32 + 8) u |L| |y|, entry by entry."""
    m = case[0]
    M = factor(ctx, covariance(*case))
    L = tlr.tlr_mat_tile(M, 0, 0).cpu().numpy()
    z = L @ np.random.default_rng(m).standard_normal(m)
    y = tlr.tlr_solve(M, torch.from_numpy(z).cuda())[0].cpu().numpy()
    M.close()
    off = np.abs(L.astype(WIDE) @ y.astype(WIDE) - z)
    assert np.all(off <= (32 + m / 32 + 8) * 2.0**-53 * (np.abs(L) @ np.abs(y)))

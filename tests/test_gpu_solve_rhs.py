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


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("row", [1, 31, 40, 255, 383, 395])
def test_rows_above_a_non_finite_entry(ctx, bad, row):
    """Forward substitution: what stands above an entry does not depend on it."""
    m, n = 256, 400
    A = covariance(n, 1 / 20, 0.5, 0.1, 1)
    tiles = np.zeros((3, m, m))
    for t, (i, j) in enumerate([(0, 0), (1, 0), (1, 1)]):
        T = A[i * m:(i + 1) * m, j * m:(j + 1) * m]
        tiles[t, :T.shape[1], :T.shape[0]] = T.T
    M = tlr.TlrMatrix(ctx, n, m, m)
    tlr.tlr_compress(M, torch.from_numpy(tiles.reshape(-1)).cuda(), 1e-9)
    tlr.tlr_potrf(M, 1e-9)
    z = torch.from_numpy(np.random.default_rng(3).standard_normal(n)).cuda()
    ref = tlr.tlr_solve(M, z)[0]
    z[row] = bad
    y = tlr.tlr_solve(M, z)[0]
    M.close()
    assert torch.equal(y[:row], ref[:row])
    assert not torch.isfinite(y[row]) and not bool(torch.isfinite(y[row:]).all())

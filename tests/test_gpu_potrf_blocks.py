"""The diagonal tile's Cholesky around its block widths: tiles factored by one
cluster (up to 288 rows), in two to four blocks, and ragged last blocks.  The
factor and its use of L^-1 are checked on a two-tile matrix (backward error of
an FP64 Cholesky, m u |A| with room), and the failing row of a non-positive
pivot in every block."""
import numpy as np
import pytest
import torch

import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tlr.Context(0)
    yield c
    c.close()


def covariance(n):
    i = np.arange(n)
    return np.exp(-0.01 * np.abs(i[:, None] - i[None, :])) + 0.05 * np.eye(n)


def load(ctx, A, nb):
    n = A.shape[0]
    nt = -(-n // nb)
    tiles = np.zeros((nt * (nt + 1) // 2, nb, nb))
    for i in range(nt):
        for j in range(i + 1):
            t = A[i * nb:(i + 1) * nb, j * nb:(j + 1) * nb]
            tiles[i * (i + 1) // 2 + j, :t.shape[1], :t.shape[0]] = t.T
    M = tlr.TlrMatrix(ctx, n, nb, nb)
    tlr.tlr_compress(M, torch.from_numpy(tiles.reshape(-1)).cuda(), 1e-13)
    return M


@pytest.mark.parametrize("nb", [16, 32, 33, 287, 288, 289, 321, 576, 577, 800, 865, 1000, 1024])
def test_factor(ctx, nb):
    n = nb + nb // 2
    A = covariance(n)
    M = load(ctx, A, nb)
    tlr.tlr_potrf(M, 1e-13)
    L = np.zeros((n, n))
    L[:nb, :nb] = tlr.tlr_mat_tile(M, 0, 0).cpu().numpy()
    L[nb:, nb:] = tlr.tlr_mat_tile(M, 1, 1).cpu().numpy()
    U, V = (t.cpu().numpy() for t in tlr.tlr_mat_tile(M, 1, 0))
    L[nb:, :nb] = U @ V.T
    assert np.all(L[:nb, :nb] == np.tril(L[:nb, :nb])) and np.all(L[nb:, nb:] == np.tril(L[nb:, nb:]))
    assert np.abs(L[:nb, :nb] @ L[:nb, :nb].T - A[:nb, :nb]).max() <= 4e-15
    assert np.abs(L @ L.T - A).max() <= 1e-11  # the off-diagonal tile is truncated at 1e-13 sigma
    z = np.random.default_rng(nb).standard_normal(n)
    y, logdet, _ = tlr.tlr_solve(M, torch.from_numpy(z).cuda())
    assert np.abs(L @ y.cpu().numpy() - z).max() <= 1e-12 * n
    assert abs(logdet - 2 * np.log(np.diag(L)).sum()) <= 1e-12 * n
    M.close()


@pytest.mark.parametrize("row", [0, 31, 32, 287, 288, 300, 575, 576, 637, 799])
def test_failing_row(ctx, row):
    A = np.eye(800)
    A[row, row] = -1.0
    M = load(ctx, A, 800)
    with pytest.raises(tlr.TlrError) as e:
        tlr.tlr_potrf(M, 1e-13)
    assert e.value.code == tlr.TLR_ERR_NOT_SPD and e.value.info == row
    M.close()

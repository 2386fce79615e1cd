"""The single-precision Jacobi sweeps (jacobi_rotate32) over their register
counts: sample sizes from below one row group to past the last, odd and even.
The rank is the count of singular values above eps, and |T - U V'|_2 <= 1.1 eps
(the bound of tests/test_gpu_tlr.py)."""
import numpy as np
import pytest
import torch

import paper_2402_09356_gb300 as tlr
from test_gpu_qr_sizes import EPS, known_tile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,r", [(800, 340), (800, 370), (800, 424), (800, 429)])
def test_large_samples(nb, r):
    check(nb, r)


@pytest.mark.parametrize("r", [2, 21, 45, 64, 82, 97, 114, 131, 148, 163, 180, 197, 211, 228, 241, 250, 275])
def test_known_spectrum(r):
    check(300, r)


def check(nb, r):
    ctx = tlr.Context(0)
    tiles = np.zeros((3, nb, nb))
    tiles[0], tiles[2] = np.eye(nb), np.eye(nb)
    T = known_tile(nb, nb, r, r)
    tiles[1] = T.T  # column major
    A = tlr.TlrMatrix(ctx, 2 * nb, nb, nb)
    dev = torch.from_numpy(tiles.reshape(-1)).cuda()
    for _ in range(2):  # from the default sample size, then from the known rank
        tlr.tlr_compress(A, dev, EPS)
        assert tlr.tlr_mat_ranks(A)[1, 0] == r
        U, V = tlr.tlr_mat_tile(A, 1, 0)
        assert np.linalg.norm(T - U.cpu().numpy() @ V.cpu().numpy().T, 2) <= 1.1 * EPS
    A.close()
    ctx.close()

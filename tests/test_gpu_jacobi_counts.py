"""Counters of the Jacobi sweeps, on a tile whose columns' squared norms
underflow single precision: its FP32 sweeps check every pair and rotate none, and
FP64 sweeps finish it."""
import numpy as np
import pytest
import torch

import paper_2402_09356_gb300 as tlr
from test_gpu_qr_sizes import EPS, known_tile

pytestmark = pytest.mark.gpu


def test_counts_of_a_tile_finished_in_fp64():
    nb, r, scale = 176, 150, 1e-24
    ctx = tlr.Context(0)
    tiles = np.zeros((3, nb, nb))
    tiles[0], tiles[2] = np.eye(nb), np.eye(nb)
    T = scale * known_tile(nb, nb, r, 1)
    tiles[1] = T.T  # column major
    A = tlr.TlrMatrix(ctx, 2 * nb, nb, nb)
    tlr.tlr_profile(ctx, True)
    before = tlr.tlr_kernel_stats(ctx)
    tlr.tlr_compress(A, torch.from_numpy(tiles.reshape(-1)).cuda(), EPS * scale)
    k = {n: v - before[n] for n, v in tlr.tlr_kernel_stats(ctx).items()}
    st = tlr.tlr_compress_stats(ctx)
    assert tlr.tlr_mat_ranks(A)[1, 0] == r
    A.close()
    ctx.close()
    # one FP32 sweep a compression, kept when FP64 sweeps finish the tile
    assert st["sweeps"] > 0 and st["svd_global"] == 0
    assert st["sweeps32"] == st["tiles"]
    # samples of 161 to 176 columns: the norms and a dot product for each pair
    low, high = (s * s * (s + 1.0) for s in (161, 176))
    assert k["jacobi16_clusters"] > 0
    assert low * k["jacobi16_clusters"] <= k["jacobi16_flops"] <= high * k["jacobi16_clusters"]

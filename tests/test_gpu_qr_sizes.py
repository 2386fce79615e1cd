"""The compression's QR (k_qr_factor, k_qr_form) over its sizes: tiles of a
known spectrum, from one row group to the largest tile, sample sizes of every
cluster size, odd and ragged tiles.  The rank is the count of singular values
above eps, and |T - U V'|_2 <= 1.1 eps (the bound of tests/test_gpu_tlr.py)."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu

EPS = 1e-7


@pytest.fixture(scope="module")
def ctx():
    c = tlr.Context(0)
    yield c
    c.close()


def known_tile(m, k, r, seed):
    """m x k with r singular values from 1 down to 10 eps and a tail 1e-3 eps."""
    g = np.random.default_rng(seed)
    full = min(m, k)
    s = np.full(full, 1e-3 * EPS)
    if r:
        s[:r] = np.logspace(0, np.log10(10 * EPS), r) if r > 1 else 1.0
    u = np.linalg.qr(g.standard_normal((m, full)))[0]
    v = np.linalg.qr(g.standard_normal((k, full)))[0]
    return (u * s) @ v.T


@pytest.mark.parametrize("nb,cut,r", [(16, 0, 3), (33, 0, 5), (200, 7, 40), (257, 0, 70), (512, 100, 120),
                                      (640, 0, 150), (800, 0, 0), (800, 799, 1), (801, 0, 200), (1024, 0, 300)])
def test_known_spectrum(ctx, nb, cut, r):
    n = 2 * nb - cut
    m = nb - cut
    T = known_tile(m, nb, r, nb + r)
    tiles = np.zeros((3, nb, nb))
    tiles[0], tiles[2] = np.eye(nb), np.eye(nb)
    tiles[1, :, :m] = T.T  # column major
    A = tlr.TlrMatrix(ctx, n, nb, nb)
    dev = torch.from_numpy(tiles.reshape(-1)).cuda()
    for _ in range(2):  # from the default sample size, then from the known rank
        tlr.tlr_compress(A, dev, EPS)
        assert tlr.tlr_mat_ranks(A)[1, 0] == r
        U, V = tlr.tlr_mat_tile(A, 1, 0)
        E = T - U.cpu().numpy() @ V.cpu().numpy().T
        assert np.linalg.norm(E, 2) <= 1.1 * EPS
    A.close()


@pytest.mark.parametrize("n,nb", [(330, 100), (1000, 333), (1500, 520), (1700, 801), (2100, 1024)])
@pytest.mark.parametrize("precision", [tlr.TLR_PREC_FP64, tlr.TLR_PREC_MIXED, tlr.TLR_PREC_TENSOR])
def test_likelihood(ctx, n, nb, precision):
    theta = (1.0, 0.1, 0.5)
    xy = synth.jittered_grid(n, 5)
    z = oracle.simulate_z(xy, theta, synth.standard_normal(n, 6))
    d = torch.from_numpy(xy).cuda()
    xyo = torch.empty_like(d)
    perm = tlr.tlr_order(ctx, d, "hilbert", xy_out=xyo)
    zo = tlr.tlr_gather(ctx, perm, torch.from_numpy(z).cuda())
    ref = oracle.loglik_dense(xy, z, theta)
    L = tlr.TlrMatrix(ctx, n, nb, nb)
    for _ in range(2):
        r = tlr.tlr_loglik(L, xyo, zo, theta, tlr.Options(nb=nb, eps=EPS, maxrank=nb, precision=precision))
        for k in ("loglik", "logdet", "quad"):
            assert abs(r[k] - ref[k]) <= 10 * EPS * abs(ref[k]), k
    L.close()

"""y = L^-1 z and z = L w with a kept factor over their sizes: tiles from one
block of 16 rows to 1,024, ragged last tiles, tiles of rank 0, more columns
than one CTA takes, compact storage, in place; against the dense matrix of the
factor's own tiles (forward substitution and product in FP64: n u times the
condition of the factor, here below 1e-11)."""
import numpy as np
import pytest
import torch

import synth
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu


def dense_factor(M):
    n, nb, nt = M.n, M.nb, M.nt
    L = np.zeros((n, n))
    for i in range(nt):
        a, b = i * nb, min(n, (i + 1) * nb)
        L[a:b, a:b] = tlr.tlr_mat_tile(M, i, i).cpu().numpy()
        for j in range(i):
            U, V = tlr.tlr_mat_tile(M, i, j)
            L[a:b, j * nb:(j + 1) * nb] = U.cpu().numpy() @ V.cpu().numpy().T
    return L


@pytest.mark.parametrize("n,nb,eps", [(1, 16, 1e-7), (16, 16, 1e-7), (45, 16, 1e-7), (200, 33, 1e-9),
                                      (1000, 64, 1e-2), (1500, 200, 1e-9), (1700, 500, 1e-7), (2049, 1024, 1e-7),
                                      (2500, 801, 1e-5)])
@pytest.mark.parametrize("compact", [False, True])
def test_solve_and_product(n, nb, eps, compact):
    ctx = tlr.Context(0)
    theta = (1.0, 0.05, 0.5)
    xy = torch.from_numpy(synth.jittered_grid(n, 3)).cuda()
    xyo = torch.empty_like(xy)
    tlr.tlr_order(ctx, xy, "hilbert", xy_out=xyo)
    z = torch.from_numpy(synth.standard_normal(n, 4)).cuda()
    M = tlr.TlrMatrix(ctx, n, nb, nb)
    opts = tlr.Options(nb=nb, eps=eps, maxrank=nb)
    r = tlr.tlr_loglik(M, xyo, z, theta, opts)
    if compact:
        M2 = tlr.TlrMatrix(ctx, n, nb, nb, rank_map=tlr.tlr_mat_ranks(M))
        M.close()
        M = M2
        r = tlr.tlr_loglik(M, xyo, z, theta, opts)
    L = dense_factor(M)
    y, logdet, quad = tlr.tlr_solve(M, z)
    h = z.cpu().numpy()
    ref = np.linalg.solve(L, h)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
    assert abs(logdet - 2 * np.log(np.diag(L)).sum()) <= 1e-12 * n
    assert abs(quad - ref @ ref) <= 1e-11 * (ref @ ref)
    assert abs(logdet - r["logdet"]) <= 1e-12 * n
    w = tlr.tlr_lmul(M, z).cpu().numpy()
    assert np.linalg.norm(w - L @ h) <= 1e-12 * np.linalg.norm(L @ h)
    inplace = z.clone()
    tlr.tlr_solve(M, inplace, inplace)
    assert torch.equal(inplace, y)
    M.close()
    ctx.close()

"""A factorisation of more tile pairs than fit the descriptor ring at once: with
850 tile rows the update of a middle column has 425 x 425 = 180,625 products,
whose descriptors of 96 bytes take more than its 16 MB."""
import pytest
import torch

import synth
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu


def test_many_small_tiles():
    n, eps, theta = 13600, 1e-7, (1.0, 0.3, 0.5)
    ctx = tlr.Context(0)
    xy = torch.from_numpy(synth.jittered_grid(n, 3)).cuda()
    xyo = torch.empty_like(xy)
    tlr.tlr_order(ctx, xy, "hilbert", xy_out=xyo)
    z = torch.from_numpy(synth.standard_normal(n, 4)).cuda()
    got = {}
    for nb in (16, 400):
        M = tlr.TlrMatrix(ctx, n, nb, min(nb, 128))
        got[nb] = tlr.tlr_loglik(M, xyo, z, theta, tlr.Options(nb=nb, eps=eps, maxrank=min(nb, 128)))
        M.close()
    ctx.close()
    # tiles off by eps each make |Sigma - Sigma~| <= 850 eps = 8.5e-5 against a
    # smallest eigenvalue of about 0.01: every term of the likelihood within 1%
    for k in ("logdet", "quad"):
        assert abs(got[16][k] - got[400][k]) <= 1e-2 * abs(got[400][k])

"""The diagonal tile of smooth fields without a nugget, whose Cholesky factor
has pivots spread over many orders of magnitude: an explicit inverse of a wide
diagonal block loses digits there that substitution keeps.  The factor and its
inverse may be no worse than those of the Cholesky algorithm that inverts
blocks of 32 columns only, restated here, times 1.75 for another order of
rounding (blocks of 288 inverted whole: 2.3 to 6 times)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_09356_gb300 as tlr

pytestmark = pytest.mark.gpu

WIDE = np.longdouble


def covariance(m, h, nu, beta, seed):
    """Matern covariance of m points of a perturbed grid of spacing h."""
    g = np.random.default_rng(seed)
    side = int(np.ceil(np.sqrt(m)))
    p = np.arange(m)
    x, y = ((q + 0.5 + 0.8 * (g.random(m) - 0.5)) * h for q in (p % side, p // side))
    d = np.sqrt((x[:, None] - x)**2 + (y[:, None] - y)**2)
    return oracle.matern(d.ravel(), (1.0, beta, nu)).reshape(m, m)


def product(a, b):
    """a @ b to more than 70 bits of the rows' and columns' largest entries: four
    slices of 20 bits each, whose products and sums are exact in 64 bits."""
    def slices(v, axis):
        r = np.asarray(v, WIDE)
        scale = np.exp2(np.ceil(np.log2(np.maximum(np.abs(v).max(axis=axis, keepdims=True), 1e-300)))).astype(WIDE)
        r = r / scale
        out = []
        for k in range(4):
            unit = WIDE(2)**(20 * k + 19)
            q = np.rint(r * unit) / unit
            out.append(np.asarray(q * scale, float))
            r = r - q
        return out
    A, B = slices(a, 1), slices(b, 0)
    return sum((A[i] @ B[j]).astype(WIDE) for i in range(4) for j in range(4 - i))


def factor32(A):
    """L and L^-1 with inverses of 32 x 32 diagonal blocks."""
    A, m = A.copy(), A.shape[0]
    X = np.eye(m)
    for p in range(0, m, 32):
        e = min(m, p + 32)
        L = np.linalg.cholesky(A[p:e, p:e])
        inv = np.eye(e - p)  # by forward substitution
        for c in range(e - p):
            inv[c] /= L[c, c]
            inv[c + 1:] -= np.outer(L[c + 1:, c], inv[c])
        A[p:e, p:e] = L
        A[e:, p:e] = A[e:, p:e] @ inv.T
        X[p:e, :e] = inv @ X[p:e, :e]
        A[e:, e:] -= A[e:, p:e] @ A[e:, p:e].T
        X[e:, :e] -= A[e:, p:e] @ X[p:e, :e]
    return np.tril(A), np.tril(X)


def norm(a):
    return float(np.sqrt((np.asarray(a, WIDE)**2).sum()))


@pytest.fixture(scope="module")
def ctx():
    c = tlr.Context(0)
    yield c
    c.close()


def factor(ctx, A, W=None, eps=1e-14):
    """Factor with tile size m of [[A, W'], [W, I]] (or of A alone); the matrix."""
    m = A.shape[0]
    n = m + (0 if W is None else W.shape[0])
    tiles = np.zeros((1 if W is None else 3, m, m))
    tiles[0] = A
    if W is not None:
        tiles[1, :, :n - m] = W.T  # column major
        tiles[2, :n - m, :n - m] = np.eye(n - m)
    M = tlr.TlrMatrix(ctx, n, m, min(m, 64))
    tlr.tlr_compress(M, torch.from_numpy(tiles.reshape(-1)).cuda(), eps)
    tlr.tlr_potrf(M, eps)
    return M


def factor_errors(ctx, case):
    A = covariance(*case)
    M = factor(ctx, A)
    L = tlr.tlr_mat_tile(M, 0, 0).cpu().numpy()
    M.close()
    ref = factor32(A)[0]
    return norm(product(L, L.T) - A), norm(product(ref, ref.T) - A)


def inverse_errors(ctx, case):
    """An off-diagonal tile U0 (L G)' of rank 8 becomes U (X L G)', X = L^-1:
    L times it against what it was."""
    A = covariance(*case)
    m = A.shape[0]
    Lr, Xr = factor32(A)
    g = np.random.default_rng(case[-1])
    U0 = np.linalg.qr(g.standard_normal((32, 8)))[0]
    V0 = 0.1 * (Lr @ np.linalg.qr(g.standard_normal((m, 8)))[0])
    W = U0 @ V0.T
    M = factor(ctx, A, W)
    L = tlr.tlr_mat_tile(M, 0, 0).cpu().numpy()
    U, V = (t.cpu().numpy() for t in tlr.tlr_mat_tile(M, 1, 0))
    M.close()
    got = product(L, V @ U.T) - W.T
    return norm(got), norm(product(Lr, (Xr @ V0) @ U0.T) - W.T)


FACTOR = [(800, 1 / 200, 0.5, 0.1, 1), (400, 1 / 100, 1.0, 0.1, 1), (800, 1 / 45, 2.0, 0.1, 2), (800, 1 / 28, 2.5, 0.1, 2)]
INVERSE = [(512, 1 / 70, 2.5, 0.1, 1), (512, 1 / 70, 2.5, 0.1, 2), (800, 1 / 28, 2.5, 0.1, 1), (800, 1 / 28, 2.5, 0.1, 2)]


@pytest.mark.parametrize("case", FACTOR)
def test_factor(ctx, case):
    got, ref = factor_errors(ctx, case)
    assert got <= 1.75 * ref


@pytest.mark.parametrize("case", INVERSE)
def test_inverse(ctx, case):
    got, ref = inverse_errors(ctx, case)
    assert got <= 1.75 * ref

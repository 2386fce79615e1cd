"""What the framework's speed is measured on: passes through its public entry points.

The calls are those of a maximum-likelihood study (Sec. 5 of the paper): order the locations, generate and compress the
covariance, factor it, solve with the factor, draw data from it, and above all evaluate the log-likelihood, one dataset
or several at once, on each precision path.  Locations are the perturbed regular grid of the repository's workloads;
observations are a random field with the case's Matern covariance (random cosine features of its spectral density).
"""
import math
import random

import numpy as np
import torch

import paper_2402_09356_gb300 as tlr

_DEV = "cuda:0"
_PREC = {"fp64": tlr.TLR_PREC_FP64, "mixed": tlr.TLR_PREC_MIXED, "tensor": tlr.TLR_PREC_TENSOR}
_CTX = None


def _context():
    """A program keeps one library context (streams, descriptor rings) for its life."""
    global _CTX
    if _CTX is None:
        _CTX = tlr.Context(0)
    return _CTX


def listed():
    return [
        # Every run begins by ordering its locations and permuting its data; Hilbert is the fastest order of the study.
        {"name": "order_hilbert_n40000", "kind": "order", "method": "hilbert", "n": 40000},
        # The study's other tree-like order, at the same size.
        {"name": "order_kdtree_n40000", "kind": "order", "method": "kdtree", "n": 40000},
        # The study's statistical order (maximum-minimum distance), at the smallest size of its memory table.
        {"name": "order_maxmin_n10000", "kind": "order", "method": "maxmin", "n": 10000},
        # The covariance tiles of the memory table (tile 1000), for a user who looks at Sigma itself.
        {"name": "generate_n10000", "kind": "generate", "n": 10000, "nb": 1000, "beta": 0.1, "nu": 1.0},
        # The paper's own route on those tiles: compress, factor, solve, as separate calls.
        {"name": "unfused_n10000", "kind": "unfused", "n": 10000, "nb": 1000, "eps": 1e-7, "beta": 0.03, "nu": 0.5},
        # A kept factor used again: L^-1 z for another data vector.
        {"name": "solve_n20000", "kind": "solve", "n": 20000, "nb": 800, "eps": 1e-7, "beta": 0.1, "nu": 0.5},
        # A kept factor used to draw data, z = L w.
        {"name": "lmul_n20000", "kind": "lmul", "n": 20000, "nb": 800, "eps": 1e-7, "beta": 0.1, "nu": 0.5},
        # The smallest whole evaluation, from host arrays (copy, order, evaluate): the 40 x 40 parity workload.
        {"name": "host_fp64_n1600", "kind": "host", "n": 1600, "nb": 200, "eps": 1e-9, "beta": 0.1, "nu": 0.5,
         "precision": "fp64"},
        # One step of a likelihood search in full precision, at a size of the paper's Table 2.
        {"name": "loglik_fp64_n16000", "kind": "loglik", "n": 16000, "nb": 800, "eps": 1e-7, "beta": 0.1, "nu": 0.5,
         "precision": "fp64"},
        # The paired-FP32 path on a ragged size, a smoother field of short range, a smaller tile.
        {"name": "loglik_mixed_n11025", "kind": "loglik", "n": 11025, "nb": 512, "eps": 1e-7, "beta": 0.03, "nu": 1.0,
         "precision": "mixed"},
        # The headline workload: 200 x 200 locations on the tensor path.
        {"name": "loglik_tensor_n40000", "kind": "loglik", "n": 40000, "nb": 800, "eps": 1e-7, "beta": 0.1, "nu": 0.5,
         "precision": "tensor"},
        # The batched workload: datasets of 2,000 to 20,000 locations, each with its own theta, in one call.
        {"name": "batch_mixed_8", "kind": "batch", "count": 8, "mix": 3, "n_min": 2000, "n_max": 20000, "nb": 800,
         "eps": 1e-7, "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["order", "order", "generate", "unfused", "solve", "lmul", "host", "loglik", "loglik", "loglik",
                       "batch"])
    if kind == "order":
        method = rng.choice(["hilbert", "morton", "random", "kdtree", "maxmin"])
        return {"kind": kind, "method": method, "n": _log_int(rng, 400, 10000 if method == "maxmin" else 90000)}
    # fields of the study's range that stay well enough conditioned for every path to agree
    theta = {"beta": round(rng.uniform(0.03, 0.12), 4), "nu": round(rng.uniform(0.4, 0.8), 4)}
    if kind == "generate":
        theta = {"beta": round(rng.uniform(0.03, 0.3), 4), "nu": round(rng.uniform(0.4, 2.5), 4)}
        return {"kind": kind, "n": _log_int(rng, 500, 10000), "nb": rng.choice([200, 333, 512, 800, 1000]), **theta}
    nb = rng.choice([400, 500, 512, 640, 800, 1000])
    eps = rng.choice([1e-5, 1e-7, 1e-7])
    if kind == "unfused":
        return {"kind": kind, "n": _log_int(rng, 1000, 10000), "nb": nb, "eps": eps, **theta}
    if kind in ("solve", "lmul"):
        return {"kind": kind, "n": _log_int(rng, 1000, 20000), "nb": nb, "eps": eps, **theta}
    precision = rng.choice(["fp64", "mixed", "tensor"])
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 900, 5000), "nb": nb, "eps": eps, "precision": precision, **theta}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 8), "mix": rng.randint(10, 10**6), "n_min": 2000, "n_max": 12000,
                "nb": rng.choice([512, 800]), "eps": eps, "precision": precision}
    return {"kind": kind, "n": _log_int(rng, 1000, 16000 if precision == "fp64" else 24000), "nb": nb, "eps": eps,
            "precision": precision, **theta}


# ---- inputs ----------------------------------------------------------------------------------------------------------


def _generator(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed))
    return g


def _grid(n, g):
    """n locations of a perturbed grid in (0, 1)^2, x then y."""
    side = math.isqrt(n - 1) + 1
    h = 1.0 / side
    p = torch.arange(n, device=_DEV)
    u = torch.rand(2, n, generator=g, device=_DEV, dtype=torch.float64)
    cell = torch.stack([p % side, p // side]).double()
    return ((cell + 0.5) * h + (2.0 * u - 1.0) * 0.4 * h).reshape(-1).contiguous()


def _curve(xy, method):
    """The permutation along a space-filling curve of 16-bit coordinates (ties keep their order)."""
    n = xy.numel() // 2
    q = torch.round(xy.clamp(0, 1) * 65535.0).long()
    qx, qy = q[:n], q[n:]
    d = torch.zeros_like(qx)
    swap = torch.zeros_like(qx)
    comp = torch.zeros_like(qx)
    for b in range(15, -1, -1):
        bx, by = (qx >> b) & 1, (qy >> b) & 1
        if method == "morton":
            d = (d << 2) | (by << 1) | bx
            continue
        bx, by = bx ^ comp, by ^ comp
        bx, by = torch.where(swap == 1, by, bx), torch.where(swap == 1, bx, by)
        quad = (bx << 1) | (bx ^ by)
        d = (d << 2) | quad
        swap = swap ^ ((quad == 0) | (quad == 3)).long()
        comp = comp ^ (quad == 3).long()
    return torch.sort(d, stable=True)[1]


def _field(xy, theta, g, features=512):
    """Observations at xy: a sum of cosines with frequencies from the Matern spectral density (2 nu degrees of freedom)."""
    _, beta, nu = theta
    n = xy.numel() // 2
    w = torch.randn(features, 2, generator=g, device=_DEV, dtype=torch.float64)
    # chi^2 with 2 nu degrees of freedom = 2 Gamma(nu)
    chi2 = 2.0 * torch._standard_gamma(torch.full((features, 1), nu, device=_DEV, dtype=torch.float64), generator=g)
    w = w / (beta * chi2.sqrt())
    phase = 2.0 * math.pi * torch.rand(features, generator=g, device=_DEV, dtype=torch.float64)
    z = torch.zeros(n, device=_DEV, dtype=torch.float64)
    for a in range(0, n, 8192):
        b = min(n, a + 8192)
        z[a:b] = torch.cos(torch.outer(xy[a:b], w[:, 0]) + torch.outer(xy[n + a:n + b], w[:, 1]) + phase).sum(1)
    return z * math.sqrt(2.0 / features)


def _theta(case):
    return (1.0, case["beta"], case["nu"])


def _dataset(n, theta, g, method=None):
    """Locations and observations, in the order of a curve if one is named."""
    xy = _grid(n, g)
    z = _field(xy, theta, g)
    if method:
        p = _curve(xy, method)
        xy = torch.cat([xy[:n][p], xy[n:][p]]).contiguous()
        z = z[p].contiguous()
    return xy, z


def _members(case):
    """(n, theta) of each dataset of a batch."""
    r = random.Random(case["mix"])
    return [(r.randint(case["n_min"], case["n_max"]),
             (r.uniform(0.5, 2.0), r.uniform(0.03, 0.1), r.uniform(0.4, 0.8))) for _ in range(case["count"])]


def _options(case):
    return tlr.Options(nb=case["nb"], eps=case["eps"], precision=_PREC[case.get("precision", "fp64")])


class _Device:
    """A view of device memory for torch.as_tensor; the tensor keeps the memory's owner alive."""

    def __init__(self, owner, address, shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f8", "data": (address, False), "version": 2,
                                         "strides": None}


def _diagonal(mat):
    """The factor's diagonal tiles (the matrix's own memory), tile t column major in slice t."""
    at = mat.layout()
    return torch.as_tensor(_Device(mat, at["D"], (at["nt"], at["nb"], at["nb"])), device=_DEV)


def prepare(case, seed):
    ctx = _context()
    g = _generator(seed)
    kind = case["kind"]
    s = {"case": case, "ctx": ctx}
    if kind == "order":
        s["xy"], s["z"] = _dataset(case["n"], (1.0, 0.1, 0.5), g)
        return s
    if kind == "batch":
        s["sets"] = [_dataset(n, theta, g, "morton") for n, theta in _members(case)]
        s["mats"] = [tlr.TlrMatrix(ctx, n, case["nb"]) for n, _ in _members(case)]
        s["D"] = [_diagonal(m) for m in s["mats"]]
        return s
    n, theta = case["n"], _theta(case)
    if kind == "generate":
        s["xy"], _ = _dataset(n, theta, g, "hilbert")
        return s
    s["mat"] = tlr.TlrMatrix(ctx, n, case["nb"])
    s["D"] = _diagonal(s["mat"])
    if kind == "host":
        xy, z = _dataset(n, theta, g)
        s["xy"], s["z"] = xy.cpu().pin_memory(), z.cpu().pin_memory()
        return s
    s["xy"], s["z"] = _dataset(n, theta, g, "hilbert")
    if kind == "unfused":
        s["tiles"] = tlr.tlr_generate(ctx, s["xy"], case["nb"], theta)
    elif kind in ("solve", "lmul"):
        tlr.tlr_loglik(s["mat"], s["xy"], s["z"], theta, _options(case))
    return s


def _numbers(r):
    return np.array([r["loglik"], r["logdet"], r["quad"]])


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "order":
        xyo = torch.empty_like(s["xy"])
        perm = tlr.tlr_order(ctx, s["xy"], case["method"], xy_out=xyo)
        return {"perm": perm, "xy": xyo, "z": tlr.tlr_gather(ctx, perm, s["z"])}
    if kind == "generate":
        return {"tiles": tlr.tlr_generate(ctx, s["xy"], case["nb"], _theta(case))}
    if kind == "unfused":
        tlr.tlr_compress(s["mat"], s["tiles"], case["eps"])
        tlr.tlr_potrf(s["mat"], case["eps"])
        y, logdet, quad = tlr.tlr_solve(s["mat"], s["z"])
        return {"y": y, "numbers": np.array([logdet, quad]), "D": s["D"]}
    if kind == "solve":
        y, logdet, quad = tlr.tlr_solve(s["mat"], s["z"])
        return {"y": y, "numbers": np.array([logdet, quad])}
    if kind == "lmul":
        return {"z": tlr.tlr_lmul(s["mat"], s["z"])}
    if kind == "host":
        r = tlr.tlr_loglik_host(s["mat"], s["xy"], s["z"], _theta(case), _options(case), order="hilbert")
        return {"numbers": _numbers(r), "D": s["D"]}
    if kind == "loglik":
        r = tlr.tlr_loglik(s["mat"], s["xy"], s["z"], _theta(case), _options(case))
        return {"numbers": _numbers(r), "D": s["D"]}
    res, status = tlr.tlr_loglik_batch(s["mats"], [x for x, _ in s["sets"]], [z for _, z in s["sets"]],
                                       [t for _, t in _members(case)], _options(case))
    return {"numbers": [_numbers(r) for r in res], "status": np.array(status), "D": s["D"]}


# ---- the work no implementation can leave out ---------------------------------------------------------------------------


def _rank_sum(n, nb, eps):
    """Estimated sum of the off-diagonal ranks: about two neighbours a tile with a rank of a fifth of the tile, a dozen
    for the others, in proportion to the digits of eps."""
    nt = -(-n // nb)
    near = min(2 * nt, nt * (nt - 1) // 2)
    return (near * 0.2 * nb + (nt * (nt - 1) // 2 - near) * 12.0) * (-math.log10(eps) / 7.0)


def _factor_work(n, nb, eps, generate):
    """Bytes and flops of one evaluation: locations and data in, factor out; 40 operations a covariance entry, the
    diagonal Cholesky, the compression, the low-rank updates and solves."""
    nt, ranks = -(-n // nb), _rank_sum(n, nb, eps)
    lower = n * (n + nb) / 2.0
    flops = (40.0 * lower if generate else 0.0) + nt * nb**3 / 3.0 + 10.0 * nb * nb * ranks + 2.0 * nt / 3.0 * nb * ranks * 24
    return {"bytes": 24.0 * n + 8.0 * (n * nb / 2.0 + 2.0 * nb * ranks), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "order":
        n = case["n"]
        # locations and data read, permutation, locations and data written
        return {"bytes": 24.0 * n + 32.0 * n, "flops": (n * n * 5.0 if case["method"] == "maxmin" else 0.0)}
    if kind == "generate":
        nt = -(-case["n"] // case["nb"])
        entries = nt * (nt + 1) / 2 * case["nb"]**2
        return {"bytes": 16.0 * case["n"] + 8.0 * entries, "flops": 40.0 * entries}
    if kind == "batch":
        each = [_factor_work(n, case["nb"], case["eps"], True) for n, _ in _members(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    n, nb = case["n"], case["nb"]
    if kind in ("solve", "lmul"):
        held = n * nb / 2.0 + 2.0 * nb * _rank_sum(n, nb, case["eps"])
        return {"bytes": 16.0 * n + 8.0 * held, "flops": 2.0 * held}
    w = _factor_work(n, nb, case["eps"], kind != "unfused")
    if kind == "unfused":
        w["bytes"] += 8.0 * n * (n + nb) / 2.0
    return w


# ---- the same results from plain dense algebra in 64 bits -------------------------------------------------------------------


def _correlation(d, beta, nu):
    """Matern correlation: closed forms at nu = 1/2, 3/2, 5/2, else the integral of exp(-x cosh t) cosh(nu t)."""
    x = d / beta
    if nu == 0.5:
        return torch.exp(-x)
    if nu == 1.5:
        return (1.0 + x) * torch.exp(-x)
    if nu == 2.5:
        return (1.0 + x + x * x / 3.0) * torch.exp(-x)
    zero = x == 0
    x = torch.where(zero, torch.ones_like(x), x)
    # the trapezoid rule with the factor exp(-x) taken out: cosh t - 1 = 2 sinh^2(t / 2)
    step, k = 0.1, torch.zeros_like(x)
    for i in range(140):
        t = i * step
        k += (step if i else 0.5 * step) * math.cosh(nu * t) * torch.exp(x * (-2.0 * math.sinh(0.5 * t)**2))
    c = torch.exp((1.0 - nu) * math.log(2.0) - math.lgamma(nu) + nu * torch.log(x) - x) * k
    return torch.where(zero, torch.ones_like(c), c)


def _covariance(xy, theta, lower=True):
    n = xy.numel() // 2
    out = torch.zeros(n, n, device=_DEV, dtype=torch.float64)
    for a in range(0, n, 1024):
        b = min(n, a + 1024)
        e = b if lower else n
        d = torch.sqrt((xy[a:b, None] - xy[None, :e])**2 + (xy[n + a:n + b, None] - xy[None, n:n + e])**2)
        out[a:b, :e] = theta[0] * _correlation(d, theta[1], theta[2])
    return out


def _dense(xy, z, theta):
    """Cholesky factor, L^-1 z and (l, log-determinant, quadratic term)."""
    n = z.numel()
    c = _covariance(xy, theta)
    f = torch.linalg.cholesky(c)
    del c
    y = torch.linalg.solve_triangular(f, z[:, None], upper=False)[:, 0]
    logdet, quad = 2.0 * float(f.diagonal().log().sum()), float(y @ y)
    return f, y, np.array([-0.5 * (n * math.log(2.0 * math.pi) + logdet + quad), logdet, quad])


def _diagonal_of(f, nb):
    """The diagonal tiles of a dense factor, laid out like the library's (column major, zero padded)."""
    n = f.shape[0]
    nt = -(-n // nb)
    d = torch.zeros(nt, nb, nb, device=_DEV, dtype=torch.float64)
    for t in range(nt):
        a, b = t * nb, min(n, (t + 1) * nb)
        d[t, :b - a, :b - a] = f[a:b, a:b].T
    return d


def exact(case, seed):
    kind = case["kind"]
    g = _generator(seed)
    if kind == "order":
        if case["method"] not in ("hilbert", "morton"):
            return None
        n = case["n"]
        xy, z = _dataset(n, (1.0, 0.1, 0.5), g)
        p = _curve(xy, case["method"])
        return {"perm": p, "xy": torch.cat([xy[:n][p], xy[n:][p]]), "z": z[p]}
    if kind == "batch":
        out = {"numbers": [], "status": None, "D": []}
        sets = [_dataset(n, theta, g, "morton") for n, theta in _members(case)]
        for (xy, z), (n, theta) in zip(sets, _members(case)):
            f, _, numbers = _dense(xy, z, theta)
            out["numbers"].append(numbers)
            out["D"].append(_diagonal_of(f, case["nb"]))
        return out
    n, nb, theta = case["n"], case["nb"], _theta(case)
    if n > 24000:
        return None
    if kind == "generate":
        xy, _ = _dataset(n, theta, g, "hilbert")
        c = _covariance(xy, theta, lower=False)
        nt = -(-n // nb)
        tiles = torch.zeros(nt * (nt + 1) // 2, nb, nb, device=_DEV, dtype=torch.float64)
        for i in range(nt):
            for j in range(i + 1):
                t = c[i * nb:(i + 1) * nb, j * nb:(j + 1) * nb]
                tiles[i * (i + 1) // 2 + j, :t.shape[1], :t.shape[0]] = t.T
        return {"tiles": tiles.reshape(-1)}
    xy, z = _dataset(n, theta, g, None if kind == "host" else "hilbert")
    if kind == "host":
        p = _curve(xy, "hilbert")
        xy, z = torch.cat([xy[:n][p], xy[n:][p]]), z[p]
    if kind == "lmul":
        f, _, _ = _dense(xy, z, theta)
        return {"z": f @ z}
    f, y, numbers = _dense(xy, z, theta)
    if kind == "solve":
        return {"y": y, "numbers": numbers[1:]}
    if kind == "unfused":
        return {"y": y, "numbers": numbers[1:], "D": _diagonal_of(f, nb)}
    return {"numbers": numbers, "D": _diagonal_of(f, nb)}

"""Binary64 solves of data that spans many binades: small values beside large ones
keep their digits, as with the FP64 stencil.

Two iterations of CG from zero give, point by point,

    x = a0 b + a1 (r + b1 b),  r = b - a0 A b,

so an error of the stencil at a point shows there, however small the point's values
are.  The error is compared with S = a0 |b| + a1 (|b| + a0 |A| |b| + b1 |b|) of the same
point.  Every operation there rounds by 2^-53 of a term of S; the scalars' relative
errors are those of dot products of L <= 1024 terms a lane, (1 + k) L 2^-53 each with k
the ratio of the sums of |terms| and terms ((p, A p), twice; the residual's
cancellation enters (r, r) once more), k <= 8 for all inputs here and asserted: below
4 x 9 x 9 x 1024 x 2^-53 < 2^-34.  Values truncated at 2^-58 of a large neighbour's would be
off by S itself.

The multigrid's binary64 passes (sweeps, residuals, middle levels, p and A p) on the
same inputs: the oracle's iterates within 1e-11 (norm-wise), the bound of the
other multigrid tests."""
import numpy as np
import pytest
import torch

import lap5_inputs as gen
import oracle
import paper_1803_03797_gb300 as lap5cg

pytestmark = pytest.mark.gpu

KINDS = ["gauss", "spike", "checker", "binades", "columns", "blocks"]
ROUTES = {"ring": dict(ring_slots=4, resident=-1), "resident": {}}


def _data(kind, nx, ny):
    rng = np.random.default_rng(nx * 31 + ny)
    y, x = np.mgrid[0:ny, 0:nx].astype(np.float64)
    sign = np.where(rng.random((ny, nx)) < 0.5, -1.0, 1.0)
    if kind == "gauss":  # a few columns wide: the tails leave 2^-58 of the peak's strip behind
        return np.exp(-((x - nx // 2) ** 2 + (y - ny // 2) ** 2) / 50.0).clip(1e-130)
    if kind == "binades":
        return sign * np.exp2(-rng.uniform(0, 90, (ny, nx)))
    if kind == "columns":
        return sign * np.exp2(-1.5 * x) * rng.uniform(1, 2, (ny, nx))
    if kind == "blocks":  # zero regions beside uniform ones
        return rng.uniform(-1, 1, (ny, nx)) * (((x // 23) + (y // 7)) % 2)
    b = np.where((x + y) % 2 == 0, 1.0, -1.0) * 2.0 ** -60 * (kind == "checker")
    b[ny // 3, nx // 3] = 1.0
    return b


def _stencil(u, sign=-1):
    y = 4 * u
    y[:, 1:] += sign * u[:, :-1]
    y[:, :-1] += sign * u[:, 1:]
    y[1:] += sign * u[:-1]
    y[:-1] += sign * u[1:]
    return y


def _two_steps(b):
    """x after two steps, the S of each point, the largest ratio of the dot products."""
    b = b.astype(np.longdouble)
    g0, ab = (b * b).sum(), _stencil(b)
    a0 = g0 / (b * ab).sum()
    r = b - a0 * ab
    b1 = (r * r).sum() / g0
    p = r + b1 * b
    ap = _stencil(p)
    a1 = (r * r).sum() / (p * ap).sum()
    s = a0 * abs(b) + a1 * (abs(b) + a0 * _stencil(abs(b), 1) + b1 * abs(b))
    k = [(abs(b * ab)).sum() / (b * ab).sum(), (abs(p * ap)).sum() / (p * ap).sum(),
         a0 * np.linalg.norm(ab.astype(np.float64)) / np.linalg.norm(r.astype(np.float64))]
    return a0 * b + a1 * p, s, max(k)


@pytest.mark.parametrize("variant", ["classic", "newcg"])
@pytest.mark.parametrize("route", list(ROUTES))
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx,ny", [(64, 40), (131, 33), (258, 97), (400, 130)])
def test_small_values_beside_large_ones(variant, route, kind, nx, ny):
    b = _data(kind, nx, ny)
    ref, s, k = _two_steps(b)
    assert k <= 8
    t = torch.zeros((ny, (nx + 3) // 4 * 4), dtype=torch.float64)
    t[:, :nx] = torch.from_numpy(b)
    x, info = lap5cg.cg_solve(t.cuda(), tol=0.0, maxit=2, variant=variant, nx=nx,
                              opts=lap5cg.default_opts(**ROUTES[route]))
    assert lap5cg.decode_info(info)[0]["iters"] == 2
    assert (abs(x.cpu().numpy()[:, :nx] - ref) <= 2.0 ** -34 * s).all()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx,ny", [(153, 309), (400, 613)])
def test_multigrid_iterates_match_the_oracle(kind, nx, ny):
    b = _data(kind, nx, ny)
    for k in (1, 3):
        x, info = lap5cg.cg_solve(torch.from_numpy(b).cuda(), tol=0.0, maxit=k, precision="mg_f64")
        xo, io = oracle.cg_pcg(b, tol=0.0, maxit=k)
        assert lap5cg.decode_info(info)[0]["iters"] == io["iters"]
        assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-11 * np.linalg.norm(xo)

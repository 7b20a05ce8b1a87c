"""The binary64 stencil in fixed point (row-ring kernels) against CG in extended
precision: no further from it than the FP64 stencil of the register-march
kernels.

Both kernels run k iterations of Algorithm 1 (and 2) on data of different
dynamic range: uniform, smooth, a single spike (the operand's rows then span many
binades), rows scaled from 1 to 2^-60.  The reference is Algorithm 1 in numpy's
longdouble (64-bit significands or more).  The fixed-point sum's error is below
the FP64 sum's in the 2-norm, but the iterates' errors also hold the scalars' and
updates' roundings, equally in both and random: a factor of 2, plus 4 units of
2^-53 an iteration, bounds the comparison of two such errors."""
import numpy as np
import pytest
import torch

import paper_1803_03797_gb300 as lap5cg

pytestmark = pytest.mark.gpu


def _stencil(u):
    y = 4 * u
    y[:, 1:] -= u[:, :-1]
    y[:, :-1] -= u[:, 1:]
    y[1:] -= u[:-1]
    y[:-1] -= u[1:]
    return y


def _cg(b, k):
    b = b.astype(np.longdouble)
    x, r = np.zeros_like(b), b.copy()
    p, g = r.copy(), (b * b).sum()
    for _ in range(k):
        z = _stencil(p)
        a = g / (p * z).sum()
        x += a * p
        r -= a * z
        g, old = (r * r).sum(), g
        p = r + (g / old) * p
    return x


def _data(kind, nx, ny):
    rng = np.random.default_rng(nx + ny)
    b = rng.uniform(-1, 1, (ny, nx))
    if kind == "smooth":
        b = np.sin(np.arange(1, ny + 1) * np.pi / (ny + 1))[:, None] * np.sin(np.arange(1, nx + 1) * np.pi / (nx + 1))
        b += 1e-3 * rng.standard_normal((ny, nx))
    elif kind == "spike":
        b *= 0
        b[ny // 3, nx // 3] = 1.0
    elif kind == "rows":
        b *= np.exp2(-np.arange(ny) * 60.0 / ny)[:, None]
    return b


@pytest.mark.parametrize("variant", ["classic", "newcg"])
@pytest.mark.parametrize("kind", ["uniform", "smooth", "spike", "rows"])
@pytest.mark.parametrize("nx,ny", [(64, 40), (130, 33), (258, 97), (400, 130)])
def test_fixed_point_stencil_is_as_exact_as_fp64(variant, kind, nx, ny):
    k, b = 12, _data(kind, nx, ny)
    ref = _cg(b, k)
    ld = (nx + 3) // 4 * 4
    t = torch.zeros((ny, ld), dtype=torch.float64)
    t[:, :nx] = torch.from_numpy(b)
    err = {}
    for name, slots in (("fixed", 4), ("fp64", -1)):
        x, info = lap5cg.cg_solve(t.cuda(), tol=0.0, maxit=k, variant=variant, nx=nx,
                                  opts=lap5cg.default_opts(ring_slots=slots, resident=-1))
        assert lap5cg.decode_info(info)[0]["iters"] == k
        err[name] = float(np.linalg.norm(x.cpu().numpy()[:, :nx] - ref) / np.linalg.norm(ref))
    assert err["fixed"] <= 2 * err["fp64"] + 4 * k * 2.0 ** -53, err


@pytest.mark.parametrize("bad", [float("inf"), float("nan"), 1e308])
def test_values_outside_the_fixed_point_range(bad):
    b = torch.rand(40, 128, dtype=torch.float64, device="cuda")
    b[7, 9] = bad
    for slots in (4, -1):
        _, info = lap5cg.cg_solve(b, tol=1e-8, maxit=50, opts=lap5cg.default_opts(ring_slots=slots, resident=-1))
        assert lap5cg.decode_info(info)[0]["status"] == lap5cg.ERR_NONFINITE

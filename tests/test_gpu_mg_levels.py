"""The multigrid V-cycle's middle levels (one kernel, rows split over the CTAs)
against the oracle's V-cycle PCG, at the sizes where the split changes: the first
grid with a distributed level, one row a CTA, several rows a CTA, more CTAs on a
coarse level than the finer one has, one-row and one-column coarsest levels, odd
and even sides.

Binary64: the bound of the oracle comparison of the other multigrid tests (1e-11
after 1, 3 and 6 iterations).  Binary32 V-cycle: the same number of iterations to
1e-8 within 2 and the true residual."""
import pytest
import torch

import lap5_inputs as gen
import oracle
import paper_1803_03797_gb300 as lap5cg
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

SHAPES = [(70, 69), (67, 140), (153, 309), (310, 152), (611, 70), (3, 2000), (2000, 9), (400, 613)]


def _solve(b, nx, precision, **kw):
    x, info = lap5cg.cg_solve(torch.from_numpy(b).cuda(), precision=precision, nx=nx, **kw)
    return x.cpu().numpy()[:, :nx], lap5cg.decode_info(info)[0]


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_binary64_iterates_match_the_oracle(nx, ny):
    b = gen.uniform_rhs(nx, ny, seed=nx + ny)
    for k in (1, 3, 6):
        x, rec = _solve(b, nx, "mg_f64", tol=0.0, maxit=k)
        xo, io = oracle.cg_pcg(b, tol=0.0, maxit=k)
        assert rec["iters"] == io["iters"] and rec["status"] == io["status"]
        assert rel_err(x, xo) <= 1e-11


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_binary32_vcycle_converges_like_binary64(nx, ny):
    b = gen.uniform_rhs(nx, ny, seed=nx + ny)
    _, r32 = _solve(b, nx, "mg_f32", tol=1e-8, maxit=200)
    _, r64 = _solve(b, nx, "mg_f64", tol=1e-8, maxit=200)
    assert r32["status"] == r64["status"] == lap5cg.OK
    assert abs(r32["iters"] - r64["iters"]) <= 2
    assert max(r32["relres_true"], r64["relres_true"]) <= 3e-8

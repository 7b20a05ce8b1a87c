"""Chip-resident solves (state vectors in the SMs' registers and shared memory)
against the streaming kernels, at the sizes where the decomposition changes:
one CTA, two rows a CTA and the first size with three, ragged last lane
vectors, a last item that only some warps have, the most items a thread, and the
first grid that no longer fits (which must take the streaming kernels).

The two kernels differ in the order of their dot products' sums only.  k <= 30
iterations from the same data then stay within 1e-10 relative (the bound of
the other kernel pairs' tests: 30 iterations times a few units in the last
place of the scalars, amplified by the condition of the iteration); binary32
within 1e-4."""
import numpy as np
import pytest
import torch

import lap5_inputs as gen
import paper_1803_03797_gb300 as lap5cg
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

SHAPES = [(16, 2), (17, 3), (31, 305), (33, 304), (64, 306), (129, 303), (100, 100), (1024, 24), (1026, 61),
          (513, 457), (515, 610), (2048, 302), (800, 912), (1024, 1064), (1022, 1066), (1500, 1500)]


def _solve(b, nx, **kw):
    opts = lap5cg.default_opts(**kw.pop("opts", {}))
    x, info = lap5cg.cg_solve(b, nx=nx, opts=opts, **kw)
    return x.cpu().numpy()[:, :nx].astype(np.float64), lap5cg.decode_info(info)[0]


def _rhs(nx, ny, dtype):
    return torch.from_numpy(gen.uniform_rhs(nx, ny, seed=nx + 7 * ny, ld=(nx + 3) // 4 * 4)).to("cuda", dtype)


@pytest.mark.parametrize("precision,variant,tol", [("f64", "classic", 1e-10), ("f64", "newcg", 1e-10),
                                                   ("f32", "classic", 1e-4)])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_resident_matches_streaming(precision, variant, tol, nx, ny):
    b = _rhs(nx, ny, torch.float32 if precision == "f32" else torch.float64)
    k = min(30, nx * ny // 2)
    kw = dict(tol=0.0, maxit=k, variant=variant, precision=precision)
    xa, ra = _solve(b, nx, **kw)
    xb, rb = _solve(b, nx, opts=dict(resident=-1), **kw)
    assert ra["status"] == rb["status"] and ra["iters"] == rb["iters"] == k
    assert rel_err(xa, xb) <= tol


@pytest.mark.parametrize("nx,ny", [s for s in SHAPES if s[0] * s[1] <= 800 * 912])
def test_resident_refinement_matches_streaming(nx, ny):
    b = _rhs(nx, ny, torch.float64)
    kw = dict(tol=1e-10, maxit=100000, precision="ir_f32")
    xa, ra = _solve(b, nx, **kw)
    xb, rb = _solve(b, nx, opts=dict(resident=-1), **kw)
    assert ra["status"] == rb["status"] == lap5cg.OK
    # the bounds of the refinement's parity with the oracle
    assert abs(ra["outer_iters"] - rb["outer_iters"]) <= 1
    assert abs(ra["iters"] - rb["iters"]) <= max(2, 0.01 * rb["iters"])
    assert ra["relres_true"] <= 1e-10


@pytest.mark.parametrize("variant", ["classic", "newcg"])
@pytest.mark.parametrize("scale", [2.0 ** -470, 2.0 ** -330, 2.0 ** 330, 2.0 ** 500])
def test_resident_sums_over_the_exponent_range(variant, scale):
    # powers of two scale every quantity exactly; near the ends of the range the
    # sums leave the fixed-point path (products reach 2^-970 .. 2^1022)
    b = _rhs(200, 150, torch.float64)
    x, r = _solve(b, 200, tol=1e-6, maxit=2000, variant=variant)
    xs, rs = _solve(b * scale, 200, tol=1e-6, maxit=2000, variant=variant)
    assert r["status"] == rs["status"] == lap5cg.OK and abs(r["iters"] - rs["iters"]) <= 1
    assert rel_err(xs / scale, x) <= 1e-6


def test_resident_time_limit_ends_in_a_status():
    # a 50 ns limit on every wait; waits poll L2, so all CTAs leave within a few
    # microseconds and the context stays usable
    b = _rhs(700, 700, torch.float64)
    _, r = _solve(b, 700, tol=1e-10, maxit=5000, opts=dict(timeout_s=5e-8))
    assert r["status"] == lap5cg.ERR_SYNC_TIMEOUT
    _, r = _solve(b, 700, tol=1e-6, maxit=5000)
    assert r["status"] == lap5cg.OK


@pytest.mark.parametrize("precision,variant", [("f64", "classic"), ("f64", "newcg"), ("f32", "classic")])
def test_resident_batch_matches_streaming(precision, variant):
    # sides for every team size the chip is split into, fewer rows than a team has
    # CTAs, and one that no team holds
    shapes = [(64, 64), (40, 9), (700, 5), (300, 300), (512, 400), (600, 610), (1040, 1000), (1600, 1500)]
    dtype = torch.float32 if precision == "f32" else torch.float64
    bs = [_rhs(nx, ny, dtype) for nx, ny in shapes]
    nxs = [nx for nx, _ in shapes]
    kw = dict(tol=0.0, maxit=30, variant=variant, precision=precision, nx_list=nxs)
    xa, ia = lap5cg.cg_solve_batched(bs, **kw)
    xb, ib = lap5cg.cg_solve_batched(bs, opts=lap5cg.default_opts(resident=-1), **kw)
    for nx, a, b, ra, rb in zip(nxs, xa, xb, lap5cg.decode_info(ia), lap5cg.decode_info(ib)):
        assert ra["status"] == rb["status"] and ra["iters"] == rb["iters"] == 30
        assert rel_err(a.double().cpu().numpy()[:, :nx], b.double().cpu().numpy()[:, :nx]) <= (
            1e-4 if precision == "f32" else 1e-10)

"""Streaming solves of small grids (options that the chip-resident kernels leave to them):
the default launch is no slower than the best of some explicit warp counts (within
15 %, the spread of repeated timings and of neighbouring sizes), and gives the same
iterates within the bound of the other launch-shape tests."""
import pytest
import torch

import lap5_inputs as gen
import paper_1803_03797_gb300 as lap5cg
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

MODES = {"classic": ("classic", dict(resident=-1)), "newcg": ("newcg", dict(resident=-1)),
         "replaced": ("newcg", dict(rr_period=10)), "stabilised": ("newcg", dict(stabilized=1))}


def _solve(b, mode, warps):
    variant, kw = MODES[mode]
    opts = lap5cg.default_opts(warps_per_cta=warps, **kw)
    best = float("inf")
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        x, _ = lap5cg.cg_solve(b, tol=0.0, maxit=100, variant=variant, opts=opts)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("n", [64, 150, 300, 400])
def test_default_warps_are_the_fast_ones(mode, n):
    b = torch.from_numpy(gen.uniform_rhs(n, n, seed=n)).cuda()
    assert _solve(b, mode, 0) <= 1.15 * min(_solve(b, mode, w) for w in (5, 8, 16))


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("nx,ny", [(1, 9), (64, 64), (129, 303), (400, 400), (1000, 60)])
def test_same_iterates_as_16_warps(mode, nx, ny):
    variant, kw = MODES[mode]
    b = torch.from_numpy(gen.uniform_rhs(nx, ny, seed=nx + ny, ld=gen.pitch(nx, 8))).cuda()
    k = min(30, nx * ny - 1)
    xs = [lap5cg.cg_solve(b, tol=0.0, maxit=k, variant=variant, nx=nx,
                          opts=lap5cg.default_opts(warps_per_cta=w, **kw))[0].cpu().numpy()[:, :nx] for w in (0, 16)]
    assert rel_err(xs[0], xs[1]) <= 1e-10

"""A multigrid solve that breaks down leaves x as it was in every row, and the next solve
in the same workspace is not affected.

Breakdowns: a smooth right-hand side near the end of binary64's range ((b, b) is
finite, (r, z) overflows), and one beyond binary32's range for a binary32 V-cycle.
Grids with the single-CTA levels only and with the middle levels split over the SMs."""
import pytest
import torch

import lap5_inputs as gen
import paper_1803_03797_gb300 as lap5cg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(70, 69), (200, 150), (1000, 700)])
@pytest.mark.parametrize("precision", ["mg_f64", "mg_f32"])
def test_breakdown_leaves_x_and_the_workspace_usable(precision, nx, ny):
    # binary64: (b, b) = scale^2 (nx + 1) (ny + 1) / 4 = 2^1022, and (r, z) is larger by 1 / lambda_min of the
    # lowest mode, 250 at least (the V-cycle reproduces it within a factor of two): beyond 2^1024
    scale = 2.0 ** 512 / ((nx + 1) * (ny + 1)) ** 0.5 if precision == "mg_f64" else 2.0 ** 200
    big = torch.from_numpy(gen.sine_mode(nx, ny, 1, 1) * scale).cuda()
    b = torch.from_numpy(gen.uniform_rhs(nx, ny, seed=nx)).cuda()
    x0 = torch.from_numpy(gen.uniform_rhs(nx, ny, seed=ny)).cuda()
    ws = torch.empty(lap5cg.workspace_size(nx, ny, nx, "classic", precision), dtype=torch.uint8, device="cuda")
    kw = dict(precision=precision, workspace=ws)
    first, _ = lap5cg.cg_solve(b, tol=1e-10, maxit=200, **kw)
    for _ in range(20):
        x, info = lap5cg.cg_solve(big, x0=x0, tol=1e-10, maxit=50, **kw)
        rec = lap5cg.decode_info(info)[0]
        assert rec["status"] == lap5cg.ERR_BREAKDOWN and rec["iters"] == 0
        assert torch.equal(x, x0)
        x, info = lap5cg.cg_solve(b, tol=1e-10, maxit=200, **kw)
        assert lap5cg.decode_info(info)[0]["status"] == lap5cg.OK
        assert torch.equal(x, first)

"""opts.timeout_s bounds the waits of batched teams and of the multigrid's middle levels:
with a 50 ns limit every exchange (an L2 round trip at least) runs out, the solve
ends with a status, every instance has its record, and the context and the
workspace stay usable.  Without an option the limit is 2 s."""
import pytest
import torch

import lap5_inputs as gen
import paper_1803_03797_gb300 as lap5cg

pytestmark = pytest.mark.gpu


def _rhs(nx, ny):
    return torch.from_numpy(gen.uniform_rhs(nx, ny, seed=nx + ny)).cuda()


@pytest.mark.parametrize("precision,variant", [("f64", "classic"), ("f64", "newcg"), ("ir_f32", "classic")])
def test_batched_teams(precision, variant):
    shapes = [(512, 500), (400, 300), (256, 260)] * 12
    bs = [_rhs(nx, ny) for nx, ny in shapes]
    nxs, nys = [s[0] for s in shapes], [s[1] for s in shapes]
    ws = torch.empty(lap5cg.batched_workspace_size(nxs, nys, nxs, variant, precision), dtype=torch.uint8, device="cuda")
    info = torch.full((len(bs) * lap5cg.INFO_BYTES,), 0x7f, dtype=torch.uint8, device="cuda")
    kw = dict(tol=1e-6, maxit=5000, variant=variant, precision=precision, workspace=ws)
    _, info = lap5cg.cg_solve_batched(bs, opts=lap5cg.default_opts(timeout_s=5e-8), info=info, **kw)
    assert {r["status"] for r in lap5cg.decode_info(info)} == {lap5cg.ERR_SYNC_TIMEOUT}
    _, info = lap5cg.cg_solve_batched(bs, **kw)
    assert {r["status"] for r in lap5cg.decode_info(info)} == {lap5cg.OK}


@pytest.mark.parametrize("precision", ["mg_f32", "mg_f64"])
def test_multigrid_middle_levels(precision):
    nx, ny = 1000, 700
    b, x0 = _rhs(nx, ny), _rhs(ny, nx).reshape(ny, nx)
    ws = torch.empty(lap5cg.workspace_size(nx, ny, nx, "classic", precision), dtype=torch.uint8, device="cuda")
    kw = dict(tol=1e-8, maxit=100, precision=precision, workspace=ws)
    for _ in range(3):  # the limit is the call's, not the cached graph's
        x, info = lap5cg.cg_solve(b, x0=x0, opts=lap5cg.default_opts(timeout_s=5e-8), **kw)
        rec = lap5cg.decode_info(info)[0]
        assert rec["status"] == lap5cg.ERR_SYNC_TIMEOUT and rec["iters"] == 0
        assert torch.equal(x, x0)
        _, info = lap5cg.cg_solve(b, x0=x0, **kw)
        assert lap5cg.decode_info(info)[0]["status"] == lap5cg.OK

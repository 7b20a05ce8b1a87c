"""Solves whose warp units are a few rows tall: either side of the shortest unit
that keeps the wide lanes (eight binary32 or four binary64 columns), against the
FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lap5_inputs as gen  # noqa: E402
import oracle  # noqa: E402
import paper_1803_03797_gb300 as lap5cg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [3, 4, 5, 7, 8])
@pytest.mark.parametrize("precision", ["ir_f32", "ir_bf16pr", "f64"])
def test_short_units_match_oracle(precision, rows):
    # 8 CTAs of 16 warps on 5 strips of 256 (f64: 128) columns: 25 units a strip, `rows` rows each
    nx, ny, tol = 1030 if precision != "f64" else 516, 25 * rows, 1e-10
    b = gen.uniform_rhs(nx, ny, seed=7, ld=gen.pitch(nx, 32))
    x, info = lap5cg.cg_solve(torch.from_numpy(b).cuda(), tol=tol, maxit=10 ** 6, precision=precision, nx=nx,
                              opts=lap5cg.default_opts(ctas=8))
    rec = lap5cg.decode_info(info)[0]
    assert rec["status"] == lap5cg.OK and rec["relres_true"] <= tol, rec
    xo, _ = oracle.cg_classic(b, tol=1e-13, maxit=10 ** 6, nx=nx)
    x, xo = x.cpu().numpy()[:, :nx], xo[:, :nx]
    # both residuals are below tol |b|: |x - x*| <= kappa (tol + 1e-13) |x*| in the 2-norm
    assert np.linalg.norm(x - xo) <= gen.condition_number(nx, ny) * 2 * tol * np.linalg.norm(xo)

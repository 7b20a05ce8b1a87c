"""Reproducible mode: the default launch is no slower than the best of the explicit warp
counts (within 15 %, the spread of repeated timings and of neighbouring sizes)."""
import pytest
import torch

import lap5_inputs as gen
import paper_1803_03797_gb300 as lap5cg

pytestmark = pytest.mark.gpu


def _ms(b, variant, warps):
    opts = lap5cg.default_opts(reproducible=1, warps_per_cta=warps)
    best = float("inf")
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        lap5cg.cg_solve(b, tol=0.0, maxit=100, variant=variant, opts=opts)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.parametrize("variant", ["classic", "newcg"])
@pytest.mark.parametrize("n", [100, 500, 1500])
def test_default_warps_are_the_fast_ones(variant, n):
    b = torch.from_numpy(gen.uniform_rhs(n, n, seed=n)).cuda()
    assert _ms(b, variant, 0) <= 1.15 * min(_ms(b, variant, w) for w in (4, 8, 16))

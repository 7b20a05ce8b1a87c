"""The cluster-resident kernels (small.cu), which default calls reach for binary32 NewCG
and for what the chip-resident kernels leave: asked for through team_ctas, for
every precision, variant and cluster size, single and batched, against the oracle.

team_ctas chooses another kernel than the default call and than the streaming one;
30 iterations on data without symmetry round differently in binary64, so the bits of x
show which one ran.  (Binary32 iterates agree to the bit, the sums being exact
enough; there the time of an iteration tells, which differs by a factor of two and more.)"""
import numpy as np
import pytest
import torch

import lap5_inputs as gen
import oracle
import paper_1803_03797_gb300 as lap5cg
from tests.helpers import rel_err

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16), (100, 100), (1, 7), (17, 300), (250, 120), (255, 31)]


def _solve(b, nx, **kw):
    opts = lap5cg.default_opts(**kw.pop("opts"))
    x, info = lap5cg.cg_solve(b, nx=nx, opts=opts, **kw)
    return x, lap5cg.decode_info(info)[0]


@pytest.mark.parametrize("variant", ["classic", "newcg"])
@pytest.mark.parametrize("team", [1, 4, 16])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_binary64_matches_the_oracle(variant, team, nx, ny):
    b = gen.uniform_rhs(nx, ny, seed=5 * nx + ny, ld=gen.pitch(nx, 8))
    t = torch.from_numpy(b).cuda()
    k = min(30, nx * ny - 1)
    x, rec = _solve(t, nx, tol=0.0, maxit=k, variant=variant, opts=dict(team_ctas=team))
    xo, io = oracle.cg_solve(b, variant=variant, tol=0.0, maxit=k, nx=nx)
    assert rec["iters"] == io["iters"]
    assert rel_err(x.cpu().numpy()[:, :nx], xo[:, :nx]) <= 1e-10
    x, rec = _solve(t, nx, tol=1e-10, maxit=20000, variant=variant, opts=dict(team_ctas=team))
    _, io = oracle.cg_solve(b, variant=variant, tol=1e-10, maxit=20000, nx=nx)
    assert rec["status"] == lap5cg.OK and abs(rec["iters"] - io["iters"]) <= 2
    assert rec["relres_true"] <= 3 * max(io["relres_true"], 1e-10)


@pytest.mark.parametrize("variant,tol", [("classic", 1e-4), ("newcg", 1e-3)])
@pytest.mark.parametrize("team", [0, 1, 4, 16])
@pytest.mark.parametrize("nx,ny", [(100, 100), (31, 90), (200, 200)])
def test_binary32_matches_the_oracle(variant, tol, team, nx, ny):
    b = gen.uniform_rhs(nx, ny, seed=nx + 3 * ny, ld=gen.pitch(nx, 8)).astype(np.float32)
    x, _ = _solve(torch.from_numpy(b).cuda(), nx, tol=0.0, maxit=30, variant=variant, precision="f32",
                  opts=dict(team_ctas=team))
    xo, _ = oracle.cg_solve(b.astype(np.float64), variant=variant, tol=0.0, maxit=30, nx=nx)
    assert rel_err(x.cpu().numpy().astype(np.float64)[:, :nx], xo[:, :nx]) <= tol


@pytest.mark.parametrize("variant", ["classic", "newcg"])
@pytest.mark.parametrize("team", [4, 16])
def test_a_batch_of_more_than_one_launch(variant, team):
    rng = np.random.default_rng(23)
    shapes = [(int(rng.integers(16, 90)), int(rng.integers(16, 90))) for _ in range(100)]
    shapes[10:10] = [(700, 300), (300, 700)]  # left to the team kernel
    bs = [gen.uniform_rhs(nx, ny, seed=900 + k, ld=gen.pitch(nx, 8, 32)) for k, (nx, ny) in enumerate(shapes)]
    xs, info = lap5cg.cg_solve_batched([torch.from_numpy(b).cuda() for b in bs], tol=1e-10, maxit=100000,
                                       variant=variant, precision="f64", nx_list=[s[0] for s in shapes],
                                       opts=lap5cg.default_opts(team_ctas=team))
    for k, (rec, (nx, ny)) in enumerate(zip(lap5cg.decode_info(info), shapes)):
        xo, io = oracle.cg_solve(bs[k], variant=variant, tol=1e-10, maxit=100000, nx=nx)
        assert rec["status"] == lap5cg.OK and abs(rec["iters"] - io["iters"]) <= 2, (k, rec)
        bound = gen.condition_number(nx, ny) * max(1e-10, io["relres_true"])
        assert rel_err(xs[k].cpu().numpy()[:, :nx], xo[:, :nx]) <= bound, k


def _bits(b, nx, variant, **opts):
    return _solve(b, nx, tol=0.0, maxit=30, variant=variant, opts=opts)[0]


# the chip-resident kernels' range: from the smallest grids to the largest that fit; and
# beyond it, or where flat grids are left to the streaming kernels
@pytest.mark.parametrize("variant,nx,ny,resident", [
    ("classic", 64, 40, True), ("classic", 1024, 1064, True), ("classic", 1100, 1100, False),
    ("newcg", 100, 100, True), ("newcg", 680, 608, True), ("newcg", 700, 700, False),
    ("classic", 3000, 100, False), ("classic", 3400, 304, True)])
def test_which_binary64_grids_are_chip_resident(variant, nx, ny, resident):
    b = torch.from_numpy(gen.uniform_rhs(nx, ny, seed=nx + ny)).cuda()
    default, streaming = (_bits(b, nx, variant, resident=r) for r in (0, -1))
    assert torch.equal(default, _bits(b, nx, variant, resident=0))
    assert torch.equal(default, streaming) == (not resident)


@pytest.mark.parametrize("n,resident", [(100, True), (1400, True), (1500, False)])
def test_which_binary32_grids_are_chip_resident(n, resident):
    b = torch.from_numpy(gen.uniform_rhs(n, n, seed=n)).to("cuda", torch.float32)
    ms = {}
    for r in (0, -1):
        opts = lap5cg.default_opts(resident=r)
        ms[r] = float("inf")
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            lap5cg.cg_solve(b, tol=0.0, maxit=300, precision="f32", opts=opts)
            e1.record()
            torch.cuda.synchronize()
            ms[r] = min(ms[r], e0.elapsed_time(e1))
    assert (ms[0] < 0.75 * ms[-1]) == resident, ms


@pytest.mark.parametrize("variant", ["classic", "newcg"])
def test_team_ctas_takes_the_cluster_kernel(variant):
    b = torch.from_numpy(gen.uniform_rhs(100, 90, seed=8)).cuda()
    default, streaming, cluster = (_bits(b, 100, variant, **o) for o in ({}, dict(resident=-1), dict(team_ctas=16)))
    assert not torch.equal(cluster, default) and not torch.equal(cluster, streaming)

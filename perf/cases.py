"""The measured cases of lap5cg: what its users have it do, through the
package's public calls.

A case is one of

  apply     y = A x (residual checks, operators of outer solvers)
  solve     one right-hand side or a stack, to a tolerance or a fixed number
            of iterations
  batched   many grids of different sizes in one call
  grad      a differentiable solve with a quadratic loss, forward and adjoint

Sizes are those of this repository's workloads (the paper's 100 x 100, the
4096^2 and 8192^2 benchmarks, the batched sides, the 2048^2 differentiable
solve) or generic ones between them; odd sides and padded pitches occur as they
do in a user's grids.
"""
import math
import random

import torch

import paper_1803_03797_gb300 as lap5cg

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # the smallest call: the operator on the paper's largest grid, where launch and call overhead are the time
        {"name": "apply_f64_100", "kind": "apply", "nx": 100, "ny": 100, "ld": 100, "dtype": "f64"},
        # the operator on the largest grid, in the storage type a preconditioner keeps its fields in
        {"name": "apply_bf16_8192", "kind": "apply", "nx": 8192, "ny": 8192, "ld": 8192, "dtype": "bf16"},
        # the paper's largest grid with the paper's method (Algorithm 2), to the default tolerance
        solve("newcg_f64_100", 100, 100, "newcg", "f64", tol=1e-10),
        # a ragged grid of a few hundred points a side (one subdomain of a larger problem) with classic CG
        solve("classic_f64_417x333", 417, 333, "classic", "f64", tol=1e-10),
        # the headline workload, 4096^2 in binary64: each algorithm for a fixed number of iterations
        solve("classic_f64_4096", 4096, 4096, "classic", "f64", iters=200, rhs="manufactured"),
        solve("newcg_f64_4096", 4096, 4096, "newcg", "f64", iters=200, rhs="manufactured"),
        # the binary32 iteration on the largest grid (a smoother, or the first phase of a longer solve)
        solve("classic_f32_8192", 8192, 8192, "classic", "f32", iters=100),
        # mixed precision on a middle-sized grid: binary64 accuracy at binary32 speed
        solve("ir_f32_1024", 1024, 1024, "classic", "ir_f32", tol=1e-10),
        # time to solution at the headline size: the preconditioned solve a production user would pick
        solve("mg_f32_4096", 4096, 4096, "classic", "mg_f32", tol=1e-10, rhs="manufactured"),
        # the preconditioned solve in binary64 throughout on an odd grid with a padded pitch
        solve("mg_f64_1500x1003", 1500, 1003, "classic", "mg_f64", tol=1e-10, ld=1504),
        # many grids of different sizes in one call (a sweep over subdomains or parameters)
        {"name": "batched_ir_f32_48", "kind": "batched", "count": 48, "lo": 64, "hi": 512, "shapes": 4,
         "precision": "ir_f32", "tol": 1e-10},
        # a differentiable solve inside a training loop: forward, loss and adjoint
        {"name": "grad_mg_f32_2048x2", "kind": "grad", "nx": 2048, "ny": 2048, "ld": 2048, "nrhs": 2,
         "precision": "mg_f32", "tol": 1e-10},
    ]


def solve(name, nx, ny, variant, precision, tol=0.0, iters=0, ld=None, rhs="uniform", nrhs=1):
    """A solve to the relative residual tol, or (tol = 0) of exactly iters iterations."""
    c = {"kind": "solve", "nx": nx, "ny": ny, "ld": nx if ld is None else ld, "variant": variant,
         "precision": precision, "tol": tol, "iters": iters, "rhs": rhs, "nrhs": nrhs}
    return c if name is None else dict(c, name=name)


def draw(rng):
    kind = rng.choice(["apply", "apply", "krylov", "krylov", "fixed", "fixed", "fixed", "ir", "mg", "mg", "batched",
                       "grad"])
    if kind == "apply":
        nx, ny = sides(rng, 16, 8192)
        return {"kind": "apply", "nx": nx, "ny": ny, "ld": pitch(rng, nx), "dtype": rng.choice(["f64", "f32", "bf16"])}
    if kind == "krylov":  # small and middle-sized grids, to the default tolerance
        variant = rng.choice(["classic", "newcg"])
        nx, ny = sides(rng, 16, 128 if variant == "newcg" else 700)
        return solve(None, nx, ny, variant, "f64", tol=1e-10, ld=pitch(rng, nx))
    if kind == "fixed":  # large grids, a fixed number of iterations
        variant, precision = rng.choice([("classic", "f64"), ("newcg", "f64"), ("classic", "f32")])
        nx, ny = sides(rng, 700, 4096 if precision == "f64" else 8192)
        return solve(None, nx, ny, variant, precision, iters=rng.randint(50, 100), ld=pitch(rng, nx),
                     rhs=rng.choice(["uniform", "manufactured"]))
    if kind == "ir":
        nx, ny = sides(rng, 64, 1024)
        return solve(None, nx, ny, "classic", "ir_f32", tol=1e-10, ld=pitch(rng, nx))
    if kind == "mg":
        nx, ny = sides(rng, 64, 4096)
        return solve(None, nx, ny, "classic", rng.choice(["mg_f32", "mg_f64"]), tol=1e-10, ld=pitch(rng, nx),
                     rhs=rng.choice(["uniform", "manufactured"]), nrhs=rng.choice([1, 1, 2]))
    if kind == "batched":
        return {"kind": "batched", "count": rng.randint(8, 48), "lo": 64, "hi": rng.randint(128, 512),
                "shapes": rng.randint(5, 1 << 20), "precision": rng.choice(["ir_f32", "ir_f32", "f64"]), "tol": 1e-10}
    nx, ny = sides(rng, 128, 2048)
    return {"kind": "grad", "nx": nx, "ny": ny, "ld": nx, "nrhs": rng.randint(1, 4), "precision": "mg_f32",
            "tol": 1e-10}


def sides(rng, lo, hi):
    """Two sides spread over the logarithm of [lo, hi], at most a factor of four apart."""
    nx = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ny = nx * math.exp(rng.uniform(-math.log(4), math.log(4)))
    return min(hi, max(lo, int(nx))), min(hi, max(lo, int(ny)))


def pitch(rng, nx):
    """The row pitch: mostly nx itself, else nx rounded up to 8 elements."""
    return nx if rng.random() < 0.7 else (nx + 7) // 8 * 8


def batch_shapes(case):
    """(nx, ny, ld) of each grid of a batched case: sides uniform in [lo, hi], pitches multiples of 4."""
    rng = random.Random(case["shapes"])
    got = []
    for _ in range(case["count"]):
        nx, ny = rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"])
        got.append((nx, ny, (nx + 3) // 4 * 4))
    return got


def uniform(gen, nx, ny, ld, dtype, nrhs=1):
    """U[-1, 1), padding columns zero; (ny, ld), or (nrhs, ny, ld) for a stack."""
    t = torch.zeros((nrhs, ny, ld), dtype=torch.float64, device="cuda")
    t[:, :, :nx] = torch.rand((nrhs, ny, nx), dtype=torch.float64, device="cuda", generator=gen) * 2 - 1
    t = t.to(dtype)
    return t[0] if nrhs == 1 else t


def manufactured(gen, nx, ny, ld, dtype, nrhs=1):
    """The lowest mode's right-hand side plus noise: A u* + 1e-3 N(0, 1), u* = sin(pi x) sin(pi y)."""
    i = torch.arange(1, nx + 1, dtype=torch.float64, device="cuda") * (math.pi / (nx + 1))
    j = torch.arange(1, ny + 1, dtype=torch.float64, device="cuda") * (math.pi / (ny + 1))
    lam = 4 - 2 * math.cos(math.pi / (nx + 1)) - 2 * math.cos(math.pi / (ny + 1))
    t = torch.zeros((nrhs, ny, ld), dtype=torch.float64, device="cuda")
    t[:, :, :nx] = lam * torch.sin(j)[:, None] * torch.sin(i)[None, :]
    t[:, :, :nx] += 1e-3 * torch.randn((nrhs, ny, nx), dtype=torch.float64, device="cuda", generator=gen)
    t = t.to(dtype)
    return t[0] if nrhs == 1 else t


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = {"case": case}
    if case["kind"] == "apply":
        s["x"] = uniform(gen, case["nx"], case["ny"], case["ld"], DTYPES[case["dtype"]])
    elif case["kind"] == "solve":
        dtype = torch.float32 if case["precision"] == "f32" else torch.float64
        rhs = manufactured if case["rhs"] == "manufactured" else uniform
        s["b"] = rhs(gen, case["nx"], case["ny"], case["ld"], dtype, case["nrhs"])
    elif case["kind"] == "batched":
        shapes = batch_shapes(case)
        s["bs"] = [uniform(gen, nx, ny, ld, torch.float64) for nx, ny, ld in shapes]
        s["nx"] = [nx for nx, _, _ in shapes]
    else:
        s["b"] = uniform(gen, case["nx"], case["ny"], case["ld"], torch.float64, case["nrhs"])
        s["target"] = torch.randn(s["b"].shape, dtype=torch.float64, device="cuda", generator=gen)
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "apply":
        return lap5cg.lap5_apply(state["x"], nx=case["nx"])
    if case["kind"] == "solve":
        x, _ = lap5cg.cg_solve(state["b"], tol=case["tol"], maxit=case["iters"] or 20000, variant=case["variant"],
                               precision=case["precision"], nx=case["nx"])
        return x
    if case["kind"] == "batched":
        xs, _ = lap5cg.cg_solve_batched(state["bs"], tol=case["tol"], precision=case["precision"],
                                        nx_list=state["nx"])
        return xs
    b = state["b"].detach().requires_grad_()
    x = lap5cg.solve(b, tol=case["tol"], precision=case["precision"])
    loss = 0.5 * (x - state["target"]).square().sum()
    loss.backward()
    return {"x": x.detach(), "loss": loss.detach(), "grad": b.grad}


def work(case):
    """Bytes and operations a pass cannot do without.

    apply: x read, y written, five operations a point.  A solve whose search
    vectors do not fit on the chip has to read and write r and p once an
    iteration (each iteration's scalars depend on all of the one before), with
    19 operations a point (stencil 5, two dot products 4, three updates 6, and
    the direction's halo); b is read and x written once.  Iteration counts to
    a tolerance are the usual ones of the method: about 3.3 times the longer
    side for CG to 1e-10, 1.5 times that in the refinement, 15 for the
    multigrid-preconditioned solve with about 60 operations a point more.
    """
    if case["kind"] == "batched":
        elem = 4 if case["precision"] == "ir_f32" else 8
        parts = [solve_work(nx, ny, elem, 8, 3.3 * max(nx, ny) * (1.5 if elem == 4 else 1.0), 1)
                 for nx, ny, _ in batch_shapes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n = case["nx"] * case["ny"]
    if case["kind"] == "apply":
        elem = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
        return {"bytes": 2 * elem * n, "flops": 5 * n}
    nrhs = case["nrhs"]
    if case["precision"].startswith("mg"):
        passes = 2 if case["kind"] == "grad" else 1
        elem = 4 if case["precision"] == "mg_f32" else 8
        # an iteration reads and writes r, p and the preconditioned residual, the last in the V-cycle's type
        return {"bytes": passes * nrhs * n * (16 + 15 * (32 + 2 * elem)), "flops": passes * nrhs * n * 15 * 79}
    io = 4 if case["precision"] == "f32" else 8
    elem = 8 if case["precision"] == "f64" else 4
    iters = case["iters"] or 3.3 * max(case["nx"], case["ny"]) * (1.5 if case["precision"] == "ir_f32" else 1.0)
    by, fl = solve_work(case["nx"], case["ny"], elem, io, iters, nrhs)
    return {"bytes": by, "flops": fl}


def solve_work(nx, ny, elem, io, iters, nrhs):
    n = nx * ny
    on_chip = 3 * elem * n <= 32 << 20  # r, p and x in the SMs' shared memory
    return (nrhs * n * (2 * io + (0 if on_chip else iters * 4 * elem)), nrhs * n * iters * 19)


# The same outputs in 64 bits, from plain torch.

def stencil64(x):
    y = 4 * x
    y[..., :, 1:] -= x[..., :, :-1]
    y[..., :, :-1] -= x[..., :, 1:]
    y[..., 1:, :] -= x[..., :-1, :]
    y[..., :-1, :] -= x[..., 1:, :]
    return y


def sine(x):
    """The type-I sine transform along the last dimension (its own inverse up to 2 / (n + 1))."""
    n = x.shape[-1]
    z = torch.zeros(x.shape[:-1] + (2 * (n + 1),), dtype=x.dtype, device=x.device)
    z[..., 1:n + 1] = x
    z[..., n + 2:] = -x.flip(-1)
    return torch.fft.rfft(z).imag[..., 1:n + 1] * -0.5


def direct64(b):
    """A^-1 b through the sine transforms that diagonalise A; b without padding."""
    ny, nx = b.shape[-2:]
    k = torch.arange(1, nx + 1, dtype=torch.float64, device=b.device) * (math.pi / (nx + 1))
    m = torch.arange(1, ny + 1, dtype=torch.float64, device=b.device) * (math.pi / (ny + 1))
    lam = 4 * torch.sin(k / 2).square()[None, :] + 4 * torch.sin(m / 2).square()[:, None]
    h = sine(sine(b).transpose(-1, -2)).transpose(-1, -2) / lam
    return sine(sine(h).transpose(-1, -2)).transpose(-1, -2) * (4.0 / ((nx + 1) * (ny + 1)))


def iterate64(b, iters):
    """x after iters steps of CG from zero (the iterates of both algorithms are the same in exact arithmetic)."""
    x, r = torch.zeros_like(b), b.clone()
    p, g = r.clone(), (b * b).sum()
    for _ in range(iters):
        z = stencil64(p)
        alpha = g / (p * z).sum()
        x += alpha * p
        r -= alpha * z
        g, old = (r * r).sum(), g
        p = r + (g / old) * p
    return x


def placed(core, like):
    out = torch.zeros_like(like, dtype=torch.float64)
    out[..., :core.shape[-1]] = core
    return out


def exact(case, seed):
    s = prepare(case, seed)
    if case["kind"] == "batched":
        return [placed(direct64(b[:, :nx]), b) for b, nx in zip(s["bs"], s["nx"])]
    if case["kind"] == "apply":
        return placed(stencil64(s["x"][:, :case["nx"]].double()), s["x"])
    if case["kind"] == "grad":
        x = direct64(s["b"])
        d = x - s["target"]
        return {"x": x, "loss": 0.5 * d.square().sum(), "grad": direct64(d)}
    core = s["b"][..., :case["nx"]].double()
    return placed(iterate64(core, case["iters"]) if case["iters"] else direct64(core), s["b"])

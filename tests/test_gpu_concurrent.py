"""Host threads that solve grids of different sizes through one kernel.  The
dynamic shared memory limit belongs to the kernel, not to a launch: a thread that
sets it to its own grid's size lowers it under another thread's launch, which the
driver then refuses.  The threads share the default stream, so the solves
themselves run one after another; the host calls race."""
import threading

import pytest
import torch

import paper_1803_03797_gb300 as lap5cg

pytestmark = pytest.mark.gpu


def _hammer(calls, n):
    failures = []

    def work(call):
        try:
            for _ in range(n):
                call()
        except Exception as e:  # noqa: BLE001 -- reported below
            failures.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failures, failures[0]


def _grid(nx, ny):
    return torch.rand(ny, nx, dtype=torch.float64, device="cuda") - 0.5


# pairs that run the same kernel (seven items a thread, NewCG three) with different
# amounts of shared memory, up to the most the resident kernels take
@pytest.mark.parametrize("variant,shapes", [("classic", [(3400, 304), (1024, 1064)]),
                                            ("newcg", [(1400, 304), (1000, 456)])])
def test_resident_solves_of_two_sizes_in_two_threads(variant, shapes):
    def solver(nx, ny):
        b = _grid(nx, ny)
        x, info = torch.zeros_like(b), torch.empty(lap5cg.INFO_BYTES, dtype=torch.uint8, device="cuda")
        ws = torch.empty(lap5cg.workspace_size(nx, ny, nx, variant), dtype=torch.uint8, device="cuda")
        return lambda: lap5cg.cg_solve(b, tol=0.0, maxit=1, variant=variant, out=x, info=info, workspace=ws)

    _hammer([solver(*s) for s in shapes], 1500)


def test_batches_of_two_sizes_in_two_threads():
    def solver(nx, ny):
        bs = [_grid(nx, ny)]
        xs, info = [torch.zeros_like(bs[0])], torch.empty(lap5cg.INFO_BYTES, dtype=torch.uint8, device="cuda")
        ws = torch.empty(lap5cg.batched_workspace_size([nx], [ny], [nx], "classic", "f64"), dtype=torch.uint8,
                         device="cuda")
        return lambda: lap5cg.cg_solve_batched(bs, xs, tol=0.0, maxit=1, precision="f64", info=info, workspace=ws)

    _hammer([solver(1024, 1064), solver(2048, 456)], 1500)

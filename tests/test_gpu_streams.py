"""Calls on a side stream (non-blocking, as torch makes them) while the default stream is still busy: the first solve of a
handle, which allocates and clears its workspace, gives what it gives on an idle default stream.

Bars: 1e-9 for the level-set solves (stopped at 1e-12), 1e-7 for the momentum solve to 1e-10 and 1e-6 for the
velocity-pressure solve to 1e-12, the bars of the same entry points elsewhere in these tests."""
import pytest
import torch

import workloads
from oracle import momentum
from test_gpu_parity import cuda, make_op, rel

pytestmark = pytest.mark.gpu


def free(wl):
    """The applied vector with zero Dirichlet data."""
    f = wl.x.copy()
    f[momentum.Problem.from_workload(wl).constrained()] = 0.0
    return f


CALLS = {
    "normal": (lambda op, wl: op.projected_normal(), 1e-9),
    "advect": (lambda op, wl: op.advect_levelset(1), 1e-9),
    "reinitialize": (lambda op, wl: op.reinitialize(cuda(wl.phi), 2), 1e-9),
    "solve": (lambda op, wl: op.solve(cuda(wl.x), rtol=1e-10), 1e-7),
    "solve_saddle": (lambda op, wl: op.solve_saddle(cuda(free(wl)), rtol=1e-12, max_iter=2000), 1e-6),
}


@pytest.mark.parametrize("n", [4, 12])
@pytest.mark.parametrize("name", sorted(CALLS))
def test_first_solve_on_a_side_stream(name, n):
    call, bar = CALLS[name]
    wl = workloads.random_workload(n, 2, 60 + n, geom="sphere", dirichlet_faces=0x1F)
    want = call(make_op(wl), wl)[0].cpu().numpy()
    op = make_op(wl)
    a = torch.rand(4096, 4096, device="cuda")
    torch.full((1 << 24,), float("nan"), device="cuda")  # what a fresh allocation may hold
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    for _ in range(20):  # some milliseconds of work on the default stream
        a = a @ a
        a = a / a.abs().max()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        got = call(op, wl)[0]
    side.synchronize()
    got = got.cpu().numpy()
    assert rel(got, want) <= bar


@pytest.mark.parametrize("n,p", [(3, 2), (20, 2), (9, 3)])
def test_schur_applies_on_two_streams(n, p):
    """Applies of one handle on two streams at a time: each its own vector's product, bit for bit."""
    op = make_op(workloads.random_workload(n, p, 80 + n, geom="sphere", dirichlet_faces=0x1F))
    g = torch.Generator(device="cuda").manual_seed(n)
    xs = [torch.rand(op.n_p, generator=g, device="cuda", dtype=torch.float64) for _ in range(2)]
    want = [op.apply_schur(x) for x in xs]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(50):
        for k, st in enumerate(streams):
            with torch.cuda.stream(st):
                got[k].append(op.apply_schur(xs[k]))
    torch.cuda.synchronize()
    for k in range(2):
        assert all(torch.equal(y, want[k]) for y in got[k])

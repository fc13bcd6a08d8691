"""Solves with overlapped launches inside a caller's graph that forks and joins: their first kernel then depends on
more than the kernel before it in the stream."""
import pytest

from paper_1909_05423_gb300 import workloads
from tests.gpu_common import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "mixed_f64io"])
def test_fork_and_join(dtype):
    need_gpu()
    import paper_1909_05423_gb300 as pp
    shapes = [(20, 24, 64), (33, 64, 32)]
    plans = [pp.Plan(s, bc, (1.0 / 64,) * 3, dtype) for s, bc in zip(shapes, ("NNPPND", "PPPPDD"))]
    f = [torch.zeros(s, dtype=torch.float64, device="cuda") for s in shapes]
    u = [torch.zeros_like(t) for t in f]
    w = torch.zeros_like(u[0])
    for p, a, b in zip(plans, f, u):
        p.solve(a, out=b)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    with torch.cuda.graph(g):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        f[0].mul_(2.0)
        plans[0].solve(f[0], out=u[0], stream=main)
        plans[1].solve(f[1], out=u[1], stream=side)
        side.wait_stream(main)
        main.wait_stream(side)
        plans[0].solve(u[0], out=w, stream=main)   # after the join
        plans[1].solve(u[1], out=u[1], stream=main)
    for seed in range(3):
        src = [torch.from_numpy(workloads.uniform_source(s, seed=100 + seed)).cuda() for s in shapes]
        for a, b in zip(f, src):
            a.copy_(b)
        g.replay()
        torch.cuda.synchronize()
        once = plans[0].solve(2.0 * src[0])
        assert torch.equal(u[0], once) and torch.equal(w, plans[0].solve(once))
        assert torch.equal(u[1], plans[1].solve(plans[1].solve(src[1])))
    for p in plans:
        p.close()


def test_streams_and_events():
    """Solves that alternate between two streams by events, each in place on the other's result."""
    need_gpu()
    import paper_1909_05423_gb300 as pp
    shape = (24, 48, 64)
    plan = [pp.Plan(shape, "NNDDND", (1.0 / 64,) * 3, "f64") for _ in range(2)]
    f = torch.from_numpy(workloads.uniform_source(shape, seed=104)).cuda()
    ref = f.clone()
    for _ in range(20):
        ref = plan[0].solve(ref) * 50.0
        torch.cuda.synchronize()
    for _ in range(5):
        x = f.clone()
        st = [torch.cuda.Stream() for _ in range(2)]
        for s in st:
            s.wait_stream(torch.cuda.current_stream())
        for i in range(20):
            with torch.cuda.stream(st[i % 2]):
                plan[i % 2].solve(x, out=x, stream=st[i % 2])
                x.mul_(50.0)
                st[(i + 1) % 2].wait_stream(st[i % 2])
        torch.cuda.synchronize()
        assert torch.equal(x, ref)
    for p in plan:
        p.close()

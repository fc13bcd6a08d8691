"""A batch does not write to its member plans: solves of a plan from one host thread while another captures batches
with it on the same stream (a plan's use on one stream), each result against the same call alone."""
import threading

import pytest

from tests.gpu_common import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("options", [None, {"autotune": 1}])
def test_solves_beside_batches(options):
    need_gpu()
    import paper_1909_05423_gb300 as pp
    shape = (24, 128, 256)  # lengths whose kernels differ between a batch and a solve
    sp = (1.0 / 256,) * 3
    plan = pp.Plan(shape, "NNDDND", sp, "f64", options)
    other = pp.Plan((16, 64, 64), "PPPPDD", sp, "f64")
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        f = torch.rand(shape, dtype=torch.float64, device="cuda")
        g = torch.rand((16, 64, 64), dtype=torch.float64, device="cuda")
        outs = [torch.empty_like(f) for _ in range(40)]
        batch = [[torch.empty_like(f), torch.empty_like(g)] for _ in range(24)]
        alone = plan.solve(f, stream=st).clone()
        shapes, split = plan.launch_shapes(), plan.z_split()
        first = pp.solve_batched([plan, other], [f, g], [torch.empty_like(f), torch.empty_like(g)], stream=st)
        first = [t.clone() for t in first]
    st.synchronize()
    done, errors = threading.Event(), []

    def solves():
        try:
            n = 0
            while not done.is_set() or n < len(outs):
                plan.solve(f, out=outs[n % len(outs)], stream=st)
                n += 1
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    t = threading.Thread(target=solves)
    t.start()
    try:
        for us in batch:  # new outputs: a new capture each
            pp.solve_batched([plan, other], [f, g], us, stream=st)
    finally:
        done.set()
        t.join()
    st.synchronize()
    assert not errors, errors
    assert all(torch.equal(u, alone) for u in outs)
    assert all(torch.equal(u[0], first[0]) and torch.equal(u[1], first[1]) for u in batch)
    assert plan.launch_shapes() == shapes and plan.z_split() == split
    plan.close()
    other.close()

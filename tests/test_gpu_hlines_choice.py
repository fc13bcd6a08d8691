"""Which grids take the block-scaled line kernels, and every kind of transform on grids that do (whole solves at 1e-12
relative L2, the tolerance of the FP64-class path): lines along x, against the same solve with the double-float
kernels, lines along y with a partial tile and complex columns along y and z, against the oracle."""
import numpy as np
import pytest

from paper_1909_05423_gb300 import workloads
from tests.gpu_common import gpu_solve, need_gpu, rel_l2, torch

pytestmark = pytest.mark.gpu
TOL = 1e-12
SP = (0.1, 0.1, 0.1)
# (threads, lines per CTA) of the block-scaled kernels by complex points, x and y
X = {64: (128, 32), 128: (128, 16), 256: (128, 8), 512: (256, 8), 1024: (128, 2)}
Y = {64: (128, 32), 128: (128, 16), 256: (128, 8), 512: (256, 8), 1024: (512, 8)}


@pytest.fixture(scope="module", autouse=True)
def _setup(oracle):
    need_gpu()


def _shapes(shape, bc, **options):
    import paper_1909_05423_gb300 as pp
    plan = pp.Plan(shape, bc, SP, "f64", options or None)
    got = plan.launch_shapes()
    plan.close()
    return got


def _check(oracle, shape, bc, seed):
    f = workloads.uniform_source(shape, seed=seed, remove_mean=False)
    assert rel_l2(gpu_solve(f, bc, SP), oracle.solve(f, bc, SP)) <= TOL, (shape, bc)


KINDS = pytest.mark.parametrize("kind", ["PP", "NN", "DD", "DN", "ND"])


@KINDS
@pytest.mark.parametrize("n", [256, 512, 1024, 2048])
def test_large_grids_x(n, kind):
    """An x tile that is not full at the end of the grid."""
    shape, bc = ((1 << 24) // (n * 70) + 1, 70, n), kind + "DDNN"
    got = _shapes(shape, bc)
    assert got["x-forward"] == X[n // 2] and got["x-inverse"] == X[n // 2]
    f = np.random.default_rng(93).uniform(-1, 1, shape)
    assert rel_l2(gpu_solve(f, bc, SP), gpu_solve(f, bc, SP, options=dict(threads_x=128, threads_y=128))) <= TOL, bc


@KINDS
@pytest.mark.parametrize("n", [128, 256, 512, 1024, 2048])
def test_large_grids_y(oracle, n, kind):
    for nx, bc in ((10, "DN" + kind + "DD"), (12, "PP" + kind + "DD")):
        shape = ((1 << 19 if n < 1024 else 5 << 18) // (n * nx) + 3, n, nx)
        if not (bc == "PPPPDD" and n > 1024):
            got = _shapes(shape, bc)
            assert got["y-forward"] == got["y-inverse"] == Y[n if bc == "PPPPDD" else n // 2]
        _check(oracle, shape, bc, 94)


def test_unaligned_arrays():
    """Caller arrays at an 8-byte offset (scalar loads and stores) give the same bits."""
    import paper_1909_05423_gb300 as pp
    shape = (257, 256, 256)
    n = shape[0] * shape[1] * shape[2]
    f = torch.rand(n + 1, dtype=torch.float64, device="cuda")
    u = torch.empty(n + 1, dtype=torch.float64, device="cuda")
    for bc in ("NNDDDD", "PPNNDD", "DNNDDD"):
        plan = pp.Plan(shape, bc, SP, "f64")
        assert plan.launch_shapes()["x-forward"] == X[128]
        a = plan.solve(f[1:].view(shape), out=u[1:].view(shape)).clone()
        assert torch.equal(a, plan.solve(f[1:].clone().view(shape))), bc
        plan.close()


@pytest.mark.parametrize("n,nx", [(64, 280), (512, 36), (1024, 48)])
def test_z_columns(oracle, n, nx):
    shape = (n, 30, nx)
    f = workloads.uniform_source(shape, seed=95, remove_mean=False)
    assert rel_l2(gpu_solve(f, "PPNDPP", SP, options=dict(z_method=2)), oracle.solve(f, "PPNDPP", SP)) <= TOL


@pytest.mark.parametrize("shape,bc,axis", [((2, 8, 1024), "NNDDNN", "x"), ((6, 16, 2048), "DNPPDD", "x"), ((14, 64, 128), "PPDDNN", "x"),
                                           ((100, 100, 1024), "NNDDNN", "x"), ((400, 512, 128), "NNDDNN", "x"),
                                           ((8, 256, 16), "NNDDNN", "y"), ((4, 2048, 16), "PPNNDD", "y")])
def test_small_grids_keep_the_double_float_kernels(shape, bc, axis):
    """A CTA's latency decides there, and the double-float kernels' is the shorter one."""
    own = _shapes(shape, bc)
    for d in ("-forward", "-inverse"):
        n = shape[2] if axis == "x" else shape[1]
        assert own[axis + d] != (X if axis == "x" else Y)[n // 2], own


def test_where_small_grids_take_them():
    """1024 real cells along y and complex columns of up to 512 points: faster at any number of lines."""
    assert _shapes((2, 1024, 4), "NNDDDD")["y-forward"] == Y[512]
    assert _shapes((2, 64, 4), "PPPPDD")["y-forward"] == Y[64]
    assert _shapes((2, 512, 4), "PPPPDD")["y-forward"] == Y[512]


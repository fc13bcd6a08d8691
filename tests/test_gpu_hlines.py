"""The block-scaled FP64-class line kernels (power-of-two lengths from 64 complex points): every kind of
transform along x and y, partial tiles, C2C lines along y and z, and the inputs that decide a line's scale,
against the oracle at the tolerance of the FP64-class path (1e-12 relative L2)."""
import math

import numpy as np
import pytest

from paper_1909_05423_gb300 import _lib, workloads
from tests.gpu_common import gpu_solve, need_gpu, rel_l2, torch

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _setup(oracle):
    need_gpu()


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("kind", ["PP", "NN", "DD", "DN", "ND"])
def test_lines_of_every_kind(oracle, n, kind):
    """n-cell lines along x and along y (64: C2C columns only, and the double-float kernels beside them);
    10 columns leave a partial tile, 3 planes of 2 rows a partial x tile."""
    for shape, bc in (((3, 2, n), kind + "DDNN"), ((3, n, 10), "DN" + kind + "DD"), ((3, n, 12), "PP" + kind + "DD")):
        f = workloads.uniform_source(shape, seed=81, remove_mean=False)
        sp = (0.1, 0.1, 0.1)
        assert rel_l2(gpu_solve(f, bc, sp), oracle.solve(f, bc, sp)) <= TOL, (shape, bc)


@pytest.mark.parametrize("n", [64, 256, 1024])
def test_z_lines(oracle, n):
    f = workloads.uniform_source((n, 6, 8), seed=82, remove_mean=False)
    sp = (0.1, 0.1, 0.1)
    u = gpu_solve(f, "PPNDPP", sp, options=dict(z_method=2))
    assert rel_l2(u, oracle.solve(f, "PPNDPP", sp)) <= TOL


def _sources(n):
    x = (np.arange(n) + 0.5) / n
    one = np.ones((5, n, n))
    blob = np.exp(-((x - 0.4) / 0.05) ** 2)
    yield "constant", one
    yield "blob", one * blob[None, None, :] * blob[None, :, None]  # rows and columns down to 1e-60 of the peak
    yield "one mode", one * np.cos(3 * math.pi * x)[None, None, :] * np.sin(2 * math.pi * x)[None, :, None]
    yield "one cell", np.where(np.arange(5 * n * n).reshape(5, n, n) == 2 * n * n + 7 * n + 9, 1.0, 0.0)
    yield "zero rows", np.where(np.arange(n)[None, :, None] % 3 == 1, 1.0, 0.0) * one


@pytest.mark.parametrize("bc", ["NNDDDD", "PPPPDD", "DNNNDD"])
def test_line_scales(oracle, bc):
    """Smooth, concentrated and partly zero lines, and magnitudes at both ends of the documented range."""
    n = 128
    sp = (1.0 / n,) * 3
    for name, f in _sources(n):
        f = np.ascontiguousarray(f)
        ref = oracle.solve(f, bc, sp)
        for scale in (1.0, 1e-20, 1e25):
            assert rel_l2(gpu_solve(f * scale, bc, sp), ref * scale) <= TOL, (name, scale)
    assert not gpu_solve(np.zeros((5, n, n)), bc, sp).any()


def test_unaligned_arrays():
    """Caller arrays at an 8-byte offset (scalar loads and stores) give the same bits."""
    import paper_1909_05423_gb300 as pp
    shape = (3, 128, 256)
    for bc in ("NNDDDD", "PPNNDD", "DNNDDD"):
        plan = pp.Plan(shape, bc, (1.0 / 256,) * 3, "f64")
        n = shape[0] * shape[1] * shape[2]
        f = torch.rand(n + 1, dtype=torch.float64, device="cuda")
        u = torch.empty(n + 1, dtype=torch.float64, device="cuda")
        a = plan.solve(f[1:].view(shape), out=u[1:].view(shape)).clone()
        b = plan.solve(f[1:].clone().view(shape))
        assert torch.equal(a, b), bc
        plan.close()


@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf])
def test_non_finite_source(bad):
    """A non-finite value reaches the range report and the solution, as on the other kernels."""
    import paper_1909_05423_gb300 as pp
    shape = (6, 128, 128)
    f = workloads.uniform_source(shape, seed=83)
    f[2, 3, 4] = bad
    plan = pp.Plan(shape, "NNDDNN", (1.0 / 128,) * 3, "f64")
    u = plan.solve(torch.from_numpy(f).cuda())
    torch.cuda.synchronize()
    with pytest.raises(_lib.PPError) as e:
        plan.status()
    assert e.value.status == _lib.PP_ERR_RANGE
    assert not torch.isfinite(u[2]).any()
    plan.close()


def test_solve_inside_a_captured_graph():
    """The overlapped launches of a small grid record into a caller's graph and replay on new data."""
    import paper_1909_05423_gb300 as pp
    shape = (20, 24, 64)
    plan = pp.Plan(shape, "NNPPND", (1.0 / 64,) * 3, "f64")
    f, u = (torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2))
    plan.solve(f, out=u)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.solve(f, out=u, stream=torch.cuda.current_stream())
        plan.solve(u, out=u, stream=torch.cuda.current_stream())
    for seed in range(3):
        f.copy_(torch.from_numpy(workloads.uniform_source(shape, seed=90 + seed)))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(u, plan.solve(plan.solve(f)))
    plan.close()

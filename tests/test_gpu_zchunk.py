"""The partitioned z solve where plans take it by themselves: periodic z (Sherman-Morrison on chunks), the
adjoint, and the singular mode's CTA, at the edges of chunks and of the carry window, against the oracle.

Tolerances are those of the solver's other parity tests: 1e-12 relative L2 for FP64-class plans, 1e-6 for
single-precision transforms."""
import numpy as np
import pytest

from paper_1909_05423_gb300 import workloads
from tests.gpu_common import gpu_solve, need_gpu, rel_l2, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup(oracle):
    need_gpu()


def _tol(dtype):
    return 1e-12 if dtype == "f64" else 1e-6


@pytest.mark.parametrize("dtype", ["f64", "mixed_f64io"])
@pytest.mark.parametrize("nz", [3, 7, 8, 9, 16, 17, 100, 129, 640])
def test_periodic_z_chunks(oracle, nz, dtype):
    """One chunk, whole chunks, a last chunk of one row and of several, and more chunks than the window;
    long lines of small grids hold modes that decay slowly (the doubling, the near -1 products)."""
    for shape, bc in (((nz, 8, 12), "PPPPPP"), ((nz, 6, 10), "NNDDPP"), ((nz, 12, 8), "DNPPPP")):
        sp = (1.0 / shape[2], 1.0 / shape[1], 1.0 / max(nz, 16))
        f = workloads.uniform_source(shape, seed=71, remove_mean=bc == "PPPPPP")
        assert rel_l2(gpu_solve(f, bc, sp, dtype), oracle.solve(f, bc, sp)) <= _tol(dtype), bc


@pytest.mark.parametrize("nz", [2, 5, 31, 257])
@pytest.mark.parametrize("how", ["solve", "solve_adjoint"])
def test_default_split_and_adjoint(oracle, nz, how):
    """A plan that chose the partitioned solve by its size, forward and adjoint (S is symmetric)."""
    import paper_1909_05423_gb300 as pp
    shape = (nz, 10, 18)
    sp = (1.0 / 18, 1.0 / 10, 1.0 / 40)
    for bc in ("NNDDND", "PPNNDD", "NDPPNN"):
        plan = pp.Plan(shape, bc, sp, "f64")
        assert plan.z_split() == 8
        plan.close()
        f = workloads.uniform_source(shape, seed=72, remove_mean=False)
        assert rel_l2(gpu_solve(f, bc, sp, how=how), oracle.solve(f, bc, sp)) <= 1e-12, bc


@pytest.mark.parametrize("nz,split", [(2, 1), (2, 8), (3, 0), (255, 1), (255, 16), (300, 0), (4096, 1), (4100, 1)])
def test_singular_mode(oracle, nz, split):
    """The singular mode by one CTA with its rows in registers (one or several a thread), and by one
    thread where a line has more rows than a CTA holds (4100 rows on the sweeps' 256 threads)."""
    for bc, nx, ny in (("NNNNNN", 4, 6), ("PPNNNN", 6, 4), ("PPPPPP", 4, 4)):
        if nz < 3 and bc[4] == "P":
            continue
        shape = (nz, ny, nx)
        sp = (1.0 / nx, 1.0 / ny, 1.0 / nz)
        f = workloads.uniform_source(shape, seed=73)
        u = gpu_solve(f, bc, sp, options=dict(z_split=split))
        assert rel_l2(u, oracle.solve(f, bc, sp)) <= 1e-12, bc
        assert abs(u.mean()) <= 1e-12 * np.abs(u).max()

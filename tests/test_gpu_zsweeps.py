"""The z sweeps where small grids would take the partitioned solve by themselves: Sherman-Morrison on whole lines
(z_method = 1, or any z_split, on periodic z) and the transposed Thomas sweeps (the adjoint with z_split = 1), with
and without the singular mode, against the oracle; and what a plan reports about its z solve."""
import pytest

from paper_1909_05423_gb300 import workloads
from tests.gpu_common import gpu_solve, need_gpu, rel_l2

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-12, "mixed_f64io": 1e-6, "mixed_f32io": 1e-6}


@pytest.fixture(scope="module", autouse=True)
def _setup(oracle):
    need_gpu()


@pytest.mark.parametrize("dtype", ["f64", "mixed_f64io"])
@pytest.mark.parametrize("nz", [3, 8, 17, 129, 640])
def test_periodic_sweeps(oracle, nz, dtype):
    for shape, bc in (((nz, 8, 12), "PPPPPP"), ((nz, 6, 10), "NNDDPP"), ((nz, 12, 8), "NNPPPP"), ((nz, 20, 18), "DNNNPP")):
        sp = (1.0 / shape[2], 1.0 / shape[1], 1.0 / max(nz, 16))
        f = workloads.uniform_source(shape, seed=91, remove_mean=False)
        ref = oracle.solve(f, bc, sp)
        for options in ({"z_method": 1}, {"z_split": 1}):
            assert rel_l2(gpu_solve(f, bc, sp, dtype, options=options), ref) <= TOL[dtype], (bc, options)


@pytest.mark.parametrize("dtype", ["f64", "mixed_f64io", "mixed_f32io"])
@pytest.mark.parametrize("nz", [2, 5, 31, 257])
def test_transposed_sweeps(oracle, nz, dtype):
    """S is symmetric: the adjoint through the transposed factorisation is the solve."""
    shape = (nz, 10, 18)
    sp = (1.0 / 18, 1.0 / 10, 1.0 / 40)
    for bc in ("NNDDND", "PPNNDD", "NDPPNN", "NNNNNN"):
        f = workloads.uniform_source(shape, seed=92, remove_mean=bc == "NNNNNN")
        u = gpu_solve(f, bc, sp, dtype, how="solve_adjoint", options={"z_split": 1})
        assert rel_l2(u, oracle.solve(f, bc, sp)) <= TOL[dtype], bc


def test_reported_split():
    import paper_1909_05423_gb300 as pp
    sp = (0.1, 0.1, 0.1)
    for options, want in (({}, 8), ({"z_method": 1}, 1), ({"z_method": 2}, 1), ({"z_split": 1}, 1), ({"z_split": 32}, 1),
                          ({"z_method": 1, "autotune": 1}, 1), ({"z_method": 1, "z_split": 16}, 1)):
        plan = pp.Plan((64, 8, 12), "NNDDPP", sp, options=options)
        assert plan.z_split() == want, options
        assert plan.z_method() == ("transform" if options.get("z_method") == 2 else "sherman-morrison")
        plan.close()
    # a split that would take too many chunks, accepted for periodic z
    plan = pp.Plan((5000, 4, 4), "NNDDPP", sp, options={"z_split": 8})
    assert plan.z_split() == 1
    plan.close()
    # the autotuner chooses between the sweeps and the transform when the split is given
    plan = pp.Plan((64, 8, 12), "NNDDPP", sp, options={"z_split": 8, "autotune": 1})
    assert plan.z_split() == 1 and plan.z_method() in ("sherman-morrison", "transform")
    plan.close()


@pytest.mark.parametrize("shape,bc,dtype,want", [
    ((8, 512, 512), "NNDDNN", "f64", 1), ((2, 256, 256), "PPDDDD", "f64", 1), ((32, 512, 512), "NNDDNN", "f64", 1),
    ((8, 256, 512), "NNDDNN", "mixed_f64io", 1), ((3, 448, 448), "NNDDPP", "f64", 1), ((12, 256, 256), "NNDDPP", "mixed_f64io", 1),
    ((32, 256, 256), "NNDDNN", "f64", 8), ((256, 256, 256), "NNDDNN", "f64", 16), ((64, 64, 64), "NNDDNN", "mixed_f64io", 8),
    ((192, 192, 192), "NNDDPP", "f64", 8)])
def test_default_by_size(shape, bc, dtype, want):
    """Short lines of large planes take the sweeps, which are done with them in less time than the chunks' CTAs need."""
    import paper_1909_05423_gb300 as pp
    plan = pp.Plan(shape, bc, (0.1, 0.1, 0.1), dtype)
    assert plan.z_split() == want
    plan.close()


@pytest.mark.parametrize("dtype", ["f64", "mixed_f64io"])
@pytest.mark.parametrize("nz", [3, 12, 40, 41, 57])
@pytest.mark.parametrize("bc", ["NNNNNN", "PPNNNN", "PPPPPP"])
def test_singular_mode_short_lines(oracle, bc, nz, dtype):
    """The singular mode by one thread (up to 40 rows) and by a CTA, in front of the sweeps and of the chunks."""
    shape = (nz, 6, 8)
    sp = (1.0 / 8, 1.0 / 6, 1.0 / nz)
    f = workloads.uniform_source(shape, seed=97)
    ref = oracle.solve(f, bc, sp)
    for options in ({"z_split": 1}, None):
        assert rel_l2(gpu_solve(f, bc, sp, dtype, options=options), ref) <= TOL[dtype], options

"""The scale of the block-scaled line kernels on lines of a few cells, whose sum of magnitudes sets it, through whole
solves at 1e-12 relative L2, the tolerance of the FP64-class path: lines along y against the oracle, lines along x,
which take these kernels in large grids only, against the same solve with the double-float kernels.  Every plane holds the same line
at another magnitude between 1 and 2: the scale is a power of two, so a line can leave its integers at some
magnitudes only."""
import numpy as np
import pytest

from tests.gpu_common import gpu_solve, need_gpu, rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-12
MAGS = tuple(1.0 + k / 24.0 for k in range(24))
SP = (0.1, 0.1, 0.1)


@pytest.fixture(scope="module", autouse=True)
def _setup(oracle):
    need_gpu()


def _across(n, values):
    """Factors of the lines of a plane, so many that the grid has at least `values` cells: the block-scaled kernels
    are taken from 2^24 cells on along x, from 2^19 on (1024 complex points: 5 2^18) along y."""
    m = -(-values // (len(MAGS) * n))
    while m % 2 or any(m % p == 0 for p in range(11, m + 1) if all(p % q for q in range(2, int(p ** 0.5) + 1))):
        m += 1
    return np.random.default_rng(n).uniform(-2, 2, max(m, 4))


def _x_lines(line):
    """[plane, ny, nx]: MAGS[plane] x line[i] across[j], the line along x."""
    across = _across(len(line), 1 << 24)
    return np.array(MAGS)[:, None, None] * across[None, :, None] * line[None, None, :]


def _y_lines(line):
    across = _across(len(line), 1 << 19 if len(line) < 1024 else 5 << 18)
    return np.array(MAGS)[:, None, None] * line[None, :, None] * across[None, None, :]


def _check(oracle, f, bc):
    assert rel_l2(gpu_solve(f, bc, SP), oracle.solve(f, bc, SP)) <= TOL, bc


def _check_x(f, bc):
    assert rel_l2(gpu_solve(f, bc, SP), gpu_solve(f, bc, SP, options=dict(threads_x=128, threads_y=128))) <= TOL, bc


@pytest.mark.parametrize("n", [128, 256, 512, 2048])
@pytest.mark.parametrize("kind", ["DN", "ND"])
def test_four_cells_type_iv(oracle, n, kind):
    """Cells that meet in one butterfly of the first stage, after the pre-products turned them."""
    for cells in ((5 * n // 8 - 1, 5 * n // 8, 7 * n // 8 - 1, 7 * n // 8), (n // 8 - 1, n // 8, 3 * n // 8 - 1, 3 * n // 8)):
        line = np.zeros(n)
        line[list(cells)] = 1.0
        _check(oracle, _y_lines(line), "NN" + kind + "DD")
        _check(oracle, _y_lines(line), "PP" + kind + "DD")
        if n > 128:
            _check_x(_x_lines(line), kind + "NNDD")


def _aligned(M, j):
    """32 complex points that add up at 45 degrees in the second result of the odd half of butterfly j of the second
    stage (radices 8 and 8), each with the larger of its parts at 1."""
    t, z = j % 8, np.zeros(M, dtype=complex)
    for u, c in ((1, 1), (5, -1), (3, -1j), (7, 1j)):
        for v in range(8):
            n = j // 8 + u * (M // 64) + v * (M // 8)
            w = c * np.exp(-2j * np.pi * ((j // 8 + u * (M // 64)) * t % M) / M) * np.exp(-2j * np.pi * (v * t % 8) / 8)
            x = np.conj(w) * np.exp(0.25j * np.pi)
            z[n] = x / max(abs(x.real), abs(x.imag))
    return z


@pytest.mark.parametrize("M", [64, 512])
@pytest.mark.parametrize("j", [1, 5])
def test_aligned_second_stage(oracle, M, j):
    z = _aligned(M, j)
    nx = 8
    # complex columns: a real source whose x transform is z in column 1
    f = np.real(z[None, :, None] * np.exp(2j * np.pi * np.arange(nx) / nx)[None, None, :]) * (2.0 / nx)
    _check(oracle, np.array(MAGS)[:, None, None] * f, "PPPPDD")
    # real lines of 2M cells: R2C pairs (u_2k, u_2k+1), the Makhoul order of DCT-II and DST-II
    r2c = np.empty(2 * M)
    r2c[0::2], r2c[1::2] = z.real, z.imag
    mk = np.empty(2 * M)
    k = np.arange(M // 2)
    mk[4 * k], mk[4 * k + 2] = z[k].real, z[k].imag
    mk[4 * k + 3], mk[4 * k + 1] = z[M - 1 - k].real, z[M - 1 - k].imag
    for line, kind in ((r2c, "PP"), (mk, "NN"), (np.where(np.arange(2 * M) % 2, -mk, mk), "DD")):
        _check(oracle, _y_lines(line), "NN" + kind + "DD")
        if M > 64:
            _check_x(_x_lines(line), kind + "NNDD")


@pytest.mark.parametrize("n", [128, 1024])
@pytest.mark.parametrize("kind", ["PP", "NN", "DD"])
def test_one_wave_at_a_quarter(oracle, n, kind):
    """Sources of one wave whose spectrum is the middle Hermitian item of a line alone (n/4 waves; n/4 or 3n/4 half
    waves), which the inverse kinds pair with itself."""
    x = np.arange(n) + 0.5
    for m in (n // 4, 3 * n // 4):
        wave = {"PP": np.cos(2 * np.pi * m * (x - 0.5) / n + 0.3), "NN": np.cos(np.pi * m * x / n),
                "DD": np.sin(np.pi * m * x / n)}[kind]
        _check(oracle, _y_lines(wave), "NN" + kind + "DD")
        _check(oracle, _y_lines(wave), "PP" + kind + "DD")
        if n > 128:
            _check_x(_x_lines(wave), kind + "NNDD")


@pytest.mark.parametrize("kind", ["NN", "PP", "DN"])
def test_large_magnitudes(oracle, kind):
    """Lines whose sum of magnitudes is beyond FP32's range while the transforms stay within it."""
    rng = np.random.default_rng(84)
    f = np.zeros((6, 1050, 2048))
    f[:, 5::350] = rng.uniform(-5e35, 5e35, (6, 3, 2048))
    _check_x(f, kind + "DDDD")
    _check(oracle, rng.uniform(-2e35, 2e35, (10, 2048, 70)), "DD" + kind + "DD")

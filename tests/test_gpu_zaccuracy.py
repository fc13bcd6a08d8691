"""The partitioned z solve against the sweeps of the same plan arguments (FP64-class): what the chunks add to the
rounding.  The line transforms of the two are the same, so only the z solves differ."""
import numpy as np
import pytest

from tests.gpu_common import gpu_solve, need_gpu, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    need_gpu()


@pytest.mark.parametrize("rows", [8, 16, 32])
def test_weakly_dominant_modes(rows):
    """A smooth source on long lines, whose modes decay over some 15 rows: a chunk's A is close to 1 and the same all
    along the line, so an error in 1 - A would add up.  Five roundings of 2^-49 a row over 15 rows are 1.5e-14 of
    the solution in either solve, 2.2e-14 between them; the limit is 1.6 times that."""
    shape = (3000, 48, 48)
    z, y, x = ((np.arange(n) + 0.5) / n for n in shape)
    bump = lambda t, c, w: np.exp(-((t - c) ** 2) / (2 * w * w))  # noqa: E731
    f = bump(z, 0.45, 0.1)[:, None, None] * bump(y, 0.4, 0.2)[None, :, None] * bump(x, 0.6, 0.2)[None, None, :]
    sp = (1.0 / 48,) * 3
    u = gpu_solve(f, "NNDDNN", sp, options={"z_split": rows})
    assert rel_l2(u, gpu_solve(f, "NNDDNN", sp, options={"z_split": 1})) <= 3.5e-14


@pytest.mark.parametrize("rows", [8, 16, 32])
@pytest.mark.parametrize("nz", [64, 257, 1000])
def test_steps_are_those_of_the_sweeps(rows, nz):
    """Strongly dominant modes (w about 0.17): a carry that is a rounding off changes the first rows of its chunk and is
    forgotten, so nine values in ten are the sweeps' to the bit, if the steps in between round alike."""
    f = np.random.default_rng(85).uniform(-1, 1, (nz, 2, 2))
    u = gpu_solve(f, "DDDDND", (1.0, 1.0, 1.0), options={"z_split": rows})
    assert (u == gpu_solve(f, "DDDDND", (1.0, 1.0, 1.0), options={"z_split": 1})).mean() >= 0.9

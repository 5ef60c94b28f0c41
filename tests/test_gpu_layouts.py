"""A grid of the large layout (three (y, z) kernels, row-stage kernels) whose
x axis becomes periodic and open again: the general convolution in between,
its field and a replayed step against the float64 oracle (5e-6 of the
maximum, 1e-5), and afterwards the field and the steps of a context that was
open throughout, bit for bit.  A film likewise, through the film kernel of the
other row length."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.field import Field  # noqa: E402
from oracle.rk45 import RK45  # noqa: E402
from paper_1406_7635_gb300.workloads import Problem, normalise  # noqa: E402

FIELD_TOL = 5e-6
M_TOL = 1e-5


@pytest.fixture(scope="module")
def mm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm as _mm
    return _mm


def problem(nx, ny, nz):
    rng = np.random.default_rng(nx + 100 * ny + 10000 * nz)
    p = Problem(nx, ny, nz, 2e-9, 2.5e-9, 2e-9)
    p.region = rng.integers(0, 3, size=p.shape).astype(np.uint8)
    for r in range(3):
        p.msat[r], p.aex[r] = rng.uniform(6e5, 1.1e6), rng.uniform(1.0e-11, 1.6e-11)
        p.alpha[r], p.ku1[r] = rng.uniform(0.05, 0.3), rng.uniform(-1e5, 3e5)
        p.b0[r] = rng.uniform(-0.03, 0.03, 3)
    p.mask = (rng.uniform(size=p.shape) > 0.05).astype(np.uint8)
    m = np.array([1.0, 0.3, 0.2])[:, None, None, None] + 0.5 * rng.standard_normal((3,) + p.shape)
    p.m0 = normalise(m, p.magnetic())
    p.dt0 = 2e-14
    return p


@pytest.mark.parametrize("nx,ny,nz", [(32, 18, 40), (64, 33, 1)])
def test_periodic_and_back(mm, nx, ny, nz):
    p = problem(nx, ny, nz)
    a, b = mm.Context.from_problem(p), mm.Context.from_problem(p)
    field = a.get_bdemag()
    a.step(1)
    a.set_m(p.m0)
    a.set_pbc(1, 0, 0)
    q = problem(nx, ny, nz)
    q.pbc = (1, 0, 0)
    m32 = p.m0.astype(np.float32).astype(np.float64)
    ref = Field(q).terms(m32, 0.0)["demag"]
    assert np.abs(a.get_bdemag() - ref).max() <= FIELD_TOL * np.abs(ref).max()
    a.set_time(0.0, p.dt0)
    n0 = len(a.get_dt_history())
    a.step(2)
    ora = RK45(q, m=m32)
    ora.run_fixed(a.get_dt_history()[n0:])
    assert np.abs(a.get_m() - ora.m).max() <= M_TOL
    a.set_pbc(0, 0, 0)
    for c in (a, b):
        c.set_m(p.m0)
        c.set_time(0.0, p.dt0)
    assert np.array_equal(a.get_bdemag(), field)
    a.step(3)
    b.step(3)
    assert np.array_equal(a.get_m(), b.get_m()) and a.get_time() == b.get_time()
    a.close()
    b.close()

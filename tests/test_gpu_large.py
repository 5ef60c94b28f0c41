"""Grids beyond one cluster's (y, z) planes, which convolve with the three
register kernels and step with the row-stage kernels: 64-point z classes
(pz = 128, full and ragged), long y classes, short and long x rows.  Field
and torque 5e-6 of their maximum, replayed steps 1e-5, against the float64
oracle; the switches keep their answers on these grids."""
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


def block(nx, ny, nz, dmi=False):
    rng = np.random.default_rng(nx + 100 * ny + 10000 * nz)
    p = Problem(nx, ny, nz, 2e-9, 2.5e-9, 2e-9)
    p.region = rng.integers(0, 3, size=p.shape).astype(np.uint8)
    for r in range(3):
        p.msat[r], p.aex[r] = rng.uniform(6e5, 1.1e6), rng.uniform(1.0e-11, 1.6e-11)
        p.alpha[r], p.ku1[r] = rng.uniform(0.05, 0.3), rng.uniform(-1e5, 3e5)
        p.b0[r] = rng.uniform(-0.03, 0.03, 3)
        if dmi:
            p.dind[r] = rng.uniform(1e-3, 3e-3)
    p.mask = (rng.uniform(size=p.shape) > 0.05).astype(np.uint8)
    m = np.array([1.0, 0.3, 0.2])[:, None, None, None] + 0.5 * rng.standard_normal((3,) + p.shape)
    p.m0 = normalise(m, p.magnetic())
    p.dt0 = 2e-14
    return p


# (nx, ny, nz): pz = 128 full and ragged, py = 512 beside pz = 64, py = 1024,
# x rows of 16 (nx odd) and 512 complex values
GRIDS = [(20, 18, 64), (17, 21, 33), (12, 140, 17), (11, 260, 12), (300, 17, 34)]


@pytest.mark.parametrize("nx,ny,nz", GRIDS)
def test_field_and_steps_vs_oracle(mm, nx, ny, nz):
    p = block(nx, ny, nz, dmi=(nx == 17))
    ctx = mm.Context.from_problem(p)
    m32 = p.m0.astype(np.float32).astype(np.float64)
    f = Field(p)
    for got, ref in ((ctx.get_bdemag(), f.terms(m32, 0.0)["demag"]), (ctx.get_torque(), f.torque(m32, 0.0))):
        assert np.abs(got - ref).max() <= FIELD_TOL * np.abs(ref).max()
    ctx.step(2)
    ora = RK45(p, m=m32)
    ora.run_fixed(ctx.get_dt_history())
    assert np.abs(ctx.get_m() - ora.m).max() <= M_TOL
    ctx.close()


def test_switches_on_a_large_grid(mm):
    p = block(20, 18, 40)
    a, b = mm.Context.from_problem(p), mm.Context.from_problem(p)
    assert a.set_yz_kernels(0) == 0 and a.set_yz_kernels(1) == 0
    with pytest.raises(mm.MMError) as e:
        a.set_yz_kernels(2)
    assert e.value.code == -1
    a.set_wait_limit(0)                      # (no bounded waits on these grids)
    a.step(3)
    b.step(3)
    assert np.array_equal(a.get_m(), b.get_m())
    # the general stage kernels (RK23) with the same convolution
    b.set_integrator("rk23")
    b.step(3)
    assert b.get_stats()["accepted"] == 6
    # a periodic axis goes back to the general convolution, and returns
    c = mm.Context.from_problem(p)
    field = c.get_bdemag()
    c.set_pbc(0, 0, 0)
    assert np.array_equal(c.get_bdemag(), field)
    for x in (a, b, c):
        x.close()

"""The persistent film kernel (films and grids of two to four layers step with
it by default) at the edges of its splits: row lengths and column lengths of every transform size, ragged
rows, one and several rows and columns per block, periodic x, DMI,
spin-transfer torques and both integrators, against the stage kernels'
path replaying the same step sizes (two float32 paths: 5e-6) and, on small
films, against the float64 oracle (1e-5, the bar of a replayed sequence)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.rk45 import RK45  # noqa: E402
from paper_1406_7635_gb300.workloads import Problem, film_sp4, normalise  # noqa: E402

PATH_TOL = 5e-6
M_TOL = 1e-5


@pytest.fixture(scope="module")
def mm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm as _mm
    return _mm


def film(nx, ny, dmi=False, pbcx=False, stt=False, nz=1):
    rng = np.random.default_rng(1000 * nx + ny)
    p = Problem(nx, ny, nz, 2e-9, 2e-9, 1.5e-9)
    p.region = rng.integers(0, 3, size=p.shape).astype(np.uint8)
    for r in range(3):
        p.msat[r] = rng.uniform(6e5, 1.1e6)
        p.aex[r] = rng.uniform(1.0e-11, 1.6e-11)
        p.alpha[r] = rng.uniform(0.05, 0.3)
        p.ku1[r] = rng.uniform(-1e5, 3e5)
        u = rng.standard_normal(3)
        p.anis_u[r] = u / np.linalg.norm(u)
        p.b0[r] = rng.uniform(-0.03, 0.03, 3)
        p.b1[r] = rng.uniform(-0.03, 0.03, 3)
        if dmi:
            p.dind[r] = rng.uniform(1e-3, 3e-3)
        if stt:
            p.jcur[r], p.xi[r], p.pol[r], p.lam[r] = (1e13, 2e12, 1e12), 0.05, 0.5, 1.3
            p.epsp[r], p.tfree[r], p.mp[r] = 0.02, 2e-9, (0.0, 1.0, 0.2)
    p.zhang_li = p.slonczewski = stt
    p.freq, p.phase = 1e9, 0.4
    p.mask = (rng.uniform(size=p.shape) > 0.05).astype(np.uint8)
    if pbcx:
        p.pbc = (1, 0, 0)
    m = np.array([1.0, 0.3, 0.2])[:, None, None, None] + 0.5 * rng.standard_normal((3,) + p.shape)
    p.m0 = normalise(m, p.magnetic())
    p.dt0 = 2e-14
    return p


# (x rows of 16 .. 512 complex values, y classes of 16 .. 512 points, ragged
# and full, rows per block 1, 2, 3, 4)
SHAPES = [(9, 9, {}), (16, 16, {}), (17, 33, {}), (64, 17, {}), (65, 64, {}), (128, 129, {}), (200, 257, {}),
          (257, 100, {}), (256, 256, {}), (100, 445, {}), (512, 512, {}), (300, 60, {"dmi": True}),
          (100, 75, {"dmi": True}), (64, 40, {"pbcx": True, "stt": True}), (33, 20, {"stt": True}),
          (1024, 20, {"pbcx": True}), (512, 300, {"pbcx": True, "dmi": True}),
          # two to four layers: one to four rows per block, ragged layers
          (20, 30, {"nz": 4}), (96, 96, {"nz": 4}), (17, 120, {"nz": 4}), (33, 17, {"nz": 2}), (128, 64, {"nz": 2}),
          (40, 128, {"nz": 2}), (130, 33, {"nz": 3}), (30, 20, {"nz": 3, "dmi": True}),
          (64, 40, {"nz": 2, "pbcx": True, "stt": True})]


@pytest.mark.parametrize("method", ["rk45", "rk23"])
@pytest.mark.parametrize("nx,ny,kw", SHAPES)
def test_matches_the_stage_kernels(mm, nx, ny, kw, method):
    p = film(nx, ny, **kw)
    a = mm.Context.from_problem(p)
    a.set_integrator(method)
    a.step(4)
    dts = a.get_dt_history()
    b = mm.Context.from_problem(p)
    b.set_integrator(method)
    assert b.set_yz_kernels(1) == 1          # (particular (y, z) kernels: the stage kernels' graph)
    b.set_fixed_dt_sequence(dts)
    b.step(4)
    assert a.get_stats()["launches"] == 2    # first stage, then all steps
    assert b.get_stats()["launches"] > 20
    assert np.abs(a.get_m() - b.get_m()).max() <= PATH_TOL
    sa, sb = a.get_stats(), b.get_stats()
    assert sa["accepted"] == sb["accepted"] == 4
    # (the error of the last step, an alternating sum of order-1 terms times dt)
    assert abs(sa["last_err"] - sb["last_err"]) <= 1e-2 * sb["last_err"] + 1e-7
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny,kw", [(17, 9, {}), (40, 33, {"dmi": True}), (32, 20, {"pbcx": True, "stt": True}),
                                      (19, 21, {"nz": 3}), (24, 18, {"nz": 2, "dmi": True, "stt": True})])
def test_matches_the_oracle(mm, nx, ny, kw):
    p = film(nx, ny, **kw)
    ctx = mm.Context.from_problem(p)
    ctx.step(6)
    p.mp = p.mp / np.linalg.norm(p.mp, axis=1, keepdims=True)   # (the library normalises it, the oracle takes a unit vector)
    ora = RK45(p, m=p.m0.astype(np.float32).astype(np.float64))
    ora.run_fixed(ctx.get_dt_history())
    assert np.abs(ctx.get_m() - ora.m).max() <= M_TOL
    ctx.close()


def test_run_rejections_and_replay(mm):
    """run() lands on t_end; a far too large first step is rejected until it
    fits; one call of n steps equals n calls bit for bit; a replayed sequence
    ends where it ends."""
    p = film_sp4(64, 16)
    p.dt0 = 2e-12
    a, b = mm.Context.from_problem(p), mm.Context.from_problem(p)
    a.step(7)
    for _ in range(7):
        b.step(1)
    assert a.get_stats()["rejected"] > 0
    assert np.array_equal(a.get_m(), b.get_m()) and a.get_time() == b.get_time()
    t1 = a.get_time()[0] + 1e-12
    a.run(t1)
    assert a.get_time()[0] == t1
    state = a.get_state()
    a.run(t1 + 1e-12)
    b.set_state(state)
    b.run(t1 + 1e-12)
    assert np.array_equal(a.get_m(), b.get_m())
    c = mm.Context.from_problem(p)
    c.set_fixed_dt_sequence(a.get_dt_history()[:4])
    c.step(10)
    assert c.get_stats()["accepted"] == 4
    for x in (a, b, c):
        x.close()


def test_expired_wait_and_nan(mm):
    """A barrier wait that gives up reports MM_ERR_TIMEOUT and leaves m, t and
    dt; with the default limit the context continues bit for bit; NaN in m is
    MM_ERR_NONFINITE."""
    p = film_sp4(64, 16)                     # (tensor copies in the stage kernels: the limit applies)
    ref, ctx = mm.Context.from_problem(p), mm.Context.from_problem(p)
    ref.step(3)
    ctx.step(1)
    m1, t1 = ctx.get_m(), ctx.get_time()
    ctx.set_wait_limit(0)
    for _ in range(2):
        with pytest.raises(mm.MMError) as e:
            ctx.step(1)
        assert e.value.code == -6
        assert np.array_equal(ctx.get_m(), m1) and ctx.get_time() == t1
    ctx.set_wait_limit(1 << 30)
    ctx.step(2)
    assert np.array_equal(ctx.get_m(), ref.get_m()) and ctx.get_time() == ref.get_time()
    bad = m1.copy()
    bad[1, 0, 3, 5] = np.nan
    ctx.set_m(bad)
    with pytest.raises(mm.MMError) as e:
        ctx.step(1)
    assert e.value.code == -4
    ref.close()
    ctx.close()

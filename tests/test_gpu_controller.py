"""The step controller at its corners, in the film kernel and in the stage
kernels on the same problem: a first step that is rejected until it fits, a
step cap, run() landing on its end times, a replayed sequence that ends, a
rejection that would need a step below dt_min, NaN in m.  Both paths take the
same decisions: return code, accepted and rejected steps, evaluations, and the
times that are given, exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm as _mm
    return _mm


def rejected(c):
    c.set_solver(1e-5, 0.8, 3e-13, 1e-20, 1e-12)
    c.step(25)


def capped(c):
    c.set_solver(1e-5, 0.8, 1e-16, 1e-20, 3e-14)
    c.step(12)


def landing(c):
    c.set_solver(1e-4, 0.8, 2e-13, 1e-20, 1e-10)
    for k in range(1, 4):
        c.run(k * 3.3e-13)
        assert c.get_time()[0] == k * 3.3e-13


def replay(c):
    c.set_fixed_dt_sequence([1e-14 * (i % 3 + 1) for i in range(9)])
    c.step(5)
    c.step(9)


def underflow(c):
    c.set_solver(1e-9, 0.8, 5e-13, 4e-13, 1e-10)
    c.step(5)


def nan(c):
    m = c.get_m()
    m[0, 0, 0, 0] = np.nan
    c.set_m(m)
    c.step(2)


@pytest.mark.parametrize("shape", [(64, 16, 1), (40, 33, 3)])
@pytest.mark.parametrize("method", ["rk45", "rk23"])
@pytest.mark.parametrize("run,code", [(rejected, 0), (capped, 0), (landing, 0), (replay, 0), (underflow, -5), (nan, -4)])
def test_both_paths_decide_alike(mm, shape, method, run, code):
    nx, ny, nz = shape
    rng = np.random.default_rng(nx + nz)
    m = np.array([1, 0.5, 0.2])[:, None, None, None] + 0.4 * rng.standard_normal((3, nz, ny, nx))
    m = (m / np.sqrt((m * m).sum(0))).astype(np.float32)
    got = []
    for which in (0, 1):
        with mm.Context(nx, ny, nz, 3e-9, 3e-9, 3e-9) as c:
            c.set_material(0, 8e5, 1.3e-11, 0.05)
            c.set_bext(0, (0.01, 0.3, 0.0))
            if which:
                c.set_yz_kernels(which)
            c.set_integrator(method)
            c.set_m(m)
            rc = 0
            try:
                run(c)
            except mm.MMError as e:
                rc = e.code
            s = c.get_stats()
            got.append((rc, s["accepted"], s["rejected"], s["evals"]))
            if run in (replay, underflow, nan):   # (steps that no error chose)
                got[-1] += (s["t"], s["dt"])
    assert got[0] == got[1]
    assert got[0][0] == code
    if run is rejected:
        assert got[0][2] > 0

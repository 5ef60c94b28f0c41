"""Several simulations stepped at once from their own threads, each on its
own stream: films and a thin stack (whose persistent kernels take turns on the
multiprocessors), a film and a grid on the stage kernels, a large grid, a
batch and a surrogate's gradient.  Every one ends where it ends alone, bit for
bit (the gradient's split sums: 1e-5)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1406_7635_gb300.workloads import Problem, normalise  # noqa: E402


@pytest.fixture(scope="module")
def mm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm as _mm
    return _mm


def problem(nx, ny, nz):
    rng = np.random.default_rng(nx + ny + nz)
    p = Problem(nx, ny, nz, 2e-9, 2e-9, 2e-9)
    p.msat[0], p.aex[0], p.alpha[0] = 8e5, 1.3e-11, 0.1
    m = np.array([1.0, 0.3, 0.2])[:, None, None, None] + 0.3 * rng.standard_normal((3,) + p.shape)
    p.m0 = normalise(m, p.magnetic())
    p.dt0 = 2e-14
    return p


def test_simulations_at_once_end_as_alone(mm):
    grids = [(256, 256, 1, 0), (256, 200, 1, 0), (64, 16, 1, 0), (128, 128, 1, 1), (96, 96, 4, 0), (48, 40, 12, 0),
             (20, 18, 40, 0)]
    ctxs = []
    for nx, ny, nz, which in grids:
        c = mm.Context.from_problem(problem(nx, ny, nz))
        if which:
            c.set_yz_kernels(which)
        ctxs.append(c)
    states = [c.get_state() for c in ctxs]
    specs = [dict(nx=nx, ny=ny, nz=nz, dx=3e-9, dy=3e-9, dz=3e-9, msat=8e5, aex=1.3e-11, alpha=0.1, bext=(0.01, 0, 0))
             for nx, ny, nz in ((32, 32, 1), (96, 96, 4), (32, 32, 1))]
    batch = mm.Batch(specs)
    rng = np.random.default_rng(5)
    bm = [normalise(rng.standard_normal((3, s["nz"], s["ny"], s["nx"])) + np.array([3.0, 0, 0])[:, None, None, None],
                    np.ones((s["nz"], s["ny"], s["nx"]), bool)).astype(np.float32) for s in specs]
    net = mm.FNO(64, 64, width=32, layers=2, modes_x=12, modes_y=12, max_batch=2)
    u, y = torch.randn((2, 2, 3, 64, 64), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    t_end = [0.0]

    def stepper(c, s):
        def go():
            c.set_state(s)
            for n in (1, 30, 7):
                c.step(n)
            return c.get_m()
        return go

    def run_batch():
        for i, m in enumerate(bm):
            batch.set_m(i, m)
        batch.set_solver(dt0=2e-14, dt_max=4e-14)
        t_end[0] += 2.0 ** -41
        batch.run(t_end[0])
        return np.concatenate([batch.get_m(i).ravel() for i in range(len(specs))])

    def gradients():
        for _ in range(5):
            g, _ = net.grad(u, y, 2)
        return g

    jobs = [stepper(c, s) for c, s in zip(ctxs, states)] + [run_batch, gradients]
    alone = [j() for j in jobs]
    for _ in range(2):
        got, err = [None] * len(jobs), []

        def work(i):
            try:
                got[i] = jobs[i]()
            except Exception as e:               # noqa: BLE001 (reported below)
                err.append((i, e))
        threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not err, err
        for i in range(len(ctxs)):
            assert np.array_equal(got[i], alone[i]), grids[i]
        # (the batch's clock goes on: the last step of a span differs by the rounding of its end, 1e-15 of it,
        # which can turn a coefficient, at most 0.1, by one unit in the last place, and the torque in rad by that)
        assert np.abs(got[-2] - alone[-2]).max() <= 2e-6
        assert np.abs(got[-1] - alone[-1]).max() <= 1e-5 * np.abs(alone[-1]).max()
    for c in ctxs:
        c.close()
    batch.close()
    net.close()

"""The batch's fused stages at the edges of a block of cells (fewer than one,
exactly one, a little more, a remainder over several layers), with rejected
attempts and a second run from new states, against the float64 oracle
replaying each instance's own accepted steps.

Tolerance: as for every float32 trajectory of this length, 1e-5 in |m| (a few
dozen roundings of 6e-8 per stage over at most a few dozen steps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.rk45 import RK45  # noqa: E402
from paper_1406_7635_gb300.workloads import batch_instances, problem_from_instance  # noqa: E402

M_TOL = 1e-5


@pytest.mark.parametrize("shape", [(17, 9, 1), (32, 8, 1), (43, 6, 1), (20, 13, 3)])
def test_stages_vs_oracle_replay(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm
    specs, m0s = batch_instances(3, shapes=(shape,), seed=13)
    b = mm.Batch(specs)
    b.set_solver(dt0=5e-13)
    seen = [0] * len(specs)
    rejected = 0
    for run in range(2):
        starts = [np.roll(m, run, axis=-1) for m in m0s]
        for i, m in enumerate(starts):
            b.set_m(i, m)
        b.run((run + 1) * 3e-12)
        for i, m in enumerate(starts):
            dts = b.get_dt_history(i)
            p = problem_from_instance(specs[i], m)
            ora = RK45(p, m=p.m0.astype(np.float32).astype(np.float64))
            ora.run_fixed(dts[seen[i]:])
            assert np.abs(b.get_m(i).astype(np.float64) - ora.m).max() <= M_TOL
            seen[i] = len(dts)
        rejected = sum(b.get_stats(i)["rejected"] for i in range(len(specs)))
    assert rejected > 0
    b.close()

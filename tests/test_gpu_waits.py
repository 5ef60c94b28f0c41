"""Both kinds of bounded waits, each on the path that has them: the row-stage
kernels' on their tensor copies (grids of five and more layers by default, and
thin stacks with the stage kernels asked for) and the film kernel's grid
barriers (thin stacks by default).  With the wait limit at 0 cycles the first
wait gives up at once; the call reports which wait it was, m, t and dt are
those before the abandoned attempt, and with the default limit restored the
context continues bit for bit as one that never timed out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1406_7635_gb300.workloads import Problem, normalise  # noqa: E402

MM_ERR_TIMEOUT = -6
DEFAULT_WAIT = 1 << 30


@pytest.fixture(scope="module")
def mm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm as _mm
    return _mm


def tensor_copy_problem(nz):
    """20 x 30 x nz cells: rows of 32 complex values, 8 rows per block, ny even
    and nx a multiple of 4, so the row kernels move their data by tensor
    copies."""
    rng = np.random.default_rng(4242 + nz)
    shape = (nz, 30, 20)
    p = Problem(20, 30, nz, 2e-9, 2e-9, 2e-9)
    p.region = rng.integers(0, 3, size=shape).astype(np.uint8)
    for r in range(3):
        p.msat[r] = rng.uniform(6e5, 1.1e6)
        p.aex[r] = rng.uniform(1.0e-11, 1.6e-11)
        p.alpha[r] = rng.uniform(0.05, 0.3)
        p.b0[r] = rng.uniform(-0.03, 0.03, 3)
    p.mask = (rng.uniform(size=shape) > 0.05).astype(np.uint8)
    p.m0 = normalise(rng.standard_normal((3,) + shape), p.magnetic())
    return p


@pytest.mark.parametrize("nz,stage_kernels,text", [(4, True, "tensor copies"), (6, False, "tensor copies"),
                                                   (4, False, "grid barrier")])
def test_expired_wait_is_reported_and_the_context_stays_usable(mm, nz, stage_kernels, text):
    p = tensor_copy_problem(nz)

    def context():
        c = mm.Context.from_problem(p)
        if stage_kernels:
            assert c.set_yz_kernels(1) == 1
        return c

    ref = context()
    ref.step(3)
    m_ref, t_ref, s_ref = ref.get_m(), ref.get_time(), ref.get_stats()
    assert (s_ref["launches"] == 2) == (text == "grid barrier")   # (first stage, then all steps: the film kernel)
    ref.close()

    ctx = context()
    ctx.step(1)
    m1, t1, s1 = ctx.get_m(), ctx.get_time(), ctx.get_stats()
    ctx.set_wait_limit(0)
    for _ in range(2):   # the error path twice in a row
        with pytest.raises(mm.MMError) as ei:
            ctx.step(1)
        assert ei.value.code == MM_ERR_TIMEOUT
        assert text in str(ei.value)
        assert np.array_equal(ctx.get_m(), m1)
        assert ctx.get_time() == t1
        s = ctx.get_stats()
        assert (s["accepted"], s["rejected"]) == (s1["accepted"], s1["rejected"])
    ctx.set_wait_limit(DEFAULT_WAIT)
    ctx.step(2)
    assert np.array_equal(ctx.get_m(), m_ref)
    assert ctx.get_time() == t_ref
    s = ctx.get_stats()
    assert (s["accepted"], s["rejected"]) == (s_ref["accepted"], s_ref["rejected"])
    ctx.close()

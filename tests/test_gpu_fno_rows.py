"""The fused backward pass with several image rows per block: batches whose
rows are a few times the blocks that one multiprocessor count gives (four per
multiprocessor, divided over the 128-pixel ranges), so that a block refills
its tiles, keeps its weight gradient over rows and goes from one sample to the
next.  Widths that do and do not move in 16-byte loads, one and two layers.
Gradients against the float64 oracle per parameter group: relative L2 2e-2
and cosine 0.999, the bars of bfloat16 operands (2^-9 per rounding) of the
other surrogate tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.fno import backward, dft_mats, forward, init_params  # noqa: E402

C = 32
CASES = [(3, 2, 401, 130, 3, 3), (3, 2, 403, 132, 5, 3), (2, 1, 811, 60, 4, 2)]


@pytest.fixture(scope="module")
def mm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm as _mm
    return _mm


@pytest.mark.parametrize("S,L,H,W,Mx,My", CASES)
def test_gradients_vs_oracle(mm, S, L, H, W, Mx, My):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert S * H > 2 * (4 * sms // ((W + 127) // 128))   # (at least three rows in some blocks)
    rng = np.random.default_rng(78)
    params = init_params(C, L, Mx, My, seed=10)
    for k in list(params):
        if k.startswith("b") or k in ("p", "q"):
            params[k] = 0.1 * rng.standard_normal(params[k].shape)
    mats = dft_mats(H, W, Mx, My)
    u, y = rng.standard_normal((2, S, 3, H, W))
    y *= (1.0 + np.arange(S))[:, None, None, None]       # (samples that differ in weight)
    total, grads = float(np.sum(y * y)), None
    for s in range(S):
        out, cache = forward(params, u[s], L, mats)
        g = backward(params, cache, out, y[s], L, mats)
        scale = float(np.sum(y[s] * y[s])) / total       # (backward normalises by its own sample)
        grads = {k: v * scale + (grads[k] if grads else 0.0) for k, v in g.items()}
    names = ["P", "p"] + [f"{n}{l}" for l in range(L) for n in "WbR"] + ["Q", "q"]

    def flat(d, name):
        v = d[name]
        return (np.stack([v.real, v.imag], axis=-1) if name[0] == "R" else v).ravel()

    net = mm.FNO(H, W, width=C, layers=L, modes_x=Mx, modes_y=My, max_batch=S)
    net.set_params(np.concatenate([flat(params, n) for n in names]).astype(np.float32))
    ud = torch.tensor(u.astype(np.float32), device="cuda").contiguous()
    yd = torch.tensor(y.astype(np.float32), device="cuda").contiguous()
    g_gpu, _ = net.grad(ud, yd, S)
    net.close()
    off = 0
    for name in names:
        b = flat(grads, name)
        a = g_gpu[off:off + b.size].astype(np.float64)
        off += b.size
        assert np.linalg.norm(a - b) <= 2e-2 * np.linalg.norm(b), name
        assert np.dot(a, b) >= 0.999 * np.linalg.norm(a) * np.linalg.norm(b), name
    assert off == g_gpu.size

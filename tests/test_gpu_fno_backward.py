"""The fused backward pass of the width-32 surrogate at the edges of its
tiles: one layer (top and lift passes only), rows ragged in the 128-pixel
ranges and not a multiple of 4, mode counts that do not fill 16-wide product
steps, the largest it takes (2 Mx = 64) and the first it leaves to the GEMMs
(2 Mx = 66).  Gradients against the float64 oracle per parameter group:
relative L2 2e-2 and cosine 0.999, the bars of bfloat16 operands (2^-9 per
rounding) of the other surrogate tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.fno import backward, dft_mats, forward, init_params  # noqa: E402

C = 32
CASES = [(1, 1, 6, 20, 3, 2), (3, 2, 10, 130, 8, 3), (2, 2, 12, 260, 24, 4), (1, 2, 8, 64, 32, 3), (1, 2, 8, 80, 33, 3),
         (2, 3, 5, 128, 5, 2)]


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
    rng = np.random.default_rng(77)
    params = init_params(C, L, Mx, My, seed=9)
    for k in list(params):
        if k.startswith("b") or k in ("p", "q"):
            params[k] = 0.1 * rng.standard_normal(params[k].shape)
    mats = dft_mats(H, W, Mx, My)
    u, y = rng.standard_normal((2, S, 3, H, W))
    total, grads = float(np.sum(y * y)), None
    for s in range(S):
        out, cache = forward(params, u[s], L, mats)
        g = backward(params, cache, out, y[s], L, mats)
        scale = float(np.sum(y[s] * y[s])) / total     # (backward normalises by its own sample)
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
    again, _ = net.grad(ud, yd, S)
    net.close()
    off = 0
    for name in names:
        b = flat(grads, name)
        a = g_gpu[off:off + b.size].astype(np.float64)
        # (accumulated anew on each call)
        assert np.allclose(again[off:off + b.size], a, rtol=1e-3, atol=1e-5 * np.abs(a).max())
        off += b.size
        assert np.linalg.norm(a - b) <= 2e-2 * np.linalg.norm(b), name
        assert np.dot(a, b) >= 0.999 * np.linalg.norm(a) * np.linalg.norm(b), name
    assert off == g_gpu.size

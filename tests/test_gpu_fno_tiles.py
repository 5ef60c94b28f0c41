"""The surrogate's y products where a thread computes several outputs of a
column: frequencies that fill a block's groups and that leave a remainder,
several groups of blocks, rows that end inside a thread's outputs, against
the float64 oracle.

Tolerance: the dense products around them round their operands to bfloat16
(relative rounding 2^-9 per operand): 2e-2 in relative L2 norm and cosine
>= 0.999, as for the other products."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.fno import backward, dft_mats, forward, init_params  # noqa: E402

from test_gpu_fno import cosine, flatten, rel  # noqa: E402


# (S, C, H, W, Mx, My): y frequencies per block and thread: 48 of 50 by 5;
# 40 = 8 x 5 exactly; 96 in two groups of 64 (8 each); 6 x 4 of 5; rows 97 and 50
@pytest.mark.parametrize("S,C,H,W,Mx,My", [(2, 4, 97, 64, 24, 24), (1, 8, 50, 80, 32, 20), (1, 4, 100, 64, 32, 48),
                                           (1, 4, 33, 128, 48, 12)])
def test_y_products_vs_oracle(S, C, H, W, Mx, My):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1406_7635_gb300.build import build
    build()
    from paper_1406_7635_gb300 import mm
    rng = np.random.default_rng(5)
    params = init_params(C, 1, Mx, My, seed=6)
    mats = dft_mats(H, W, Mx, My)
    u, y = rng.standard_normal((S, 3, H, W)), rng.standard_normal((S, 3, H, W))
    yh = [forward(params, u[s], 1, mats) for s in range(S)]
    ysq = float(np.sum(y * y))
    g_ora = 0.0
    for s in range(S):
        g = backward(params, yh[s][1], yh[s][0], y[s], 1, mats)
        g_ora = g_ora + flatten(g, 1) * (float(np.sum(y[s] * y[s])) / ysq)
    net = mm.FNO(H, W, width=C, layers=1, modes_x=Mx, modes_y=My, max_batch=S)
    net.set_params(flatten(params, 1).astype(np.float32))
    ud = torch.tensor(u.astype(np.float32), device="cuda").contiguous()
    yd = torch.tensor(y.astype(np.float32), device="cuda").contiguous()
    out = torch.empty_like(ud)
    net.forward(ud, out, S)
    assert rel(out.cpu().numpy().astype(np.float64), np.stack([a[0] for a in yh])) < 2e-2
    g_gpu = net.grad(ud, yd, S)[0].astype(np.float64)
    off = 3 * C + C + C * C + C
    R = slice(off, off + 2 * C * C * 2 * My * Mx)
    assert cosine(g_gpu[R], g_ora[R]) >= 0.999 and rel(g_gpu[R], g_ora[R]) <= 2e-2
    net.close()

"""The surrogate's kernels at the edges of their tiles against the FP64 oracle network: channel counts
around the blocks of 4, 8, 16 and 32 outputs and of one warp, grids whose rows of positions are no
multiple of four, weights that start on 2, 4 or 16 bytes, batches past a block of four.

Tolerances as in test_gpu_fno.py (FP32 accumulation of at most 128 terms per map, a few maps deep); the
contiguous-axis products run on the CUDA cores here (tensor cores round to TF32).
"""
import numpy as np
import pytest
import torch

from oracle import fno as ofno

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _bf16(a):
    u = np.asarray(a, dtype=np.float32).view(np.uint32).astype(np.uint64)
    return ((((u + 0x7FFF + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32)).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,W,modes,layers,c_in,c_out,B",
                         [(8, 1, 2, 1, 1, 1, 1), (9, 3, 2, 2, 4, 1, 5), (10, 5, 3, 2, 3, 2, 4), (12, 8, 4, 2, 4, 5, 2),
                          (11, 17, 3, 1, 2, 9, 3), (16, 16, 6, 2, 4, 16, 9), (12, 20, 3, 3, 4, 1, 2), (8, 32, 3, 2, 33, 17, 2),
                          (9, 33, 2, 2, 5, 3, 1), (8, 48, 2, 1, 4, 33, 6), (8, 64, 3, 2, 64, 64, 2), (8, 32, 2, 1, 4, 1, 130)])
def test_forward_and_backward_match_the_oracle(n, W, modes, layers, c_in, c_out, B):
    from paper_2310_07119_gb300 import _lib as L
    from paper_2310_07119_gb300.fno import FNO
    cfg = dict(W=W, c_in=c_in, c_out=c_out, modes=modes, layers=layers)
    rng = np.random.default_rng(n + W)
    theta = rng.normal(scale=0.6 / np.sqrt(W), size=ofno.num_params(**cfg))
    x = rng.normal(size=(B, c_in, n, n, n)).astype(np.float32).astype(np.float64)
    dy = rng.normal(size=(B, c_out, n, n, n)).astype(np.float32).astype(np.float64)
    th, o = theta.astype(np.float32).astype(np.float64), 0
    for name, sh in ofno.param_shapes(**cfg):
        k = int(np.prod(sh))
        if name[0] in "PRWQ":
            th[o:o + k] = _bf16(theta[o:o + k])
        o += k
    m = FNO(n, W, modes, layers, c_in, c_out)
    L.load().twa_fno_set_tensor_cores(m.h, 0)
    m.set_params(torch.tensor(theta, dtype=torch.float32))
    y = m.forward(torch.tensor(x, dtype=torch.float32, device="cuda")).double().cpu().numpy()
    m.zero_grad()
    dx = m.backward(torch.tensor(dy, dtype=torch.float32, device="cuda"), want_dx=True).double().cpu().numpy()
    g = m.get_params(which=1).double().cpu().numpy()
    m.close()
    yo, cache = ofno.forward(th, x, **cfg, keep=True)
    go, dxo = ofno.backward(th, cache, dy, **cfg)
    assert np.max(np.abs(y - yo)) < 1e-4 * np.max(np.abs(yo))
    assert np.linalg.norm(dx - dxo) < 2e-4 * np.linalg.norm(dxo)
    o = 0
    for name, sh in ofno.param_shapes(**cfg):
        k = int(np.prod(sh))
        assert np.linalg.norm(g[o:o + k] - go[o:o + k]) <= 2e-3 * np.linalg.norm(go[o:o + k]) + 1e-9, name
        o += k

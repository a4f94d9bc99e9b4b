"""The FP64 path's streams are independent: what one stream holds changes no bit of another's."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(n, bad, change, steps=3):
    from paper_2310_07119_gb300 import Ensemble, F64_PLAIN
    ens = Ensemble([(len(n), n, 1.0)], 0.1, 4 * np.pi, 1e-3, 1e6, [4], precision=F64_PLAIN)
    rng = np.random.default_rng(2)
    psi = 1.0 + 0.3 * (rng.normal(size=(5, int(np.prod(n)))) + 1j * rng.normal(size=(5, int(np.prod(n)))))
    if bad is not None:
        change(psi[bad])
    ens.psi.copy_(torch.tensor(psi.reshape(-1)))
    series = ens.advance(steps, steps).cpu().numpy()[:, 0]
    got = torch.view_as_real(ens.fields(0)).reshape(5, -1).cpu()
    ens.close()
    return got, series


def _nan(f):
    f[5] = np.nan


def _inf(f):
    f[3] = np.inf


def _large(f):
    f *= 1e6


@pytest.mark.parametrize("n", [(64,), (8, 8), (64, 32), (8, 16, 8), (32, 32, 64)])
@pytest.mark.parametrize("change", [_nan, _inf, _large])
@pytest.mark.parametrize("bad", [0, 1, 4])          # the classical field, its neighbour, the last of an odd count
def test_a_stream_leaves_the_others_alone(n, change, bad):
    clean, _ = _run(n, None, None)
    got, series = _run(n, bad, change)
    for s in range(5):
        if s != bad:
            assert torch.equal(got[s], clean[s]), s
    finite = bool(torch.isfinite(got[bad]).all())
    assert finite == (change is _large)
    # a stream that is not finite spreads over all its own cells in a step, and over nothing else
    assert series[-1, 4] == (0 if finite or bad == 0 else int(np.prod(n)))

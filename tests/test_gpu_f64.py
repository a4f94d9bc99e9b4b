"""The FP64 path against the FP64 oracle at every line length, and its chunks and whole 1D runs.

Tolerance: a step makes at most six line transforms along each axis of at most 11 levels, a level adds
at most 2 eps relative to the field's norm, and rounding errors add at most linearly:
5 steps x 6 x 33 x 2 x 2.2e-16 < 5e-13 (the oracle's own transforms are far inside it).
"""
import numpy as np
import pytest
import torch

from oracle import sp

pytestmark = pytest.mark.gpu
TOL = 5e-13


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _ens(n, n_real, hbar=0.1, C=4 * np.pi, dt=1e-3, seed=1, n_tot=1e6, modes=True):
    from paper_2310_07119_gb300 import Ensemble, F64_PLAIN
    ens = Ensemble([(len(n), n, 1.0)], hbar, C, dt, n_tot, [n_real], precision=F64_PLAIN, want_modes=modes)
    rng = np.random.default_rng(seed)
    shape = (n_real + 1,) + tuple(reversed(n))
    psi = 1.0 + 0.3 * rng.normal(size=shape) + 0.3j * rng.normal(size=shape)
    ens.psi.copy_(torch.tensor(psi.reshape(-1)))
    return ens, psi


def _rel(a, b):
    ax = tuple(range(1, a.ndim))
    return np.max(np.sqrt(np.sum(np.abs(a - b) ** 2, axis=ax) / np.sum(np.abs(b) ** 2, axis=ax)))


@pytest.mark.parametrize("n", [(8,), (16,), (32,), (64,), (128,), (256,), (512,), (1024,), (2048,), (8, 8), (8, 2048),
                               (2048, 8), (1024, 16), (32, 512), (128, 256), (8, 8, 8), (16, 8, 64), (64, 32, 8),
                               (8, 128, 16), (8, 8, 256)])
@pytest.mark.parametrize("n_real,C", [(1, 4 * np.pi), (4, 400.0)])      # even and odd slots; kicks past 1/4
def test_steps_match_the_oracle(n, n_real, C):
    ens, psi = _ens(n, n_real, C=C)
    ens.step(5)
    got = ens.fields(0).cpu().numpy()
    ens.close()
    for _ in range(5):
        psi = sp.step(psi, 0.1, C, 1e-3, 1.0, len(n))
    assert _rel(got, psi) < TOL


@pytest.mark.parametrize("n", [(8,), (256,), (2048,), (64, 32)])
def test_a_run_equals_its_steps_and_moments(n):
    """Whole runs (1D: in one or several launches; 2048 x 60 needs one per few outputs) against
    step and moments calls: the fields to rounding, the scalars to the sums' rounding."""
    n_real, outs = (60 if n == (2048,) else 5), 9
    a, _ = _ens(n, n_real)
    b, _ = _ens(n, n_real)
    series = a.advance(2 * outs, 2).cpu().numpy()[:, 0]
    for o in range(outs + 1):
        if o:
            b.step(2)
        m = b.moments(0)["scalars"].cpu().numpy()
        assert np.allclose(series[o], m, rtol=1e-11, atol=1e-11 * np.abs(m[:4]).max())
    assert _rel(a.fields(0).cpu().numpy(), b.fields(0).cpu().numpy()) < 4 * TOL
    a.close()
    b.close()


def test_non_finite_values_are_counted():
    for n in ((256,), (16, 16)):
        ens, _ = _ens(n, 3)
        ens.fields(0)[2].view(-1)[5] = float("nan")
        s = ens.advance(0, 1).cpu().numpy()
        assert s[0, 0, 4] == 1.0
        ens.close()


def test_chunked_batches_equal_whole_ones():
    """40 streams of 2048^2 need three chunks of the Poisson workspace: slots 32..35 (a chunk's
    start) bitwise as in a batch of their own."""
    n = (2048, 2048)
    from paper_2310_07119_gb300 import Ensemble, F64_PLAIN
    big = Ensemble([(2, n, 1.0)], 0.1, 4 * np.pi, 1e-3, 1e6, [40], precision=F64_PLAIN, want_modes=False)
    g = torch.Generator(device="cuda").manual_seed(3)
    big.psi.real.normal_(1.0, 0.3, generator=g)
    small = Ensemble([(2, n, 1.0)], 0.1, 4 * np.pi, 1e-3, 1e6, [3], precision=F64_PLAIN, want_modes=False)
    small.fields(0).copy_(big.fields(0)[32:36])
    big.step(2)
    small.step(2)
    assert torch.equal(torch.view_as_real(big.fields(0)[32:36]), torch.view_as_real(small.fields(0)))
    big.close()
    small.close()

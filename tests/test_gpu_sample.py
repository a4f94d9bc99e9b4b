"""FP32 sampling (pairs of floats) against the FP64 oracle, value by value.

A value is rounded to float once from a sum that carries the classical value to 2^-48 and the noise
to 2^-36 relative (two roundings of products on top of 2^-36.7), so each component may be off by half
a unit in the last place of the result, 2^-24 |z|, and 2^-35 of the noise.
"""
import numpy as np
import pytest
import torch

from oracle import twa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sample(n, n_real, n_tot, cl, seed):
    from paper_2310_07119_gb300 import Ensemble
    ens = Ensemble([(len(n), n, 1.0)], 1.0, 1.0, 1e-3, n_tot, [n_real], want_modes=False)
    ens.sample([cl], seed)
    got = ens.fields(0).cpu().numpy().reshape(n_real + 1, -1)
    ens.close()
    return got


# fewer cells than a block, fewer values than a block, odd slot counts around the slots per thread (16
# once there is enough work), several slot groups, and the sigma at which FP64 takes over
@pytest.mark.parametrize("n,n_real,n_tot", [((8,), 1, 1e4), ((8,), 300, 1e6), ((256,), 33, 1e4), ((64, 32), 15, 1e9),
                                            ((64, 64, 64), 16, 1e9), ((128, 128, 32), 31, 1e9), ((32,), 3, 1e-12),
                                            ((32,), 3, 1e-30)])
@pytest.mark.parametrize("zero", [False, True])
def test_sample_matches_the_oracle_to_its_rounding(n, n_real, n_tot, zero):
    cells = int(np.prod(n))
    rng = np.random.default_rng(3)
    cl = np.zeros(cells, complex) if zero else rng.normal(size=cells) + 1j * rng.normal(size=cells)
    seed = 0x123456789ABCDEF1
    got = _sample(n, n_real, n_tot, cl, seed)
    ref = twa.sample(cl.reshape(tuple(reversed(n))), seed, n_real, n_tot, 1.0 / cells).reshape(n_real + 1, cells)
    noise = ref - cl[None]
    for a, b, z in ((got.real, ref.real, noise.real), (got.imag, ref.imag, noise.imag)):
        assert np.all(np.abs(a - b) <= 2.0 ** -24 * np.abs(b) + 2.0 ** -35 * np.abs(z) + 2.0 ** -149)


def test_values_that_are_no_finite_floats_pass_through():
    cl = np.array([np.inf, -np.inf, 1e300, 3.4e38, 1e-300, 0.0, 1.0, 2.0], complex)
    cl[7] = np.nan
    got = _sample((8,), 2, 1e4, cl, 5)
    ref = twa.sample(cl, 5, 2, 1e4, 1.0 / 8)
    with np.errstate(over="ignore", invalid="ignore"):
        f = ref.real.astype(np.float32)
    assert np.array_equal(np.isnan(f), np.isnan(got.real))
    assert np.array_equal(f[np.isinf(f)], got.real[np.isinf(f)])

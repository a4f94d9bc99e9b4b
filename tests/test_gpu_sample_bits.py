"""FP32 sampling against FP64 sampling rounded once: the same bits, also where the classical value and the noise
cancel, the noise is all there is, or the value is no finite float."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sample(n, n_real, n_tot, cl, precision, noise_conv):
    from paper_2310_07119_gb300 import Ensemble
    ens = Ensemble([(len(n), n, 1.0)], 1.0, 1.0, 1e-3, n_tot, [n_real], precision=precision, want_modes=False,
                   noise_conv=noise_conv)
    ens.sample([cl], 0x9E3779B97F4A7C15)
    got = torch.view_as_real(ens.psi.clone()).float()
    ens.close()
    return got


@pytest.mark.parametrize("n,n_real", [((8,), 1), ((256,), 33), ((64, 64), 7), ((128, 128, 128), 64)])
@pytest.mark.parametrize("n_tot", [1e4, 1e9, 1e-12])
@pytest.mark.parametrize("scale", [0.0, 1.0, 1e-3])
def test_float_fields_hold_the_fp64_values_rounded_once(n, n_real, n_tot, scale):
    from paper_2310_07119_gb300 import F32, F64_PLAIN
    rng = np.random.default_rng(4)
    cells = int(np.prod(n))
    cl = scale * (rng.normal(size=cells) + 1j * rng.normal(size=cells))
    for conv in (0, 1):
        a, b = (_sample(n, n_real, n_tot, cl, p, conv) for p in (F32, F64_PLAIN))
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))


def test_values_that_are_no_finite_floats_are_those_of_fp64():
    from paper_2310_07119_gb300 import F32, F64_PLAIN
    cl = np.array([np.inf, -np.inf, 1e300, 3.4028235677973366e38, 1e-300, -0.0, 2.0 ** -149, 1.0], complex)
    cl[7] = complex(np.nan, np.inf)
    a, b = (_sample((8,), 40, 1e4, cl, p, 0) for p in (F32, F64_PLAIN))
    assert torch.equal(torch.isnan(a), torch.isnan(b))
    keep = ~torch.isnan(a)
    assert torch.equal(a[keep], b[keep])

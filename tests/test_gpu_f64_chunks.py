"""The FP64 path where its workspace holds a part of a call: whole 1D runs in several launches, mode moments from
several sets of spectra."""
import numpy as np
import pytest
import torch

from tests.test_gpu_f64 import TOL, _ens, _rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n_real,launches", [(400, 10)])     # a stepping and a summing launch for 2 outputs
def test_a_run_in_several_launches_equals_its_steps_and_moments(n_real, launches):
    from paper_2310_07119_gb300 import twa_last_launch_count
    n, outs = (2048,), 9
    a, _ = _ens(n, n_real)
    b, _ = _ens(n, n_real)
    series = a.advance(2 * outs, 2).cpu().numpy()[:, 0]
    count = twa_last_launch_count(a.h)
    assert count == launches
    for o in range(outs + 1):
        if o:
            b.step(2)
        m = b.moments(0)["scalars"].cpu().numpy()
        assert np.allclose(series[o], m, rtol=1e-11, atol=1e-11 * np.abs(m[:4]).max()), o
    assert _rel(a.fields(0).cpu().numpy(), b.fields(0).cpu().numpy()) < 4 * TOL
    a.close()
    b.close()


def test_mode_moments_of_several_sets_of_spectra():
    """20 streams of 2048^2 against torch's transforms: |a_k|^2 is off by at most 1e-12 of its mean (22 levels of
    2 eps on each amplitude and its square, 64 of 2.2e-16 / 1e-12 to spare; the fields have no mean)."""
    from paper_2310_07119_gb300 import Ensemble, F64_PLAIN
    n, n_real, n_tot = (2048, 2048), 20, 1e6
    ens = Ensemble([(2, n, 1.0)], 0.1, 4 * np.pi, 1e-3, n_tot, [n_real], precision=F64_PLAIN)
    g = torch.Generator(device="cuda").manual_seed(3)
    torch.view_as_real(ens.psi).normal_(0.0, 0.3, generator=g)
    m = ens.moments(0)
    cells = n[0] * n[1]
    s2 = s4 = 0.0
    for s in range(1, n_real + 1):
        f = torch.fft.fft2(ens.fields(0)[s])
        a2 = (f.real ** 2 + f.imag ** 2) * (n_tot / cells ** 2)
        s2, s4 = s2 + a2 / n_real, s4 + a2 ** 2 / n_real
    mean = float(s2.mean())
    nk, var = m["nk_mean"].reshape(n), m["nk_var"].reshape(n)
    assert float((nk - (s2 - 0.5)).abs().max()) < 1e-12 * 40 * mean         # the largest of 4e6 modes: below 40 means
    assert float((var - (s4 - s2 - (s2 - 0.5) ** 2)).abs().max()) < 4e-12 * 40 ** 2 * mean ** 2
    ens.close()

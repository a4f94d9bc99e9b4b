"""The FP64 path's workspace is limited for the handle as a whole, and leaves room for the caller's batch."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
GB = 1 << 30


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _ens(grids, n_real):
    from paper_2310_07119_gb300 import Ensemble, F64_PLAIN
    return Ensemble([(len(n), n, 1.0) for n in grids], 0.1, 4 * np.pi, 1e-3, 1e6, n_real, precision=F64_PLAIN)


def _least(n):
    """Bytes of one half field, the moment sums and one spectrum."""
    cells = int(np.prod(n))
    return cells // n[-1] * (n[-1] // 2 + 1) * 16 + cells * (24 + 16 + 16)


def test_many_instances_share_one_limit():
    """100 instances of 17 fields of 512^2 would take 3.7 GB of Poisson fields and 6.7 GB of spectra."""
    n, n_real = (512, 512), 16
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    many = _ens([n] * 100, [n_real] * 100)
    used = free - torch.cuda.mem_get_info()[0] - many.psi.numel() * 16
    # a few percent: tables, block sums, allocation granularity
    assert used < 1.05 * (2 * GB + 100 * _least(n))
    one = _ens([n], [n_real])
    g = torch.Generator(device="cuda").manual_seed(1)
    torch.view_as_real(many.psi).normal_(0.0, 1.0, generator=g)
    one.psi.copy_(many.fields(77).reshape(-1))
    many.step(1)
    one.step(1)
    assert torch.equal(torch.view_as_real(many.fields(77)), torch.view_as_real(one.fields(0)))
    a, b = many.moments(77), one.moments(0)
    assert all(torch.equal(a[k], b[k]) for k in ("rho_mean", "nk_mean", "nk_var"))
    many.close()
    one.close()


def test_the_batch_has_room_beside_the_workspace():
    n, n_real = (1024, 1024), 88                    # a batch of 1.4 GB; half fields 0.7 GB, spectra 1.4 GB
    torch.cuda.empty_cache()
    batch = (n_real + 1) * n[0] * n[1] * 16
    fill = torch.empty(torch.cuda.mem_get_info()[0] - batch - _least(n) - GB, dtype=torch.uint8, device="cuda")
    ens = _ens([n], [n_real])                       # the handle, then the batch
    ens.psi.fill_(1.0)
    ens.step(1)
    assert all(bool(torch.isfinite(torch.view_as_real(ens.fields(0)[s])).all()) for s in (0, 41, n_real))
    ens.close()
    del fill, ens
    torch.cuda.empty_cache()


# 16 outputs at a time; none (the moment kernels)
@pytest.mark.parametrize("n_real,launches", [(60, 2), (1400, None)])
def test_large_1d_batches_run_by_their_sums_as_far_as_they_fit(n_real, launches):
    from paper_2310_07119_gb300 import twa_last_launch_count
    outs = 9
    a, b = _ens([(2048,)], [n_real]), _ens([(2048,)], [n_real])
    g = torch.Generator(device="cuda").manual_seed(2)
    torch.view_as_real(a.psi).normal_(1.0, 0.3, generator=g)
    b.psi.copy_(a.psi)
    series = a.advance(outs, 1).cpu().numpy()[:, 0]
    count = twa_last_launch_count(a.h)
    assert count == launches if launches else count > 3 * outs
    for o in range(outs + 1):
        if o:
            b.step(1)
        m = b.moments(0)["scalars"].cpu().numpy()
        # as in test_gpu_f64.py: the sums' rounding
        assert np.allclose(series[o], m, rtol=1e-11, atol=1e-11 * np.abs(m[:4]).max()), o
    a.close()
    b.close()

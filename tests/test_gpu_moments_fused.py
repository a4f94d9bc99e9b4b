"""Mode moments whose last axis is transformed and summed in one pass, and the xy-plane transform before
it, against the separate passes the profiler takes: the same bits (each mode's sums run in slot order
in both); only the total over modes, summed by other blocks, may differ by its rounding.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# last axes of 8 to 512 cells with enough lines for the fused pass, square and other planes, one stream
# and even and odd counts; and grids on the near side of each rule
@pytest.mark.parametrize("n,n_real", [((512, 256, 8), 1), ((512, 256, 16), 3), ((256, 256, 32), 2), ((256, 256, 64), 3),
                                      ((128, 128, 128), 9), ((256, 128, 256), 2), ((256, 64, 512), 1), ((64, 64, 64), 4),
                                      ((32, 32, 32), 5), ((16, 16, 8), 2), ((64, 512), 3)])
def test_fused_mode_moments_keep_their_bits(n, n_real):
    from paper_2310_07119_gb300 import Ensemble, twa_profile_enable
    ens = Ensemble([(len(n), n, 1.0)], 0.0122, 12.566, 1e-4, 1e6, [n_real])
    gen = torch.Generator(device="cuda").manual_seed(5)
    torch.view_as_real(ens.psi).normal_(1.0, 0.3, generator=gen)
    start = ens.psi.clone()
    got = []
    for prof in (False, True):
        twa_profile_enable(ens.h, prof)
        ens.psi.copy_(start)
        m = ens.moments(0)
        series = ens.advance(2, 1)      # moments with a pending kick
        got.append((m, series))
    twa_profile_enable(ens.h, False)
    (a, sa), (b, sb) = got
    for k in a:
        if k != "scalars":
            assert torch.equal(a[k], b[k]), k
    for x, y in ((a["scalars"], b["scalars"]), (sa, sb)):
        assert torch.equal(x[..., :5], y[..., :5]) and torch.equal(x[..., 6:], y[..., 6:])
        assert torch.allclose(x, y, rtol=1e-12, atol=1e-9)
    ens.close()

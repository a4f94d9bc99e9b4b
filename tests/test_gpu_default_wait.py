"""An untuned handle of long columns copies its tiles by TMA, so its bounded waits are part of what twa.h promises: a
wait that runs out is reported by twa_sync_status, and the handle goes on."""
import pytest
import torch

from paper_2310_07119_gb300 import _lib as L


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(64, 1024), (16, 2048), (16, 64, 16)])
def test_an_untuned_handle_reports_a_tile_that_never_comes(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_07119_gb300 import Ensemble, twa_debug_stall_next_tma, twa_set_wait_limit, twa_sync_status
    ens = Ensemble([(len(n), n, 1.0)], 0.1, 1.0, 1e-4, 1e6, [3])
    g = torch.Generator(device="cuda").manual_seed(1)
    psi = torch.randn(ens.psi.shape, dtype=torch.complex64, device="cuda", generator=g)

    def step():
        ens.psi.copy_(psi)
        ens.step(2)
        return torch.view_as_real(ens.psi.clone())

    want = step()
    assert twa_sync_status(ens.h) == L.TWA_OK
    twa_set_wait_limit(ens.h, 0.05)
    twa_debug_stall_next_tma(ens.h)
    step()
    assert twa_sync_status(ens.h) == L.TWA_ETIMEOUT
    assert torch.equal(step(), want)
    assert twa_sync_status(ens.h) == L.TWA_OK
    ens.close()


def test_the_header_names_the_waits_of_untuned_handles():
    text = " ".join(open(L.HEADER).read().split())
    assert "a bounded wait gave up, of the persistent launch or of a pass whose tiles TMA copies" in text

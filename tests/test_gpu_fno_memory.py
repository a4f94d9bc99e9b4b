"""The surrogate after a batch that the GPU has no room for: nothing is left of it."""
import numpy as np
import pytest
import torch

from paper_2310_07119_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("layers", [1, 3])
@pytest.mark.parametrize("part", [False, True])     # the first allocation fails, or one after several
def test_a_batch_without_room_leaves_a_working_model(layers, part):
    from paper_2310_07119_gb300.fno import FNO
    n, W = 16, 16
    m = FNO(n, W, 2, layers, 4, 1)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(2, 4, n, n, n, device="cuda", generator=g)
    dy = torch.randn(2, 1, n, n, n, device="cuda", generator=g)

    def both():
        m.zero_grad()
        y = m.forward(x)
        return y, m.backward(dy, want_dx=True), m.get_params(which=1)

    want = both()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    act = W * n ** 3 * 4                            # bytes of one activation of one input
    # part: all activations take 0.6 of what is free (layers inputs and as many outputs), the workspaces do not fit
    B = int(0.3 * free / (layers * act)) if part else 2 ** 31 - 1
    lib = L.load()
    for _ in range(2):                              # the second finds what the first left
        assert lib.twa_fno_forward(m.h, x.data_ptr(), B, dy.data_ptr(), None) == L.TWA_ENOMEM
        # the activations of the forward before are gone
        assert lib.twa_fno_backward(m.h, dy.data_ptr(), 2, None, None) == L.TWA_EINVAL
        assert torch.cuda.mem_get_info()[0] >= free
    got = both()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    m.close()

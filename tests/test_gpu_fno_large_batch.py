"""The spectral weight gradient of a batch whose inputs of one mode do not fit shared memory (more than 6400 values
of batch times width + 1: k_mix_wgrad_any), against the oracle network as in test_gpu_fno_shapes.py."""
import pytest

from tests import test_gpu_fno_shapes as shapes

pytestmark = pytest.mark.gpu
_cuda = shapes._cuda


@pytest.mark.parametrize("n,W,modes,layers,c_in,c_out,B", [(8, 64, 1, 1, 4, 1, 100), (8, 3, 2, 1, 2, 1, 1700)])
def test_batches_past_shared_memory_match_the_oracle(n, W, modes, layers, c_in, c_out, B):
    assert 2 * B * (W + 1) * 8 > 100 * 1024
    shapes.test_forward_and_backward_match_the_oracle(n, W, modes, layers, c_in, c_out, B)

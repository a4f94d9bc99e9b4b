"""The tensor-core GEMM where a CTA walks through many row tiles: the barriers' phases come round again, and the
products of a tile overlap the stores of the one before, in every form of the epilogue (accumulating, rows that
are no multiple of 16 bytes or of 16 values, all 512 accumulator columns).  Bound as in test_gpu_tc_gemm.py."""
import pytest
import torch

from paper_2310_07119_gb300 import _lib
from tests.test_gpu_tc_gemm import TOL, _call

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,Np,acc", [(128, 64, 64, 1), (64, 100, 112, 0), (32, 13, 16, 1), (64, 256, 256, 0),
                                        (64, 250, 256, 1)])
def test_every_row_of_six_tiles_a_cta(K, N, Np, acc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    P = sms * 128 * 6 + 5                           # at least six tiles for every CTA, the last one of five rows
    g = torch.Generator(device="cuda").manual_seed(K + N)
    A, B, C = (torch.randn(r, c, device="cuda", generator=g) for r, c in ((P, K), (Np, K), (P, N)))
    B[N:] = 0.0
    c0 = C.double() * acc
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rc = _call(A.data_ptr(), P, K, K, B.data_ptr(), N, Np, C.data_ptr(), N, acc, err.data_ptr())
    assert rc == 0, _lib.load().twa_last_error(None)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    a, b = A.double(), B[:N].double()
    bound = TOL * (a.abs() @ b.abs().T) + 1e-6 * (c0.abs() + 1)
    assert torch.all((C.double() - (c0 + a @ b.T)).abs() <= bound)

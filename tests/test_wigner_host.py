"""The accuracy of the float-pair functions behind the sampling of float fields, held on the host (the same
arithmetic, one lane): relative errors up to 2^-40.4 of the radius and 2^-36.6 of the directions, which the kernel's
bound on a value's error is made of (round_sum in misc.cu).  All 2^32 words give 2^-40.463, 2^-36.648 and 2^-36.648
(a quarter of an hour of one core); here every word where a reduction changes and 2e7 random ones."""
import math
import os
import subprocess

from paper_2310_07119_gb300.build import CSRC, _nvcc

HERE = os.path.dirname(os.path.abspath(__file__))


def test_float_pair_functions_hold_their_stated_accuracy(tmp_path):
    exe = str(tmp_path / "wigner_host")
    # host code only; no contraction of its products into fused multiply-adds, as on the GPU
    subprocess.run([_nvcc(), "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(HERE, "native", "wigner_host.cu"), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe, "20000000"], check=True, capture_output=True, text=True).stdout.split()
    assert int(out[0]) > 20000000
    for name, most, bits, word in zip(("radius", "cosine", "sine"), (-40.4, -36.6, -36.6), out[1::2], out[2::2]):
        assert math.isfinite(float(bits)) and float(bits) < most, (name, bits, word)

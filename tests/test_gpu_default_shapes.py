"""The pass shapes taken without the tuner give the same bits as plain single-field shapes.

Every rule of the default shapes (half-size CTAs, two-field passes by slot count, TMA and pipelined
columns, axis passes for the fields of cubes from 128 cells) only regroups the same per-line
arithmetic, so fields, scalars and mode moments must agree bitwise with the shapes of 256 threads per
CTA and, for square planes, the plane pipeline, forced through a tuner cache.
"""
import json

import pytest
import torch

pytestmark = pytest.mark.gpu

T = {8: 1, 16: 1, 32: 2, 64: 8, 128: 8, 256: 16, 512: 32, 1024: 64, 2048: 128}   # threads per line


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _plain(n, slots):
    out = {}
    g = list(n) + [1] * (3 - len(n))
    for axis in range(len(n)):
        lines = max(4 if axis else 1, 256 // T[n[axis]])
        for op in range(12):
            out[f"{g[0]}x{g[1]}x{g[2]}:slots{slots}:axis{axis}:op{op}"] = lines
    out[f"{g[0]}x{g[1]}x{g[2]}:slots{slots}:axis9:op0"] = 1
    return out


# slot counts around the two-field rule (odd below nine, even, odd above), every length as a column,
# planes with fewer columns than a full TMA tile row has, cubes on both sides of 128
@pytest.mark.parametrize("n,n_real", [((8, 32), 1), ((8, 64), 2), ((16, 128), 8), ((8, 256), 3), ((8, 512), 2), ((8, 1024), 1),
                                      ((8, 2048), 2), ((1024, 8), 1), ((2048, 16), 2), ((512, 1024), 2), ((32, 32, 32), 8),
                                      ((64, 64, 64), 3), ((64, 64, 64), 64), ((128, 128, 128), 2), ((128, 128, 16), 9),
                                      ((256, 256, 8), 1), ((64, 128, 256), 7), ((64, 32, 16), 2), ((256, 64, 128), 8),
                                      ((8, 256, 128), 9)])
def test_default_shapes_match_plain_shapes_bitwise(n, n_real, tmp_path):
    from paper_2310_07119_gb300 import Ensemble
    got = []
    for forced in (False, True):
        ens = Ensemble([(len(n), n, 1.0)], 0.0122, 12.566, 1e-4, 1e6, [n_real])
        gen = torch.Generator(device="cuda").manual_seed(7)
        if forced:
            path = tmp_path / "shapes.json"
            path.write_text(json.dumps(_plain(n, n_real + 1)))
            ens.autotune(str(path))
        torch.view_as_real(ens.psi).normal_(1.0, 0.3, generator=gen)
        series = ens.advance(4, 2)
        ens.step(1)
        m = ens.moments(0)
        got.append([torch.view_as_real(ens.psi).clone(), series, m["nk_mean"], m["nk_var"], m["rho_mean"]])
        ens.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)

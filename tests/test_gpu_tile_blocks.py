"""The tile paint's block sizes on both sides of their rules (particles per tile, interlacing, mesh), and the z pass
without the table where a block's rows are shorter or longer than its threads.

P_0 of the exactly painted FP32 meshes against FP64 meshes: FP32 values and transforms, 1e-6 of |P_0| + S/I. FP32 against
FP64 weights: 1e-5, the bound of the FP32 path."""
import numpy as np
import pytest

import synth
from oracle import estimator as E
from tests._parity import run_gpu

pytestmark = pytest.mark.gpu

L, CORNER = 900.0, (300.0, 350.0, 320.0)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _params(nmesh, window, interlaced, n):
    return E.Params(nmesh=nmesh, box_size=L, box_corner=CORNER, window=window, interlaced=interlaced, compensate=True,
                    P0=1e4, nbar=n / L ** 3)


# 128^3 has 512 tiles, 192^3 1728, 256^3 4096
@pytest.mark.parametrize("nmesh,n", [(128, 63 * 512), (128, 65 * 512), (192, 511 * 1728), (192, 513 * 1728), (256, 3000),
                                     (256, 513 * 4096)])
@pytest.mark.parametrize("window,interlaced", [("cic", False), ("tsc", False), ("tsc", True)])
def test_tile_blocks(nmesh, n, window, interlaced):
    d, r = synth.uniform_box(n // 6, L, CORNER, 3), synth.uniform_box(n - n // 6, L, CORNER, 4)
    d.pos[: n // 60] = d.pos[0]  # one crowded tile
    p, edges = _params(nmesh, window, interlaced, d.size), np.linspace(0.0, np.pi * nmesh / L, 9)
    g, f = (run_gpu(p, d, r, [0], edges, precision=prec) for prec in ("fp32", "fp64"))
    scale = np.abs(f["P"][0]) + f["stats"]["S"] / f["stats"]["I"]
    assert np.max(np.abs(g["P"] - f["P"]) / scale) < 1e-6


@pytest.mark.parametrize("nmesh", [16, 48, 64, 96, 192, 256, 384])
@pytest.mark.parametrize("precision", ["fp32", "fp32_plain"])
def test_weights_without_the_table(nmesh, precision):
    d, r = synth.uniform_box(3000, L, CORNER, 7), synth.uniform_box(9000, L, CORNER, 8)
    p, edges = _params(nmesh, "cic", True, 3000), np.linspace(0.0, np.pi * nmesh / L, 6)
    ells = [0, 1, 2, 4, 7] if nmesh < 192 else [0, 1, 2]
    f = run_gpu(p, d, r, ells, edges, precision="fp64")
    scale = np.abs(f["P"][0]) + f["stats"]["S"] / f["stats"]["I"]
    g = run_gpu(p, d, r, ells, edges, precision=precision, ylm_table=False)
    assert np.max(np.abs(g["P"] - f["P"]) / scale) < 1e-5

"""FP64 contexts (transforms in fixed point) against the FP64 oracle at every kind of row and
column plan, and over the range of magnitudes a scale is chosen for.

Tolerance: each pass is within ~1e-15 of its largest values and the estimator adds up the modes of a
bin, so 1e-12 of |P_0| + S/I leaves two orders of magnitude."""
import numpy as np
import pytest

import synth
from oracle import estimator as E
from tests._parity import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _case(nmesh, window, interlaced, scale=1.0):
    L, corner = 900.0, (300.0, 350.0, 320.0)
    d, r = synth.uniform_box(3000, L, corner, 7), synth.uniform_box(9000, L, corner, 8)
    rng = np.random.default_rng(9)
    d.weight, r.weight = (0.5 + rng.random(3000)) * scale, (0.5 + rng.random(9000)) * scale
    p = E.Params(nmesh=nmesh, box_size=L, box_corner=corner, window=window, interlaced=interlaced,
                 compensate=True, P0=1e4, nbar=3000 / L ** 3)
    return d, r, p, np.linspace(0.0, np.pi * nmesh / L, 7)


@pytest.mark.parametrize("nmesh,window,interlaced", [(16, "cic", True), (32, "tsc", True), (48, "cic", False),
                                                     (96, "tsc", True), (128, "cic", True), (192, "cic", False),
                                                     (256, "tsc", False)])
def test_fp64_transforms_match_oracle(nmesh, window, interlaced):
    d, r, p, edges = _case(nmesh, window, interlaced)
    ells = [0, 1, 2, 4] if nmesh < 192 else [0, 2]
    g = run_gpu(p, d, r, ells, edges, precision="fp64")
    o = E.multipoles(d, r, p, ells, edges)
    scale = np.abs(o["P"][0]) + o["S"] / o["I"]
    assert np.max(np.abs(g["P"] - o["P"]) / scale) < 1e-12
    np.testing.assert_array_equal(g["n_modes"], o["n_modes"])


@pytest.mark.parametrize("k", [-300, -110, -40, 40, 110, 300])
def test_powers_of_two_scale_exactly(k):
    """P is homogeneous of degree one in the completeness weights, whatever their size."""
    d, r, p, edges = _case(32, "cic", True)
    one = run_gpu(p, d, r, [0, 2], edges, precision="fp64")
    d2, r2, _, _ = _case(32, "cic", True, scale=2.0 ** k)
    got = run_gpu(p, d2, r2, [0, 2], edges, precision="fp64")
    scale = np.abs(one["P"][0]) + one["stats"]["S"] / one["stats"]["I"]
    assert np.max(np.abs(got["P"] * 2.0 ** -k - one["P"]) / scale) < 1e-12


def test_rows_of_two_warps():
    """1024^3 rows span two warps: FP64 against the FP32 transforms (their accuracy, 1e-5)."""
    d, r, p, edges = _case(1024, "cic", False)
    ells = [0, 2]
    g = run_gpu(p, d, r, ells, edges, precision="fp64", max_group_bytes=1)
    f = run_gpu(p, d, r, ells, edges, precision="fp32", max_group_bytes=1, ylm_table=False)
    scale = np.abs(g["P"][0]) + g["stats"]["S"] / g["stats"]["I"]
    assert np.max(np.abs(g["P"] - f["P"]) / scale) < 1e-5

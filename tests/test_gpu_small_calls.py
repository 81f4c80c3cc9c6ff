"""The launch graph behind repeated pspec_multipoles calls, and the tile paint on both sides of its rules on
the number of tiles (1024 or 512 threads a tile at 216 tiles, records counted and placed in shared memory up
to 4096)."""
import numpy as np
import pytest

import synth
from oracle import estimator as E
from tests._parity import gpu_estimator, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _params(nmesh, window="tsc"):
    L, corner = 900.0, (300.0, 350.0, 320.0)
    return L, corner, E.Params(nmesh=nmesh, box_size=L, box_corner=corner, window=window, interlaced=True,
                               compensate=True, P0=1e4, nbar=3000 / L ** 3)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_repeated_calls_give_what_the_first_call_gives(precision):
    """Calls past the second replay a graph: new catalogs, other bins, multipoles and tuning in between."""
    L, corner, p = _params(32)
    cats = [(synth.uniform_box(3000 + 500 * i, L, corner, 7 + i), synth.uniform_box(9000, L, corner, 8 + i)) for i in range(3)]
    e1, e2 = np.linspace(0.0, np.pi * 32 / L, 7), np.linspace(0.01, 0.08, 5)
    want = {}
    for i, (d, r) in enumerate(cats):
        for key, ells, edges in (("a", [0, 2, 4], e1), ("b", [0, 2], e2)):
            want[i, key] = run_gpu(p, d, r, ells, edges, precision=precision, ell_max=4)
    est = gpu_estimator(p, precision=precision, ell_max=4, max_particles=0 if precision == "fp64" else 20000)
    tol = 1e-12 if precision == "fp64" else 1e-13  # FP64 sums in another order only

    def check(i, key, ells, edges):
        est.paint(cats[i][0].pos, cats[i][1].pos)
        got, w = est.multipoles(ells, edges), want[i, key]
        scale = np.abs(w["P"][0]) + w["stats"]["S"] / w["stats"]["I"]
        assert np.max(np.abs(got["P"] - w["P"]) / scale) < tol, (i, key)
        np.testing.assert_array_equal(got["n_modes"], w["n_modes"])
        np.testing.assert_allclose(got["k_mean"], w["k_mean"], rtol=1e-14)
        return est.plan_info()

    first = check(0, "a", [0, 2, 4], e1)
    for i in (1, 2, 0, 1):
        info = check(i, "a", [0, 2, 4], e1)
    assert info["transforms_executed"] == first["transforms_executed"]
    for i in (2, 1, 0, 2):
        check(i, "b", [0, 2], e2)
    est.set_tuning(tile_y=1)
    for i in (0, 1, 2, 1):
        check(i, "b", [0, 2], e2)
    check(0, "a", [0, 2, 4], e1)
    est.set_profiling(True)
    check(1, "a", [0, 2, 4], e1)
    est.set_profiling(False)
    est.close()


@pytest.mark.parametrize("nmesh,window", [(96, "cic"), (96, "tsc"), (128, "tsc"), (256, "cic"), (256, "tsc"), (384, "tsc")])
def test_tile_paint_on_both_sides_of_its_rules(nmesh, window):
    """P_0 of the exactly painted FP32 meshes against the FP64 meshes: FP32 values and transforms, 1e-6."""
    L, corner, p = _params(nmesh, window)
    d, r = synth.uniform_box(20001, L, corner, 3), synth.uniform_box(60003, L, corner, 4)
    d.pos[:500] = d.pos[0]                       # one crowded tile
    r.pos[:7] += np.array([L, 0.0, -L])          # wrapped particles
    edges = np.linspace(0.0, np.pi * nmesh / L, 9)
    g = run_gpu(p, d, r, [0], edges, precision="fp32")
    f = run_gpu(p, d, r, [0], edges, precision="fp64")
    scale = np.abs(f["P"][0]) + f["stats"]["S"] / f["stats"]["I"]
    assert np.max(np.abs(g["P"] - f["P"]) / scale) < 1e-6
    assert g["stats"]["n_wrapped"] == f["stats"]["n_wrapped"] == 7

"""Mesh sides and multipoles at which the transform and binning passes take another shape.

768: FP32 blocks of four columns in storage tiles of eight (with and without the tables, both tile_y). FP64 in
fixed point: the largest radix-3 and radix-2 meshes of a kind; l = 9, 10 (polynomial weights), 12, 16 (the
recurrence on unit vectors). FP32 against FP64 of the same call: 1e-5 (exact-add) of |P_0| + S/I, the bound of the
survey tests; plain transforms 2e-5, twice that. FP64 against the oracle: 1e-12 as in the FP64 parity tests, l = 12
and 16 too (their weights' rounding stays below 1e-14)."""
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


def _case(nmesh, window="cic", interlaced=True, n=3000):
    L, corner = 900.0, (300.0, 350.0, 320.0)
    d, r = synth.uniform_box(n, L, corner, 7), synth.uniform_box(3 * n, L, corner, 8)
    p = E.Params(nmesh=nmesh, box_size=L, box_corner=corner, window=window, interlaced=interlaced, compensate=True,
                 P0=1e4, nbar=n / L ** 3)
    return d, r, p, np.linspace(0.0, np.pi * nmesh / L, 7)


def _off(got, want):
    scale = np.abs(want["P"][0]) + want["stats"]["S"] / want["stats"]["I"]
    np.testing.assert_array_equal(got["n_modes"], want["n_modes"])
    return np.max(np.abs(got["P"] - want["P"]) / scale)


def test_768():
    d, r, p, edges = _case(768, n=20000)
    # edges that leave out columns: storage tiles of which one block is past the last bin, and whole tiles
    short = edges[:-2] * 0.9
    ells = [0, 1, 2]
    ref = {k: run_gpu(p, d, r, ells, e, precision="fp64", max_group_bytes=1) for k, e in (("all", edges), ("short", short))}
    for precision, tol in (("fp32", 1e-5), ("fp32_plain", 2e-5)):
        for table in (True, False):
            est = gpu_estimator(p, precision=precision, ell_max=2, max_particles=80000, ylm_table=table,
                                max_group_bytes=0 if table else 1)
            est.paint(d.pos, r.pos)
            for tile_y in (0, 1):
                est.set_tuning(tile_y=tile_y)
                for k, e in (("all", edges), ("short", short)):
                    assert _off(est.multipoles(ells, e), ref[k]) < tol, (precision, table, tile_y, k)
            est.close()


@pytest.mark.parametrize("nmesh", [384, 512])
def test_large_fp64_meshes(nmesh):
    """FP64 against the exact-add FP32 transforms of the same meshes' size, odd l included."""
    d, r, p, edges = _case(nmesh, window="tsc", n=20000)
    ells = [0, 1, 2, 4]
    g = run_gpu(p, d, r, ells, edges, precision="fp64")
    assert _off(run_gpu(p, d, r, ells, edges, precision="fp32"), g) < 1e-5


@pytest.mark.parametrize("nmesh", [32, 48])
@pytest.mark.parametrize("ells", [[0, 3, 5, 7, 8, 9], [0, 6, 10, 11, 12, 16]])
def test_fp64_high_multipoles(nmesh, ells):
    d, r, p, edges = _case(nmesh)
    g = run_gpu(p, d, r, ells, edges, precision="fp64")
    o = E.multipoles(d, r, p, ells, edges)
    scale = np.abs(o["P"][0]) + o["S"] / o["I"]
    assert np.max(np.abs(g["P"] - o["P"]) / scale) < 1e-12
    # harmonics in groups of five: a group's first harmonic is not the multipole's
    few = run_gpu(p, d, r, ells, edges, precision="fp64", max_group_bytes=5 * nmesh ** 3 * 8)
    assert few["plan"]["group_max"] == 5
    assert np.max(np.abs(few["P"] - g["P"]) / scale) < 1e-13

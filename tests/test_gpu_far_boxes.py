"""Boxes in other length units and observers next to a mesh node: FP64 contexts weight with r^l Y_lm / r^l,
and neither factor may leave FP64's range while Y_lm of the unit vector is an ordinary number.

P is homogeneous of degree three in the length unit (with n̄ L^3 and n̄ P0 kept); a unit that is a power of
two changes no mantissa, so 1e-12 of |P_0| + S/I, the bound of the FP64 parity tests, leaves orders of magnitude."""
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


def _call(unit=1.0, observer=(0.0, 0.0, 0.0), corner=(300.0, 350.0, 320.0), nmesh=32):
    L = 900.0
    d, r = synth.uniform_box(3000, L, corner, 7), synth.uniform_box(9000, L, corner, 8)
    p = E.Params(nmesh=nmesh, box_size=L * unit, box_corner=tuple(c * unit for c in corner),
                 observer=tuple(o * unit for o in observer), window="cic", interlaced=True, compensate=True,
                 P0=1e4 * unit ** 3, nbar=3000 / L ** 3 * unit ** -3)
    d.pos, r.pos = d.pos * unit, r.pos * unit
    return d, r, p, np.linspace(0.0, np.pi * nmesh / L, 7) / unit


@pytest.mark.parametrize("k", [-240, -112, 112, 240])
def test_length_units(k):
    ells = [0, 1, 2, 4, 9, 10, 12]
    res = []
    for unit in (1.0, 2.0 ** k):
        d, r, p, edges = _call(unit)
        res.append(run_gpu(p, d, r, ells, edges, precision="fp64"))
    one, got = res
    scale = np.abs(one["P"][0]) + one["stats"]["S"] / one["stats"]["I"]
    assert np.max(np.abs(got["P"] * 2.0 ** (-3 * k) - one["P"]) / scale) < 1e-12


@pytest.mark.parametrize("off", [0.0, 1e-40, 1e-27])
def test_observer_next_to_a_node(off):
    """The weights of one node change direction with the offset; against the oracle, on unit vectors."""
    ells = [0, 1, 2, 10]
    corner = (0.0, 0.0, 0.0)
    d, r, p, edges = _call(observer=(off, -off, 2 * off), corner=corner)
    g = run_gpu(p, d, r, ells, edges, precision="fp64")
    o = E.multipoles(d, r, p, ells, edges)
    scale = np.abs(o["P"][0]) + o["S"] / o["I"]
    assert np.max(np.abs(g["P"] - o["P"]) / scale) < 1e-12

"""Which pspec_multipoles calls replay the captured launches, and that a replay finds its bin tables, tile list and
meshes whatever other entry points of the context ran in between."""
import numpy as np
import pytest

import synth
from oracle import estimator as E
from tests._parity import gpu_estimator, run_gpu

pytestmark = pytest.mark.gpu

N, L, CORNER = 32, 900.0, (300.0, 350.0, 320.0)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _params():
    return E.Params(nmesh=N, box_size=L, box_corner=CORNER, window="tsc", interlaced=True, compensate=True, P0=1e4,
                    nbar=3000 / L ** 3)


def _cats(i):
    return synth.uniform_box(3000 + 500 * i, L, CORNER, 7 + i), synth.uniform_box(9000, L, CORNER, 8 + i)


E1, E2 = np.linspace(0.0, np.pi * N / L, 7), np.linspace(0.01, 0.06, 12)


def _close(got, want, scale):
    assert np.max(np.abs(got["P"] - want["P"]) / scale) < 1e-13  # FP64 sums in another order only
    np.testing.assert_array_equal(got["n_modes"], want["n_modes"])


def test_replays_between_other_calls():
    import torch
    want = {}
    for i in (0, 1):
        w = run_gpu(_params(), *_cats(i), [0, 2, 4], E1)
        want[i] = w, np.abs(w["P"][0]) + w["stats"]["S"] / w["stats"]["I"]
    est = gpu_estimator(_params(), max_particles=20000, cache_randoms=True, cartesian=True)
    est.set_randoms(_cats(0)[1].pos)
    out = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (2 * 11, 11, 11)]

    def call(i, replays):
        est.paint(_cats(i)[0].pos, _cats(i)[1].pos)
        _close(est.multipoles([0, 2, 4], E1), *want[i])
        assert est.multipoles_replays() == replays

    for n, i in enumerate((0, 1, 0, 1, 0)):
        call(i, max(0, n - 1))  # replayed from the third call on
    others = [lambda: est.multipoles_device([0, 2], E2, *out),
              lambda: est.multipoles_range([0, 4], E2, 0, 5),
              lambda: est.multipoles_cartesian([0, 2, 4], E2),
              lambda: est.run_batch([(_cats(1)[0].pos,)], [0, 2], E2),
              lambda: est.run_batch([(_cats(1)[0].pos,)], [0, 2, 4], E1[:4])]
    for n, f in enumerate(others):
        f()
        call(n % 2, 4 + n)
    est.set_profiling(True)
    call(1, 8)  # profiled calls are launched one by one
    est.set_profiling(False)
    call(0, 9)
    est.set_tuning(bin_blocks_per_sm=1)
    for n in range(4):
        call(n % 2, 9 + max(0, n - 1))
    est.close()


def test_arguments_that_change_every_third_call():
    """A graph that was not replayed a second time is not worth its capture: the next ones wait longer."""
    est = gpu_estimator(_params(), max_particles=20000)
    est.paint(_cats(0)[0].pos, _cats(0)[1].pos)
    for _ in range(3):
        for edges in (E1, E2):
            for _ in range(3):
                est.multipoles([0, 2], edges)
    assert est.multipoles_replays() == 1
    for _ in range(8):  # a caller that stays with its arguments gets one again
        est.multipoles([0, 2], E1)
    assert est.multipoles_replays() == 1 + 8 - 4
    est.close()

"""Contexts next to each other, and the knobs of one context."""
import threading

import numpy as np
import pytest

import synth
from oracle import estimator as E
from tests._parity import gpu_estimator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def test_contexts_of_two_threads_with_other_bins():
    """Distinct contexts are independent: the binning kernels of one take 70 KB of shared memory a block, of the
    other 52 KB, and neither may take the other's allowance away between its own and its launch."""
    import torch
    res = {}

    def work(nk):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                g = torch.Generator(device="cuda").manual_seed(3)
                d, r = (torch.rand(n, 3, device="cuda", dtype=torch.float64, generator=g) * 900.0 for n in (2000, 6000))
                est = gpu_estimator(E.Params(nmesh=128, box_size=900.0, box_corner=(0.0, 0.0, 0.0), window="cic",
                                             interlaced=False, compensate=False, P0=1e4, nbar=1e-4), ell_max=2, stream=stream)
                est.paint(d, r)
                out = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (2 * nk, nk, nk)]
                edges = np.linspace(0.0, np.pi * 128 / 900.0, nk + 1)
                for _ in range(1500):
                    est.multipoles_device([0, 2], edges, *out)
                stream.synchronize()
                est.close()
            res[nk] = "ok"
        except Exception as e:  # reported below, in the test's thread
            res[nk] = repr(e)

    threads = [threading.Thread(target=work, args=(nk,)) for nk in (512, 64)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert res == {512: "ok", 64: "ok"}


@pytest.mark.parametrize("ylm_table", [True, False])
@pytest.mark.parametrize("knob", [1, 3, 9, 16, 17])
def test_ylm_harmonics_is_the_most_a_block_takes(knob, ylm_table):
    """17 harmonics of l = 8 in ceil(17 / knob) launches of the Y-weighted z pass."""
    L, corner = 900.0, (300.0, 350.0, 320.0)
    d, r = synth.uniform_box(3000, L, corner, 7), synth.uniform_box(9000, L, corner, 8)
    p = E.Params(nmesh=32, box_size=L, box_corner=corner, window="cic", interlaced=False, compensate=True, P0=1e4,
                 nbar=3000 / L ** 3)
    est = gpu_estimator(p, precision="fp32_plain", ell_max=8, ylm_table=ylm_table, max_particles=12000)
    assert est.tuning()["ylm_harmonics"] == 64
    edges = np.linspace(0.0, np.pi * 32 / L, 7)
    est.paint(d.pos, r.pos)
    want = est.multipoles([0, 8], edges)
    est.set_tuning(ylm_harmonics=knob)
    est.set_profiling(True)
    est.kernel_times()
    got = est.multipoles([0, 8], edges)
    launches = est.kernel_times()["ylm_r2c_z"]["launches"]
    assert launches == -(-17 // knob)
    np.testing.assert_allclose(got["P"], want["P"], rtol=0, atol=1e-9 * np.abs(want["P"]).max())
    est.close()


@pytest.mark.parametrize("nmesh,table,launches", [(32, True, 1), (32, False, 1), (256, True, 1), (384, True, 3)])
def test_groups_of_harmonics_by_mesh(nmesh, table, launches):
    """The default: the 17 harmonics of l = 8 in one launch on small meshes, in groups of eight at most from 384 on."""
    L, corner = 900.0, (300.0, 350.0, 320.0)
    d, r = synth.uniform_box(3000, L, corner, 7), synth.uniform_box(9000, L, corner, 8)
    p = E.Params(nmesh=nmesh, box_size=L, box_corner=corner, window="cic", interlaced=False, compensate=True, P0=1e4,
                 nbar=3000 / L ** 3)
    est = gpu_estimator(p, precision="fp32_plain", ell_max=8, ylm_table=table, max_particles=12000)
    est.paint(d.pos, r.pos)
    est.set_profiling(True)
    est.multipoles([0, 8], np.linspace(0.0, np.pi * nmesh / L, 7))
    assert est.kernel_times()["ylm_r2c_z"]["launches"] == launches
    est.close()

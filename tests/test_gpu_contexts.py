"""Contexts next to each other."""
import threading

import numpy as np
import pytest

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

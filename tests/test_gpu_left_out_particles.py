"""Which particles the catalog sums leave out: positions more than 2^38 cells from the corner or not finite,
whatever shortcut decides it (a corner far away, a corner or a default n̄ that is not a number)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, L = 32, 1000.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _sums(corner, dtype, nbar=3e-4, weights=False):
    """W_d and W_r of 300 data and 900 randoms in the box, 7 and 11 of them at the origin instead."""
    import torch
    from paper_1704_02357_gb300 import pspec
    par = pspec.Params(N, 2, 1, 1, 0, 4, L, (pspec.C.c_double * 3)(*corner), (pspec.C.c_double * 3)(0, 0, 0), 1e4, nbar)
    g = np.random.default_rng(3)
    base = np.where(np.isfinite(corner), corner, 0.0)
    cats = []
    for n, away in ((300, 7), (900, 11)):
        pos = base + g.random((n, 3)) * L
        pos[::n // away][:away] = 0.0
        cats.append(torch.as_tensor(pos, device="cuda").to(dtype).contiguous())
    w = [torch.ones(c.shape[0], dtype=torch.float64, device="cuda") for c in cats] if weights else [None, None]
    out = torch.zeros(10, dtype=torch.float64, device="cuda")
    pspec.catalog_sums_noalloc(par, cats[0], cats[1], out, data_weight=w[0], randoms_weight=w[1])
    torch.cuda.synchronize()
    return out[0].item(), out[1].item()


@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("pos", ["float64", "float32"])
def test_far_corner(pos, weights):
    """2e13 is 2^39 cells from the origin: the positions in the box count, those at the origin don't."""
    import torch
    assert _sums((2e13,) * 3, getattr(torch, pos), weights=weights) == (293.0, 889.0)
    assert _sums((500.0, 400.0, 300.0), getattr(torch, pos), weights=weights) == (300.0, 900.0)


@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("corner", [(float("nan"), 0.0, 0.0), (0.0, float("inf"), 0.0)])
def test_corner_that_is_not_a_number(corner, weights):
    import torch
    assert _sums(corner, torch.float64, weights=weights) == (0.0, 0.0)


def test_default_density_that_is_not_a_number():
    import torch
    assert _sums((500.0, 400.0, 300.0), torch.float64, nbar=float("nan")) == (0.0, 0.0)

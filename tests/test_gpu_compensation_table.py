"""The window compensation of FP64 contexts against extended precision, mode sums of a field that the
transforms give exactly.

One data and one randoms particle of weight one on nodes 0 and N/2 of the x axis: |F|^2 is 4 for odd n_x and 0 for even
ones, so B_0 of a bin is a sum of 4 mult / W^2 and the only systematic rounding left is that of 1/W. A bin holds one
|n|^2, a few dozen modes: some roundings of 1.1e-16 at most each way leave it off by about 1.5e-16, and the mean signed
error of the 125 bins with |n|^2 <= 200 by about 0.15e-16. Bound: 0.5e-16; an axis table rounded to FP64 alone puts the mean at
-1.5e-16 and 0.9e-16 (evaluated with numpy for the two forms below). CIC: the transform of a TSC particle, (3 + cos) / 4 per axis,
is itself rounded once for all modes of a plane."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, L, TOP = 48, 48.0, 200


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _axis(form):
    f = np.longdouble
    n = np.arange(-N // 2, N // 2)
    x = np.arccos(f(-1)) * n.astype(f) / f(N)
    if form == "jing":
        s2 = np.sin(x) ** 2
        return np.sqrt(1 - f(2) / 3 * s2)
    w = np.where(n == 0, f(1), np.sin(x) / np.where(n == 0, f(1), x))
    return w ** 2


@pytest.mark.parametrize("form", ["sinc", "jing"])
def test_mean_of_the_compensated_power(form):
    from paper_1704_02357_gb300 import Estimator
    est = Estimator(nmesh=N, box_size=L, box_corner=(0.0, 0.0, 0.0), observer=(-1e3, 0.0, 0.0), window="cic",
                    interlaced=False, compensate=form, precision="fp64", ell_max=0, P0=0.0, nbar=1.0)
    st = est.paint(np.array([[0.0, 0.0, 0.0]]), np.array([[24.0, 0.0, 0.0]]))
    assert (st["alpha"], st["I"], st["S"]) == (1.0, 1.0, 2.0)
    got = est.multipoles([0], 2 * np.pi / L * np.sqrt(np.arange(TOP + 1) + 0.5))  # bin b: |n|^2 = b + 1
    est.close()
    n = np.arange(-N // 2, N // 2)
    a = (1 / _axis(form)) ** 2
    nx, ny, nz = np.meshgrid(n, n, n, indexing="ij")
    p = np.where(nx % 2 == 0, np.longdouble(0), 4 * a[:, None, None] * a[None, :, None] * a[None, None, :])
    n2 = nx ** 2 + ny ** 2 + nz ** 2
    off = []
    for b in range(1, TOP + 1):
        m = n2 == b
        if not p[m].any():
            continue
        want = p[m].sum() / m.sum()
        off.append(float((np.longdouble(got["P"][0, b - 1]) + 2 - want) / want))
    assert len(off) == 125
    assert np.max(np.abs(off)) < 2e-15
    assert abs(np.mean(off)) < 0.5e-16, (form, np.mean(off), np.std(off))

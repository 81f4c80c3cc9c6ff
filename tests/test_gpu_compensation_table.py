"""The window compensation of FP64 contexts against extended precision, mode sums of a field that the
transforms give exactly.

One data and one randoms particle of weight one on nodes 0 and N/2 of the x axis: |F|^2 is 4 for odd n_x and 0 for even
ones, so B_0 of a bin is a sum of 4 mult / W^2 and the only systematic rounding left is that of 1/W. Each bin is
rounded a few times in FP64 (at most 2.2e-16 each, either way); the mean signed error of 16 bins is then below
1e-16, where an axis table rounded to FP64 alone puts it at 1.0e-16 to 2.0e-16."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, L = 48, 48.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02357_gb300 import build
    build.build()


def _axis(window, form):
    f = np.longdouble
    n = np.arange(-N // 2, N // 2)
    x = np.arccos(f(-1)) * n.astype(f) / f(N)
    if form == "jing":
        s2 = np.sin(x) ** 2
        return np.sqrt(1 - f(2) / 3 * s2 if window == "cic" else 1 - s2 + f(2) / 15 * s2 * s2)
    w = np.where(n == 0, f(1), np.sin(x) / np.where(n == 0, f(1), x))
    return w ** (2 if window == "cic" else 3)


@pytest.mark.parametrize("window", ["cic", "tsc"])
@pytest.mark.parametrize("form", ["sinc", "jing"])
def test_mean_of_the_compensated_power(window, form):
    from paper_1704_02357_gb300 import Estimator
    est = Estimator(nmesh=N, box_size=L, box_corner=(0.0, 0.0, 0.0), observer=(-1e3, 0.0, 0.0), window=window,
                    interlaced=False, compensate=form, precision="fp64", ell_max=0, P0=0.0, nbar=1.0)
    st = est.paint(np.array([[0.0, 0.0, 0.0]]), np.array([[24.0, 0.0, 0.0]]))
    assert (st["alpha"], st["I"], st["S"]) == (1.0, 1.0, 2.0)
    edges = np.linspace(0.0, np.pi, 17)
    got = est.multipoles([0], edges)
    est.close()
    # TSC of a particle on a node: weights 1/8, 3/4, 1/8 along each axis
    n = np.arange(-N // 2, N // 2)
    w = _axis(window, form)
    ph = np.arccos(np.longdouble(-1)) * 2 * n.astype(np.longdouble) / N
    t = np.ones(N, np.longdouble) if window == "cic" else (3 + np.cos(ph)) / 4
    a = (t / w) ** 2
    nx, ny, nz = np.meshgrid(n, n, n, indexing="ij")
    p = np.where(nx % 2 == 0, np.longdouble(0), 4 * a[:, None, None] * a[None, :, None] * a[None, None, :])
    n2 = nx ** 2 + ny ** 2 + nz ** 2
    b = np.searchsorted((edges * L / (2 * np.pi)) ** 2, n2.astype(float), side="right") - 1
    ok = (n2 > 0) & (nx > -N // 2) & (ny > -N // 2) & (nz > -N // 2) & (b < 16)
    want = np.array([p[ok & (b == i)].sum() / (ok & (b == i)).sum() for i in range(16)])
    off = ((got["P"][0].astype(np.longdouble) + 2 - want) / want).astype(float)
    assert np.max(np.abs(off)) < 4e-15
    assert abs(off.mean()) < 1e-16, off

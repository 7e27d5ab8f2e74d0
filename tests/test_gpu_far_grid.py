"""Float64 kicks on grids far off centre, where 64-bit integers hold the cell
but too few bits of the fraction: the kick is the bilinear interpolation at
the two-rounding coordinate's fraction, to float64's own rounding."""
import numpy as np
import pytest

import oracle
from paper_2010_11540_gb300 import build, sc, synth
from gpu_helpers import KEYS, to_gpu, to_host

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if np.finfo(LD).nmant < 63:
        pytest.skip("no extended long double")
    build.build()
    sc.load()


@pytest.mark.parametrize("x0,y0", [(0.0, 0.0), (1000.0, 0.0), (0.0, -130.0), (-1000.0, 1000.0)])
def test_kick(x0, y0):
    n, L = 4099, 5.0
    grid = (64, 64, x0 - 0.17, x0 + 0.17, y0 - 0.19, y0 + 0.19)
    rng = np.random.default_rng(2)
    parts = {k: np.zeros(n) for k in KEYS}
    parts["x"], parts["y"] = x0 + 0.02 * rng.standard_normal(n), y0 + 0.02 * rng.standard_normal(n)
    b = synth.beam()
    g, og = sc.create_grid(*grid), oracle.Geometry(*grid)
    st = to_gpu(parts)
    sc.deposit(g, st)
    sc.solve(g)
    sc.kick_push(g, st, b, L, synth.table([synth.elem(synth.DRIFT, 0.0)]))
    got = to_host(st)
    _, Ex, Ey, _ = sc.grid_read(g)
    kl = oracle.kick_strength(b) * L
    xi, eta = (parts["x"] - og.xmin) * og.inv_hx, (parts["y"] - og.ymin) * og.inv_hy
    i, j = np.floor(xi).astype(int), np.floor(eta).astype(int)
    fx, fy = (xi - i).astype(LD), (eta - j).astype(LD)
    for k, E in (("px", Ex), ("py", Ey)):
        c = [E[j, i], E[j, i + 1], E[j + 1, i], E[j + 1, i + 1]]
        ref = kl * ((1 - fy) * ((1 - fx) * c[0] + fx * c[1]) + fy * ((1 - fx) * c[2] + fx * c[3]))
        size = abs(kl) * np.max(np.abs(c), axis=0)
        # differences along x and y (each up to twice the largest field), five fused steps, and on the
        # centred grid the fraction itself, 63 cells 2^-53 of a difference
        bound = (12 + (4 * 63 if x0 == y0 == 0.0 else 0)) * 2.0 ** -53 * size
        assert np.all(np.abs(got[k] - ref) <= bound), (k, float(np.max(np.abs(got[k] - ref) / size) * 2.0 ** 53))

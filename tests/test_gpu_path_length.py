"""sg's change over drifts and thick quadrupoles, kept in float pairs where
these are short of nothing, at states where they are: particles metres off
axis, slips of a tenth of the drift; and a beam, sg close to zero among it.
Against the maps in long double; the bound is what float64 arithmetic of the
same formulas rounds."""
import numpy as np
import pytest

from paper_2010_11540_gb300 import build, sc, synth
from gpu_helpers import KEYS, to_gpu, to_host

pytestmark = pytest.mark.gpu

LD = np.longdouble
N = 20011
ULP = LD(2.0) ** -53


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if np.finfo(LD).nmant < 63:
        pytest.skip("no extended long double")
    build.build()
    sc.load()


def bunch(seed, sizes):
    rng = np.random.default_rng(seed)
    return {k: rng.uniform(-1.0, 1.0, N) * s for k, s in zip(KEYS, sizes)}


def push(parts, b, elem, precision):
    st = to_gpu(parts)
    sc.kick_push(sc.create_grid(64, 64, -0.02, 0.02, -0.015, 0.015, precision=precision), st, b, 0.0, synth.table([elem]))
    return to_host(st)["sigma"]


@pytest.mark.parametrize("precision", ["fp64", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("sizes", [
    (10.0, 0.4, 10.0, 0.4, 10.0, 1e-3),       # metres off axis
    (1.0, 0.05, 1.0, 0.05, 10.0, 1e-3),
    (8e-3, 8e-4, 8e-3, 8e-4, 10.0, 4e-3),     # a beam
    (8e-3, 8e-4, 8e-3, 8e-4, 1e-3, 4e-3),     # ... whose sg is as small as its changes
    (8e-3, 8e-4, 8e-3, 8e-4, 1e-7, 4e-3)])
@pytest.mark.parametrize("k1", [0.14, -0.5])
def test_quadrupole(precision, sizes, k1):
    parts, b, L = bunch(7, sizes), synth.beam(), 1.0
    got = push(parts, b, synth.elem(synth.QUAD, L, k1=k1), precision)
    x, px, y, py, sg, ps = (parts[k].astype(LD) for k in KEYS)
    ig, c, a = LD(1.0 / (b["gamma0"] * b["gamma0"])), 1 - ps, abs(LD(k1))
    w, m = np.sqrt(a * c), np.sqrt(c / a)
    foc = lambda u, p: (np.cos(w * L) * u + m * np.sin(w * L) * p, np.cos(w * L) * p - np.sin(w * L) / m * u)
    dfo = lambda u, p: (np.cosh(w * L) * u + m * np.sinh(w * L) * p, np.cosh(w * L) * p + np.sinh(w * L) / m * u)
    (x1, p1), (y1, q1) = (foc(x, px), dfo(y, py)) if k1 > 0 else (dfo(x, px), foc(y, py))
    D = x1 * p1 - x * px + y1 * q1 - y * py
    ref = sg + ps * (L * ig) - (L * (c * (px * px + py * py) + LD(k1) * (x * x - y * y)) + D) / (4 * c)
    # the sum's terms; float64 rounds each some times (the entries of the two matrices and their products
    # twelve times, the sum nine times, and sg three times); a pair by 14 2^-46 of terms below 2^-9 L
    mx = np.abs(x1) + np.abs(m) * np.abs(px) * 2 + np.abs(x) * 2
    mp = np.abs(p1) + np.abs(px) * 2 + np.abs(x) * 2 / np.abs(m)
    my = np.abs(y1) + np.abs(m) * np.abs(py) * 2 + np.abs(y) * 2
    mq = np.abs(q1) + np.abs(py) * 2 + np.abs(y) * 2 / np.abs(m)
    T = np.abs(ps * L * ig) + L / 4 * (px * px + py * py) + (
        mx * mp + my * mq + np.abs(x * px) + np.abs(y * py) + L * a * (x * x + y * y)) / (4 * c)
    assert np.all(np.abs(got - ref) <= ULP * (3 * np.abs(sg) + 12 * T + 3.5 * L))


@pytest.mark.parametrize("precision", ["fp64", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("kinetic,ps,ps_width", [(3e9, 0.0, 4e-3), (4e8, 0.0, 4e-3), (4e8, -0.3, 0.1), (4e8, 0.6, 0.1), (3e9, 0.05, 0.01)])
@pytest.mark.parametrize("L,sg_size", [(1.0, 10.0), (1.0, 1e-6), (300.0, 10.0)])
def test_drift(precision, kinetic, ps, ps_width, L, sg_size):
    parts, b = bunch(8, (8e-3, 2e-3, 8e-3, 2e-3, sg_size, ps_width)), synth.beam(kinetic_ev=kinetic)
    parts["psigma"] += ps
    got = push(parts, b, synth.elem(synth.DRIFT, L), precision)
    px, py, sg, ps = (parts[k].astype(LD) for k in ("px", "py", "sigma", "psigma"))
    b2 = LD(b["beta0"] * b["beta0"])
    o2 = 1 + 2 * ps + b2 * ps * ps
    pz, opb = np.sqrt(o2 - px * px - py * py), 1 + b2 * ps
    ref = sg + L * (1 - opb / pz)
    # (1+delta)^2 - p^2 rounds four times (halved by the root; terms of up to 1 + |2 ps| over pz^2), the root
    # twice, 1 + beta0^2 ps, the products and the difference once each
    T = L * np.abs(opb / pz)
    bound = T * (2 * (1 + 2 * np.abs(ps)) / (pz * pz) + 4) + L + 2 * (np.abs(sg) + np.abs(ref))
    assert np.all(np.abs(got - ref) <= ULP * bound)

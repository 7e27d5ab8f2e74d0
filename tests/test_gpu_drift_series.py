"""The drift in float pairs (maps.cuh, map_drift) at the edges of its range:
momenta of zero, below and above the series' limit and beyond it, psigma of
zero and large, short and long drifts, alone and after a quadrupole or a
sextupole; through the float64 grid and the split-TF32 grid (both take it) and
the BF16 grid (which keeps the general form), against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2010_11540_gb300 import build, sc, synth
from gpu_helpers import KEYS, to_gpu, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    sc.load()


def edge_bunch():
    p = np.array([0.0, 1e-30, -1e-12, 2e-4, -2e-3, 0.0312, 0.03125 * np.sqrt(0.5), -0.0313, 0.2])
    q = np.array([0.0, -1e-18, 3e-4, -0.022, 0.1])
    ps = np.array([0.0, 1e-9, -1e-3, 2e-2, -0.1, 0.3])
    px, py, pz = (a.ravel() for a in np.meshgrid(p, q, ps, indexing="ij"))
    n = len(px)
    rng = np.random.default_rng(3)
    return {"x": rng.uniform(-8e-3, 8e-3, n), "px": px.copy(), "y": rng.uniform(-8e-3, 8e-3, n), "py": py.copy(),
            "sigma": rng.uniform(-10.0, 10.0, n), "psigma": pz.copy()}


@pytest.mark.parametrize("precision", ["fp64", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("elems", [
    [synth.elem(synth.DRIFT, 0.0)], [synth.elem(synth.DRIFT, 0.1)], [synth.elem(synth.DRIFT, 6.1)],
    [synth.elem(synth.DRIFT, 4.0), synth.elem(synth.QUAD, 1.0, k1=-0.14), synth.elem(synth.DRIFT, 1.0),
     synth.elem(synth.SEXT, k2l=0.1), synth.elem(synth.DRIFT, 2.0)],
    [synth.elem(synth.DRIFT, 1000.0)]])
def test_edges_match_oracle(precision, elems):
    parts, b = edge_bunch(), synth.beam()
    table = synth.table(elems)
    st = to_gpu(parts)
    g = sc.create_grid(64, 64, -0.02, 0.02, -0.015, 0.015, precision=precision)
    sc.kick_push(g, st, b, 0.0, table)
    got, ref = to_host(st), oracle.copy_state(parts)
    oracle.push(ref, table, b)
    # each side rounds some tens of times, relative to the coordinate or to the element's
    # change of it (at most length x slope, times the quadrupole's gain of about 1)
    length = float(table["length"].sum())
    for k in KEYS:
        size = np.abs(ref[k]) + np.abs(parts[k]) + length * (np.abs(parts["px"]) + np.abs(parts["py"])) + 1e-12
        if k == "sigma":  # the oracle's L (1 - .../pz) cancels: 2^-52 of L each drift
            size = size + length
        assert np.all(np.abs(got[k] - ref[k]) <= 32 * 2.0 ** -52 * size), k


@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
def test_not_finite_and_huge(precision):
    """States the float pairs cannot hold take the general form: not finite stays so, huge stays right."""
    parts, b = edge_bunch(), synth.beam()
    parts["px"][:4] = [np.nan, np.inf, 1e200, 1.5]
    parts["x"][4:7] = [np.nan, 1e60, -1e30]
    table = synth.table([synth.elem(synth.QUAD, 1.0, k1=0.14), synth.elem(synth.DRIFT, 2.0)])
    st = to_gpu(parts)
    sc.kick_push(sc.create_grid(64, 64, -0.02, 0.02, -0.015, 0.015, precision=precision), st, b, 0.0, table)
    got, ref = to_host(st), oracle.copy_state(parts)
    with np.errstate(all="ignore"):
        oracle.push(ref, table, b)
    for k in KEYS:
        fin = np.isfinite(ref[k])
        assert np.array_equal(fin, np.isfinite(got[k])), k
        assert np.allclose(got[k][fin], ref[k][fin], rtol=1e-13, atol=1e-13), k


@pytest.mark.parametrize("ps", [0.0, 2e-16, 1e-3, 0.0039, 0.00392, -0.0039, -0.00392, 0.05])
def test_inverse_delta_on_both_sides_of_its_series(ps):
    """1/(1+delta) as a series and, from |2 ps + beta0^2 ps^2| = 2^-7 on, as a root: a long drift of small slopes."""
    n, L, b = 257, 1000.0, synth.beam()
    rng = np.random.default_rng(5)
    parts = {k: rng.uniform(-1.0, 1.0, n) * s for k, s in
             zip(KEYS, (8e-3, 2e-3, 8e-3, 2e-3, 10.0, 0.0))}
    parts["psigma"] = ps * (1.0 + 1e-3 * rng.uniform(-1.0, 1.0, n))
    table = synth.table([synth.elem(synth.DRIFT, L)])
    st = to_gpu(parts)
    sc.kick_push(sc.create_grid(64, 64, -0.02, 0.02, -0.015, 0.015, precision="tf32x3"), st, b, 0.0, table)
    got, ref = to_host(st), oracle.copy_state(parts)
    oracle.push(ref, table, b)
    for k in KEYS:  # bounds as above
        size = np.abs(ref[k]) + np.abs(parts[k]) + L * (np.abs(parts["px"]) + np.abs(parts["py"])) + 1e-12
        if k == "sigma":
            size = size + L
        assert np.all(np.abs(got[k] - ref[k]) <= 32 * 2.0 ** -52 * size), k

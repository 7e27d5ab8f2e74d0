"""Where float pairs must not be taken: a psigma that is not finite, has no
(1+delta) or overflows it, in segments that hold drifts alone or beside thin
sextupoles.  Every coordinate is then finite where the oracle's is, and equal
to it: called step by step and through a tracked turn, in every field type."""
import numpy as np
import pytest

import oracle
from paper_2010_11540_gb300 import build, sc, synth
from gpu_helpers import KEYS, to_gpu, to_host

pytestmark = pytest.mark.gpu

GRID = (64, 64, -0.02, 0.02, -0.015, 0.015)
ODD = [np.nan, np.inf, -np.inf, -1.0, -0.9, -1.2, 1e200, -1e200, 1e30, 2.0, -2.5]  # (-1.2, -1, -0.9: (1+delta)^2 < 0)
SEXTS = [synth.elem(synth.DRIFT, 2.0), synth.elem(synth.SEXT, k2l=0.1), synth.elem(synth.DRIFT, 0.5)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    sc.load()


@pytest.mark.parametrize("precision", ["fp64", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("elems", [[synth.elem(synth.DRIFT, 2.0)], SEXTS])
@pytest.mark.parametrize("how", ["step", "turn"])
def test_odd_psigma_as_the_oracle(precision, elems, how):
    n, b = 257, synth.beam(n_lambda=0.0)
    rng = np.random.default_rng(17)
    parts = {k: rng.uniform(-1.0, 1.0, n) * s for k, s in zip(KEYS, (8e-3, 2e-3, 8e-3, 2e-3, 10.0, 1e-3))}
    parts["psigma"][5:5 + len(ODD)] = ODD
    st, ref = to_gpu(parts), oracle.copy_state(parts)
    g = sc.create_grid(*GRID, precision=precision)
    with np.errstate(all="ignore"):
        if how == "step":
            table = synth.table(elems)
            sc.kick_push(g, st, b, 0.0, table)
            oracle.push(ref, table, b)
        else:
            lat = synth.table([synth.elem(synth.MARK)] + elems + [synth.elem(synth.MARK)] + elems)
            sc.track_turns(g, st, b, lat, 1)
            oracle.track(oracle.Geometry(*GRID), ref, b, lat, 1)
    got = to_host(st)
    for k in KEYS:
        fin = np.isfinite(ref[k])
        assert np.array_equal(fin, np.isfinite(got[k])), (k, parts["psigma"][fin != np.isfinite(got[k])])
        # (both sides round some tens of times; the path length cancels from the drifts' 5 m)
        assert np.allclose(got[k][fin], ref[k][fin], rtol=1e-13, atol=2e-14), k

"""Exact dipoles in tracked turns: segments that hold nothing but drifts, exact
dipoles (bending and of zero angle) and thin sextupoles read the particles'
psigma too, so their dispersion and path length must be the oracle's, for one
bunch and for a batch, in every field type."""
import numpy as np
import pytest

import oracle
from paper_2010_11540_gb300 import build, sc, synth
from gpu_helpers import KEYS, rel_state_err, to_gpu, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    sc.load()


HEAD = [synth.elem(synth.EXACT_BEND, 1.2, angle=0.04)]
RING = [synth.elem(synth.MARK), synth.elem(synth.DRIFT, 1.0), synth.elem(synth.EXACT_BEND, 1.5, angle=0.1),
        synth.elem(synth.MARK), synth.elem(synth.EXACT_BEND, 2.0, angle=0.0),
        synth.elem(synth.MARK), synth.elem(synth.EXACT_BEND, 2.0, angle=-0.05), synth.elem(synth.SEXT, k2l=0.5),
        synth.elem(synth.MARK), synth.elem(synth.DRIFT, 0.7), synth.elem(synth.EXACT_BEND, 1.0, angle=0.0),
        synth.elem(synth.SEXT, k2l=-0.3)]


def check(got, ref, precision):
    if precision == "fp64":  # the bound of the other float64 turns
        err = rel_state_err(got, ref)
        assert max(err.values()) < 1e-10, err
    else:  # rms, five kicks of a field good to 1e-4 or better that each change a slope by less than its spread
        for k in KEYS:
            scale = np.sqrt(np.mean(ref[k] ** 2))
            assert np.sqrt(np.mean((got[k] - ref[k]) ** 2)) < 1e-4 * scale, k


@pytest.mark.parametrize("precision", ["fp64", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("head", [False, True])
def test_turn_matches_oracle(precision, head):
    parts, b, grid, _ = synth.workload("c1", n=5000)
    lat = synth.table((HEAD if head else []) + RING)
    st = to_gpu(parts)
    sc.track_turns(sc.create_grid(*grid, precision=precision), st, b, lat, 1)
    ref = oracle.copy_state(parts)
    oracle.track(oracle.Geometry(*grid), ref, b, lat, 1)
    check(to_host(st), ref, precision)


@pytest.mark.parametrize("precision", ["fp64", "tf32x3", "bf16x3"])
def test_batch_turn_matches_oracle(precision):
    lat = synth.table(RING)
    bunches = [synth.workload("c1", n=n)[:3] for n in (5000, 1777)]
    states = [to_gpu(p) for p, _, _ in bunches]
    batch = sc.create_batch([g for _, _, g in bunches], precision=precision)
    sc.batch_track_turns(batch, states, [b for _, b, _ in bunches], [lat] * 2, 1)
    for st, (p, b, g) in zip(states, bunches):
        ref = oracle.copy_state(p)
        oracle.track(oracle.Geometry(*g), ref, b, lat, 1)
        check(to_host(st), ref, precision)

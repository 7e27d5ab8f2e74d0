"""sc_kick_push with a kick grid and a next grid of different solve forms: the
kick reads the kick grid's fields (float32 or float64) whatever the next grid
solves with, and the fused deposit is the next grid's own."""
import numpy as np
import pytest

import oracle
from paper_2010_11540_gb300 import build, sc, synth
from gpu_helpers import KEYS, to_gpu, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kick,nxt", [("tf32x3", "fp64"), ("fp64", "tf32x3"), ("fp64", "fp64"), ("bf16x3", "tf32x3")])
def test_kick_reads_the_kick_grids_fields(kick, nxt):
    build.build()
    parts, b, grid, lat = synth.workload("c1", n=5003)
    b = dict(b, n_lambda=5e11)
    seg = synth.table([synth.elem(synth.QUAD, 0.5, k1=0.5), synth.elem(synth.DRIFT, 5.0)])
    got = []
    for with_next in (False, True):
        g, h = sc.create_grid(*grid, precision=kick), sc.create_grid(*grid, precision=nxt)
        st = to_gpu(parts)
        sc.deposit(g, st)
        sc.solve(g)
        sc.kick_push(g, st, b, 5.5, seg, next_grid=h if with_next else None)
        got.append(to_host(st))
    for k in KEYS:  # the deposit does not touch the particles
        assert np.array_equal(got[0][k], got[1][k]), k
    assert np.abs(got[1]["px"] - parts["px"]).max() > 0.0
    Q, _ = oracle.deposit(oracle.Geometry(*grid), got[1]["x"], got[1]["y"])
    assert np.array_equal(sc.grid_read(h)[0], Q)

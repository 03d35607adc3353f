"""FP64 D2Q9 flows whose departure points leave the staged halo of two nodes (|v| dt from 1 to
beyond 2, in either direction along each axis), in both work splits and all kinds of tile,
against the oracle, within the FP64 bar of the parity tests (1e-11).  (The mixed form takes
the general stream there, which other tests cover.)"""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2002_09217_gb300 import inputs

from parity_util import TOL, oracle_run, rel_linf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pond():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2002_09217_gb300 import pond as mod
    mod.load()
    return mod


def flow(nx, ny, u, v, dt, hot=1.0, bc=0, steps=3):
    w = inputs.droplet(n=nx, ny=ny, Tr=0.9, radius=max(1.5, 0.25 * min(nx, ny)), width=2.0, amp=1e-3, steps=steps)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    return dataclasses.replace(w, bc_x=bc, bc_y=bc, dt=dt, T=w.T * hot, ux=u + 0.02 * np.sin(2.1 * y) + 0.0 * x,
                               uy=v + 0.02 * np.cos(1.7 * x) + 0.0 * y)


CASES = {
    "drift_37x23": lambda: flow(37, 23, 2.6, -1.9, 0.5),
    "drift_back_40x28_walls": lambda: flow(40, 28, -2.4, 0.4, 0.5, bc=1),
    "row_129x1": lambda: flow(129, 1, 2.2, 0.0, 0.5),
    "column_1x70": lambda: flow(1, 70, 0.0, -2.2, 0.5),
    "strip_50x4": lambda: flow(50, 4, 1.3, 1.4, 0.9),
    "tall_4x50": lambda: flow(4, 50, -1.3, 1.4, 0.9, bc=1),
    "hot_bump_33x17": lambda: flow(33, 17, 0.3, -0.25, 1.0, hot=3.0, steps=2),
    "beyond_two_30x9": lambda: flow(30, 9, 4.3, -3.0, 0.5),
    "either_side_of_two_24x20": lambda: flow(24, 20, 1.7, 1.6, 1.0, steps=2),
}


# grids too large for nine lanes per node: one thread per node
LARGE = {
    "drift_97x101": lambda: flow(97, 101, 2.6, -1.9, 0.5, steps=1),
    "hot_101x97_walls": lambda: flow(101, 97, 0.3, -0.25, 1.0, hot=3.0, bc=1, steps=1),
    "column_1x9153": lambda: flow(1, 9153, 0.0, -2.2, 0.5, steps=1),
    "strip_4900x2": lambda: flow(4900, 2, 2.2, 0.4, 0.5, bc=1, steps=1),
    "strip_5000x4": lambda: flow(5000, 4, 2.2, 0.4, 0.5, steps=1),
}


def check(pond, w, **kw):
    P, st, _ = oracle_run(w)
    with pond.from_workload(w, precision="fp64", **kw) as sim:
        sim.init_fields(*w.fields())
        sim.step(w.steps)
        got, stats = sim.moments(), sim.stats()
    assert stats["nonfinite"] == 0
    err = rel_linf(got, oracle.moments(P, st))
    assert max(err.values()) <= TOL["fp64"], err


@pytest.mark.parametrize("lanes,tile_x", [(0, 0), (16, 4), (16, 16)])
@pytest.mark.parametrize("case", list(CASES))
def test_nine_lanes_match_oracle(pond, case, lanes, tile_x):
    check(pond, CASES[case](), lanes_per_node=lanes, tile_x=tile_x)


@pytest.mark.parametrize("case", list(LARGE))
def test_thread_per_node_matches_oracle(pond, case):
    check(pond, LARGE[case]())


def test_thread_per_node_tile_shapes(pond):
    check(pond, flow(97, 101, -2.6, 1.9, 0.5, steps=1), tile_x=8)
    check(pond, flow(97, 101, -2.6, 1.9, 0.5, steps=1), tile_x=2)

"""The D2Q9 and D2Q16 steps in the tiles that grids of few columns and strips take by
default, with one node more or less than the tiles hold, and FP64 grids of one thread per
node, against the oracle.  Bars as in the other parity tests: 1e-11 (FP64), 1e-5 (mixed)."""
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


def droplet(nx, ny, bc, steps=4):
    w = inputs.droplet(n=nx, ny=ny, Tr=0.85, radius=max(1.5, 0.25 * min(nx, ny)), width=2.0, amp=1e-3, steps=steps)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    return dataclasses.replace(w, bc_x=bc, bc_y=bc, ux=0.1 + 0.02 * np.sin(2.1 * y) + 0.0 * x,
                               uy=-0.07 + 0.02 * np.cos(1.7 * x) + 0.0 * y)


def check(pond, w, precision, **kw):
    P, st, _ = oracle_run(w, lattice=kw.get("lattice", "d2q9"))
    with pond.from_workload(w, precision=precision, **kw) as sim:
        sim.init_fields(*w.fields())
        sim.step(w.steps)
        got = sim.moments()
        assert sim.stats()["nonfinite"] == 0
    err = rel_linf(got, oracle.moments(P, st))
    assert max(err.values()) <= TOL[precision], err


# nine lanes (1 x 12, 2 x 6, 3 x 4 tiles); thread per node (1 x 32, 2 x 16, 4 x 16, then 128)
@pytest.mark.parametrize("nx,ny,bc", [(1, 13, 0), (2, 601, 1), (3, 401, 0), (1, 3649, 1), (2, 4097, 0), (4, 1217, 1), (4, 2433, 0), (4, 3700, 0), (4, 5001, 1)])
def test_tall_mixed(pond, nx, ny, bc):
    check(pond, droplet(nx, ny, bc), "mixed")


@pytest.mark.parametrize("nx,ny,bc,lanes", [(1, 35, 1, 0), (3, 61, 0, 8), (97, 101, 0, 8), (1, 9153, 1, 0), (4, 2433, 0, 0),
                                            (2400, 4, 1, 0), (6, 1700, 0, 0)])
def test_fp64(pond, nx, ny, bc, lanes):
    check(pond, droplet(nx, ny, bc, steps=2), "fp64", lanes_per_node=lanes)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,bc", [(1, 131, 0), (2, 65, 1), (5, 33, 0)])
def test_d2q16_tall(pond, nx, ny, bc, precision):
    check(pond, droplet(nx, ny, bc), precision, lattice="d2q16")

"""Tiles that a velocity jump of several sqrt(theta) crosses at uniform temperature (a shear
layer, colliding streams), all departure points within the staged halo, against the oracle:
the populations staged in a common gauge far from a node's own must not lose its digits
(tau = 0.6, so that the collision keeps the higher moments, which lose them first).  Bars as in the other parity tests: 1e-11 (FP64) and 1e-5 (mixed)."""
import dataclasses

import numpy as np
import pytest

import oracle
from oracle import core3d as o3
from paper_2002_09217_gb300 import inputs

from parity_util import TOL, oracle_run, rel_linf

pytestmark = pytest.mark.gpu
T0 = 0.1                        # theta = p / (rho T_L) = 0.3 (T_L = 1/3) or 0.1 (T_L = 1)


@pytest.fixture(scope="module")
def pond():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2002_09217_gb300 import pond as mod
    mod.load()
    return mod


def jump(w, kind, U, TL):
    """Ideal gas of uniform T, with a one-node ripple of rho: u_x changes by U sqrt(theta)
    from one row to the next (shear) or over a few nodes of x (colliding streams between
    zero-gradient ends); dt so that |v| dt < 1."""
    s = np.sqrt(T0 / TL)
    shape = w.rho.shape
    x, y = np.arange(shape[-1])[None, :], np.arange(shape[-2])[:, None]
    side = -np.tanh((x - shape[-1] // 2) / 2.0) if kind == "collide" else np.where(y < shape[-2] // 2 + 1, 1.0, -1.0)
    side = np.broadcast_to(side, shape[-2:])
    ux = np.broadcast_to(0.5 * U * s * side + 0.1, shape).copy()
    rho = 1.0 + 0.02 * np.sin(1.7 * np.arange(shape[-1]))[None, :] + 0.02 * np.cos(2.3 * np.arange(shape[-2]))[:, None]
    rho = np.broadcast_to(rho, shape).copy()
    zero = np.zeros(shape)
    fastest = (1.0 if TL < 1.0 else np.sqrt(3 + np.sqrt(6.0))) * s + 0.5 * U * s + 0.1
    fields = dict(rho=rho, ux=ux, uy=zero + 0.03, T=zero + T0, a=0.0, b=0.0, kappa=0.0, tau=0.6, steps=3,
                  dt=float(min(0.5, 0.8 / fastest)))
    return dataclasses.replace(w, bc_x=int(kind == "collide"), **fields)


JUMPS = [("shear", 1.0), ("shear", 2.0), ("shear", 4.0), ("shear", 6.0), ("collide", 2.0), ("collide", 3.0)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("lattice,lanes", [("d2q9", 8), ("d2q9", 16), ("d2q16", 0)])
@pytest.mark.parametrize("kind,U", JUMPS)
def test_2d_jump_matches_oracle(pond, kind, U, lattice, lanes, precision):
    w = jump(inputs.droplet(n=40, ny=21, Tr=0.9, radius=4.0, steps=1), kind, U, 1.0 if lattice == "d2q16" else 1.0 / 3.0)
    P, st, _ = oracle_run(w, lattice=lattice)
    with pond.from_workload(w, precision=precision, lattice=lattice, lanes_per_node=lanes) as sim:
        sim.init_fields(*w.fields())
        sim.step(w.steps)
        got, gstats = sim.moments(), sim.stats()
    err = rel_linf(got, oracle.moments(P, st))
    assert max(err.values()) <= TOL[precision], err
    assert gstats["nonfinite"] == 0


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind,U", JUMPS)
def test_3d_jump_matches_oracle(pond, kind, U, precision):
    w = inputs.droplet3d(n=12, ny=9, nz=6, Tr=0.9, radius=2.0, width=1.5, amp=1e-3, steps=1)
    w = dataclasses.replace(jump(w, kind, U, 1.0 / 3.0), uz=np.full(w.rho.shape, -0.02))
    P = o3.Params3(nx=w.nx, ny=w.ny, nz=w.nz, bc_x=w.bc_x, bc_y=w.bc_y, bc_z=w.bc_z, a=w.a, b=w.b, R=w.R, delta=w.delta,
                   kappa=w.kappa, tau=w.tau, k_cond=w.k_cond, p_floor=w.p_floor, tol=1e-12, max_iter=20, dt=w.dt)
    ref = o3.moments(P, o3.step(P, o3.init_state(P, *w.fields()), w.steps))
    with pond.Simulation(w.nx, w.ny, **inputs.from_workload3(w, precision)) as sim:
        sim.init_fields(w.rho, w.ux, w.uy, w.T, uz=w.uz)
        sim.step(w.steps)
        got = sim.moments()
        assert sim.stats()["nonfinite"] == 0
    err = rel_linf(got, ref)
    assert max(err.values()) <= TOL[precision], err

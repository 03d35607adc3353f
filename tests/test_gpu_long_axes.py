"""Grids long in y or z (the second and third launch dimensions hold 65,535 blocks only) step
as the same grid on its side does.  Mixed form; fields within 1e-5 of each other's maximum
(the parity bar of the mixed form)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pond():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2002_09217_gb300 import pond as mod
    mod.load()
    return mod


def run(pond, lattice, shape, axis, n):
    """One step of a wave along `axis` (0 x, 1 y, 2 z) of a grid of n nodes along it."""
    k = np.arange(n)
    rho = 1.0 + 0.05 * np.sin(0.37 * k) + 0.02 * np.cos(1.9 * k)
    u = 0.03 * np.cos(0.21 * k)
    dims = (n, 1, 1) if axis == 0 else ((1, n, 1) if axis == 1 else (1, 1, n))
    full = lambda v: v.reshape(shape(dims))
    zero = np.zeros(n)
    kw = dict(nz=dims[2]) if lattice == "d3q27" else {}
    with pond.Simulation(dims[0], dims[1], lattice=lattice, a=0.0, b=0.0, dt=0.3, **kw) as sim:
        vel = [full(u if a == axis else zero) for a in range(3)]
        if lattice == "d3q27":
            sim.init_fields(full(rho), vel[0], vel[1], full(zero + 0.1), uz=vel[2])
        else:
            sim.init_fields(full(rho), vel[0], vel[1], full(zero + 0.1))
        sim.step(2)
        m = sim.moments()
        assert sim.stats()["nonfinite"] == 0
    return m["rho"].ravel(), m[("ux", "uy", "uz")[axis]].ravel(), m["T"].ravel()


@pytest.mark.parametrize("lattice,axis,n", [("d2q9", 1, 600000), ("d2q16", 1, 600000), ("d3q27", 1, 300000), ("d3q27", 2, 300000)])
def test_long_axis_steps_as_a_row_does(pond, lattice, axis, n):
    shape = (lambda d: (d[2], d[1], d[0])) if lattice == "d3q27" else (lambda d: (d[1], d[0]))
    ref, got = run(pond, lattice, shape, 0, n), run(pond, lattice, shape, axis, n)
    for r, g in zip(ref, got):
        assert np.abs(g - r).max() <= 1e-5 * np.abs(r).max()

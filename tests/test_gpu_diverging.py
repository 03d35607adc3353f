"""A run that diverges (an isothermal contact of density ratio 100 to 1,000 with hardly any
pressure floor, far outside the scheme's stable range) reports POND_ENAN and leaves the
device usable: infinite and NaN gauges never take a stencil off the grid."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("lattice", ["d2q9", "d2q16", "d3q27"])
def test_diverging_run_reports_and_leaves_the_device_usable(pond, lattice, bc, precision):
    nx, ny, nz = (24, 8, 4) if lattice == "d3q27" else (48, 24, 1)
    shape = (nz, ny, nx) if lattice == "d3q27" else (ny, nx)
    x = np.arange(nx)
    ratio = np.where((x >= nx // 4) & (x < 3 * nx // 4), 1000.0, 1.0)
    rho = np.broadcast_to(ratio, shape) * (1.0 + 0.01 * np.sin(np.arange(ny)))[:, None]
    zero = np.zeros(shape)
    kw = dict(nz=nz if lattice == "d3q27" else 1, bc_x=bc, bc_y=bc, bc_z=bc, lattice=lattice, precision=precision,
              a=0.0, b=0.0, dt=0.5, p_floor=1e-9)
    with pond.Simulation(nx, ny, **kw) as sim:
        sim.init_fields(rho, zero + 0.02, zero, 0.3 / rho)
        with pytest.raises(pond.PondError) as err:
            sim.step(4)
            sim.moments()
        assert err.value.status == 6   # POND_ENAN
        assert sim.stats()["nonfinite"] > 0
    with pond.Simulation(nx, ny, **kw) as sim:   # the device still works
        sim.init_fields(zero + 1.0, zero, zero, zero + 0.1)
        sim.step(2)
        np.testing.assert_allclose(sim.moments()["rho"], 1.0, rtol=1e-6)

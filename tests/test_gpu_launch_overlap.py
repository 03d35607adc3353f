"""Steps that may start while the stream's previous step drains: contexts interleaved on one
stream, other work between steps, and steps captured in the caller's graph give the bits of
the same steps run alone."""
import numpy as np
import pytest

from paper_2002_09217_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pond():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2002_09217_gb300 import pond as mod
    mod.load()
    return mod


# nine lanes and one thread per node on D2Q9, and D2Q16
CASES = [("d2q9", "mixed", 96, 5), ("d2q9", "mixed", 120, 70), ("d2q9", "fp64", 64, 5), ("d2q16", "mixed", 40, 12)]


def work(nx, ny):
    return inputs.droplet(n=nx, ny=ny, Tr=0.9, radius=0.3 * ny, width=2.0, amp=1e-3, steps=12)


def alone(pond, w, lattice, precision, **kw):
    with pond.from_workload(w, precision=precision, lattice=lattice, **kw) as sim:
        sim.init_fields(*w.fields())
        sim.step(w.steps)
        return sim.get_state()


def test_contexts_interleaved_on_one_stream(pond):
    import torch
    ws = [(lat, pr, work(nx, ny)) for lat, pr, nx, ny in CASES]
    ref = [alone(pond, w, lat, pr) for lat, pr, w in ws]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        sims = [pond.from_workload(w, precision=pr, lattice=lat, stream=s) for lat, pr, w in ws]
        for sim, (_, _, w) in zip(sims, ws):
            sim.init_fields(*w.fields())
        out = [{k: torch.zeros(w.ny, w.nx, dtype=torch.float64, device="cuda") for k in ("rho", "T")} for _, _, w in ws]
        for k in range(12):
            for sim, o in zip(sims, out):
                sim.step(1)
                if k % 3 == 0:      # a kernel of another kind between the steps
                    sim.moments_device(o)
        got = [sim.get_state() for sim in sims]
        for sim in sims:
            sim.close()
    for r, g in zip(ref, got):
        np.testing.assert_array_equal(g, r)


@pytest.mark.parametrize("nonlocal_", ["lagged", "current"])
@pytest.mark.parametrize("lattice,precision,nx,ny", CASES)
def test_steps_captured_in_a_graph(pond, lattice, precision, nx, ny, nonlocal_):
    import torch
    w = work(nx, ny)
    ref = alone(pond, w, lattice, precision, nonlocal_=nonlocal_)
    s = torch.cuda.Stream()
    with pond.from_workload(w, precision=precision, lattice=lattice, nonlocal_=nonlocal_, stream=s) as sim:
        sim.init_fields(*w.fields())
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            sim.step(2)
        with torch.cuda.stream(s):
            for _ in range(w.steps // 2):
                g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(sim.get_state(), ref)

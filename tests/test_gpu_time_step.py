"""The adaptive time step, cfl h / max |u_f / phi_f|: the kernel divides only the faces that
can hold the maximum, so it must be the maximum over every face's quotient, to the last bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


def _face_porosity(phi, axis):
    pad = [(0, 0)] * 3
    pad[axis] = (1, 1)
    p = np.pad(phi, pad, mode="edge")
    n = p.shape[axis]
    return 0.5 * (np.take(p, range(n - 1), axis) + np.take(p, range(1, n), axis))


# one partial block, several, eight rows a block (large grids); one uniform speed; no flow
@pytest.mark.parametrize("kind", ["varied", "uniform", "still"])
@pytest.mark.parametrize("shape", [(5, 1, 1), (2000, 1, 1), (33, 17, 1), (19, 23, 13), (130, 70, 66)])
def test_dt_is_the_exact_maximum(shape, kind):
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    flow = 0.0 if kind == "still" else 1e-4
    case = W.darcy_domain(shape, seed=3, inlet_u=flow, cfl=0.01, dt=1e-3, dt_max=1.0, p_tol=1e-8, max_cg=200)
    if kind == "uniform":
        case.porosity[:] = 0.37
        case.permeability[:] = 1e-12
    s = mdbs.Simulation(case)
    s.step(1)
    f, dt = s.fields(), s.stats()["dt"]
    s.close()
    nx, ny, nz = shape
    phi = case.porosity.reshape(nz, ny, nx)
    top = 0.0
    for name, axis in (("ux", 2), ("uy", 1), ("uz", 0)):
        if f[name].size:
            pf = _face_porosity(phi, axis)
            top = max(top, np.max(np.abs(f[name].reshape(pf.shape)) / pf))
    expected = min((0.01 * case.h) / top if top > 0 else 1.0, 1.2 * 1e-3, 1.0)
    assert dt == expected
    assert kind == "still" or dt < 1.2e-3  # the speed decided

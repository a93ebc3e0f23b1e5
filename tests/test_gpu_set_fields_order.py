"""mdbs_set_fields reads its arrays in the order of the simulation's stream: an array that a copy
queued on that stream still has to fill is checked with the values the copy brings."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


# below and above the size up to which the range check reads the caller's array
@pytest.mark.parametrize("cells", [1, 2000, 16384, 16385])
@pytest.mark.parametrize("before,after", [(0.25, 2.0), (2.0, 0.25)])
@pytest.mark.parametrize("pinned", [True, False])
def test_saturation_filled_in_stream_order(cells, before, after, pinned):
    torch = pytest.importorskip("torch")
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    c = W.darcy_domain((cells, 1, 1), seed=2, p_tol=1e-8)
    s = mdbs.Simulation(c)
    stream = torch.cuda.Stream()
    s.set_stream(stream.cuda_stream)
    old = s.fields()["alpha"]
    alpha = torch.full((cells,), before, dtype=torch.float64)
    if pinned:
        alpha = alpha.pin_memory()
    new = torch.full((cells,), after, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(200_000_000)  # about 0.1 s ahead of the copy
        alpha.copy_(new, non_blocking=True)
    if after > 1.0:
        with pytest.raises(mdbs.MdbsError) as e:
            s.set_fields(alpha.numpy(), c.ux, c.uy, c.uz, c.p)
        assert e.value.code == mdbs.ERR_ARG
        assert np.array_equal(s.fields()["alpha"], old)
    else:
        s.set_fields(alpha.numpy(), c.ux, c.uy, c.uz, c.p)
        assert np.array_equal(s.fields()["alpha"], np.full(cells, after))
    stream.synchronize()
    s.close()


@pytest.mark.parametrize("after", [2.0, 0.25])
def test_default_stream_waits_for_a_blocking_stream(after):
    """The legacy default stream, which a simulation has by default, runs behind the work of
    other blocking streams: a copy queued there fills the array first, too."""
    torch = pytest.importorskip("torch")
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    cells = 2000
    c = W.darcy_domain((cells, 1, 1), seed=2, p_tol=1e-8)
    s = mdbs.Simulation(c)
    stream = C.c_void_p()
    rt = torch.cuda.cudart()
    alpha = torch.full((cells,), 2.25 - after, dtype=torch.float64).pin_memory()
    new = torch.full((cells,), after, dtype=torch.float64, device="cuda")
    err, handle = rt.cudaStreamCreate(C.addressof(stream)), stream.value
    assert int(err) == 0
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.ExternalStream(handle)):
        torch.cuda._sleep(200_000_000)
        alpha.copy_(new, non_blocking=True)
    if after > 1.0:
        with pytest.raises(mdbs.MdbsError):
            s.set_fields(alpha.numpy(), c.ux, c.uy, c.uz, c.p)
    else:
        s.set_fields(alpha.numpy(), c.ux, c.uy, c.uz, c.p)
        assert np.array_equal(s.fields()["alpha"], np.full(cells, after))
    torch.cuda.synchronize()
    # PyTorch notes the stream with the pinned buffer's release: the buffer goes first, and the
    # stream stays for the process
    del alpha
    s.close()

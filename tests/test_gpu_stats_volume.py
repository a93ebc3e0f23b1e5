"""mdbs_field_stats_static's liquid volume where every cell counts (finite fields), over the
sizes at which its vector loads, its unrolled passes and its grid end; and its capture."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

THREADS, BLOCKS = 512, 304
GRID = THREADS * BLOCKS * 2  # one pair of cells a thread of the whole grid


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


def _fields(cells, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(0.1, 1.0, cells), rng.uniform(-0.5, 1.5, cells), rng.standard_normal(cells)


def _upload(torch, fields, shift):
    # shift 1: the fields start 8 bytes past a 16-byte boundary (no vector loads)
    dev = [torch.zeros(f.size + 1, dtype=torch.float64, device="cuda")[shift: f.size + shift] for f in fields]
    for d, f in zip(dev, fields):
        d.copy_(torch.from_numpy(f))
    return dev


def _bound(cells, phi, alpha, volume):
    """Roundings of one term's way into the sum: its product here and there, a thread's chain
    (the cells of one thread), the two chains, 5 + 4 steps of a block's tree and of the second
    stage's each, the volume; every one at most half an ulp of the sum of magnitudes."""
    blocks = min(-(-cells // (2 * THREADS)), BLOCKS)
    chain = -(-cells // (blocks * THREADS))
    return (chain + 24) * 2.0 ** -53 * volume * float(np.sum(phi * np.abs(alpha))) * (1 + 1e-9)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("cells", [1, 2, 1023, 1024, 1025, GRID - 1, GRID, GRID + 1, 4 * GRID - 2, 4 * GRID,
                                   4 * GRID + 3, 9 * GRID + 5])
def test_volume_counts_every_cell(cells, shift):
    torch = pytest.importorskip("torch")
    from paper_2003_08374_gb300 import mdbs
    phi, alpha, p = _fields(cells, cells)
    dev = _upload(torch, (phi, alpha, p), shift)
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        mdbs.field_stats_static(cells, 1e-3, *[d.data_ptr() for d in dev], out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    got = out.cpu().numpy()
    want = 1e-3 * math.fsum(phi * alpha)
    assert abs(got[0] - want) <= _bound(cells, phi, alpha, 1e-3)
    assert got[1] == alpha.min() and got[2] == alpha.max() and got[3] == 0.0


@pytest.mark.parametrize("shift", [0, 1])
def test_one_cell_anywhere_counts_once(shift):
    """A single cell that is not zero, at the ends of the pairs, of a pass of the grid and of
    the unrolled passes: the volume is that cell's, exactly."""
    torch = pytest.importorskip("torch")
    from paper_2003_08374_gb300 import mdbs
    cells = 5 * GRID + 7
    phi, alpha, p = np.ones(cells), np.zeros(cells), np.zeros(cells)
    dev = _upload(torch, (phi, alpha, p), shift)
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    for at in (0, 1, 2, 1023, 1024, GRID // 2, GRID - 1, GRID, 2 * GRID, 4 * GRID - 1, 4 * GRID, 4 * GRID + 1,
               5 * GRID - 1, 5 * GRID, cells - 2, cells - 1):
        dev[1][at] = 0.75
        mdbs.field_stats_static(cells, 1.0, *[d.data_ptr() for d in dev], out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        dev[1][at] = 0.0
        assert out.tolist() == [0.75, 0.0, 0.75, 0.0], at


def test_captured_call_replays_on_new_values():
    torch = pytest.importorskip("torch")
    from paper_2003_08374_gb300 import mdbs
    cells = 4 * GRID + 3
    dev = _upload(torch, _fields(cells, 1), 0)
    out, direct = (torch.zeros(4, dtype=torch.float64, device="cuda") for _ in range(2))

    def call(o):
        mdbs.field_stats_static(cells, 1e-3, *[d.data_ptr() for d in dev], o.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)

    call(out)  # the scratch's address is looked up before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(out)
    for seed in (2, 3):
        for d, f in zip(dev, _fields(cells, seed)):
            d.copy_(torch.from_numpy(f))
        call(direct)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, direct)

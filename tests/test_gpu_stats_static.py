"""mdbs_field_stats_static on sizes and alignments where its vector loads, its unrolled
passes and its grid end: against NumPy on the same fields."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


# one cell; a pair; one block's pairs; the whole grid's pairs, once and four times (the unrolled
# pass), one cell more and less
GRID = 304 * 512 * 2


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("cells", [1, 2, 3, 1023, 1024, 1025, GRID - 1, GRID, GRID + 1, 4 * GRID + 3])
def test_against_numpy(cells, shift):
    torch = pytest.importorskip("torch")
    from paper_2003_08374_gb300 import mdbs
    rng = np.random.default_rng(cells)
    phi, alpha, p = rng.uniform(0.1, 1.0, cells), rng.uniform(-0.5, 1.5, cells), rng.standard_normal(cells)
    alpha[cells // 2] = -0.0
    bad = 0
    if cells > 3:
        alpha[1], p[2], p[cells - 1] = np.nan, np.inf, np.nan
        phi[1] = 0.0
        bad = 3
    host = [phi, alpha, p]
    # shift 1: the fields start 8 bytes past a 16-byte boundary (no vector loads)
    dev = [torch.zeros(cells + 1, dtype=torch.float64, device="cuda")[shift: cells + shift] for _ in host]
    for d, h in zip(dev, host):
        d.copy_(torch.from_numpy(h))
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    for _ in range(2):
        mdbs.field_stats_static(cells, 1e-3, *[d.data_ptr() for d in dev], out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy()
    fine = ~np.isnan(alpha)
    assert got[1] == alpha[fine].min() and got[2] == alpha[fine].max() and got[3] == bad
    if bad:
        assert np.isnan(got[0])  # a NaN saturation makes the volume NaN
    else:
        # a sum of n terms of one sign or the other: n roundings of the running magnitude at most
        assert abs(got[0] - 1e-3 * float(np.sum(phi * alpha))) <= 2.3e-16 * cells * 1e-3 * float(np.sum(phi * np.abs(alpha)))

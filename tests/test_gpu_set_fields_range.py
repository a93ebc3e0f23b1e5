"""The saturation range check of mdbs_set_fields runs on the host up to 16384 cells and on the
device above: both refuse the same fields, wherever the value stands, and leave the state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


@pytest.mark.parametrize("cells", [1, 16384, 16385])
def test_range_check_on_both_sides_of_the_line(cells):
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    c = W.darcy_domain((cells, 1, 1), seed=2, p_tol=1e-8)
    s = mdbs.Simulation(c)
    before = s.fields()
    for bad in (np.nan, np.inf, -1e-6, 1.0 + 1e-6):
        for at in {0, cells // 2, cells - 1}:
            alpha = np.full(cells, 0.25)
            alpha[at] = bad
            with pytest.raises(mdbs.MdbsError) as e:
                s.set_fields(alpha, c.ux, c.uy, c.uz, c.p)
            assert e.value.code == mdbs.ERR_ARG
    for k, v in s.fields().items():
        assert np.array_equal(v, before[k]), k
    for fine in (-5e-10, 0.0, 1.0, 1.0 + 5e-10):
        s.set_fields(np.full(cells, fine), c.ux, c.uy, c.uz, c.p)
        assert np.array_equal(s.fields()["alpha"], np.full(cells, fine))
    s.close()

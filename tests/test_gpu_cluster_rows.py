"""The cluster solve with two and with four cells a thread, which a batch of many small domains
takes, against the per-level launches: the same values bit for bit, twice in a row."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LAUNCHES = {"smooth_rows": 1, "tail_cells": 0, "snake": 0, "sweep_kz": 0, "tail_ctas": 1}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


# one to four CTAs a domain; levels whose colours differ in number, that leave CTA 0 or not, with
# unfilled last rows; odd and even sides, one to three axes
SHAPES = [(513, 1, 1), (1023, 1, 1), (1025, 1, 1), (2049, 1, 1), (1, 1111, 1), (31, 33, 1), (45, 45, 1), (3, 341, 1),
          (64, 63, 1), (9, 20, 11), (7, 11, 13), (20, 11, 9), (11, 9, 20), (16, 16, 16), (15, 16, 17), (5, 5, 160)]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("count", [24, 60])
@pytest.mark.parametrize("shape", SHAPES)
def test_rows_equal_launches(shape, count, precision):
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    case = W.darcy_domain(shape, seed=5, precision=precision, p_tol=1e-10, max_cg=300)
    one = mdbs.Simulation(case)
    one.set_tuning(LAUNCHES)
    one.step(2)
    want, iters = one.fields(), one.stats()["cg_iters"]
    one.close()
    for _ in range(2):
        sims = [mdbs.Simulation(case) for _ in range(count)]
        batch = mdbs.Batch(sims)
        batch.step(2)
        for s in sims:
            assert s.stats()["cg_iters"] == iters, shape
            got = s.fields()
            for k in got:
                assert np.array_equal(got[k], want[k]), (shape, k)
        batch.close()
        for s in sims:
            s.close()

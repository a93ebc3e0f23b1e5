"""The loop condition of a batch is formed by the block of its finalizer that arrives last:
members whose solves end at different iterations stop where they stop alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [2, 33])
def test_members_stop_where_they_stop_alone(count, precision):
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    # above 4096 cells: the loop's launches, not the cluster solve
    shapes = [(20, 17, 13), (130, 33, 1), (4100, 1, 1), (31, 23, 19)]
    cases = [W.darcy_domain(shapes[i % 4], seed=i, precision=precision, p_tol=1e-9, max_cg=300) for i in range(count)]
    alone = []
    for c in cases:
        s = mdbs.Simulation(c)
        per_step = []
        for _ in range(3):
            s.step(1)
            per_step.append(s.stats()["cg_iters"])
        alone.append((per_step, s.fields()))
        s.close()
    sims = [mdbs.Simulation(c) for c in cases]
    batch = mdbs.Batch(sims)
    got = [[] for _ in cases]
    for _ in range(3):
        batch.step(1)
        for i, s in enumerate(sims):
            got[i].append(s.stats()["cg_iters"])
    assert [g for g in got] == [a[0] for a in alone]
    assert len({tuple(map(tuple, g)) for g in got}) > 1  # they do end at different iterations
    for s, a in zip(sims, alone):
        f = s.fields()
        for k in f:
            assert np.array_equal(f[k], a[1][k]), (s.n, k)
    batch.close()
    for s in sims:
        s.close()

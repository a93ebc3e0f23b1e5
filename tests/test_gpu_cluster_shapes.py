"""Batches of small domains whose solves take several cluster launches (one for each size of
cluster), or clusters for some and the launches for the others: members equal themselves alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


BATCHES = {
    # one large among many small: a launch for it, one for the others
    "one_large": [(64, 64, 1)] + [(100, 1, 1)] * 160,
    # all three sizes of cluster, more of each than fit at once
    "three_sizes": [(16, 15, 17), (1500, 1, 1), (31, 30, 1)] * 60,
    # four CTAs a domain and too many waves: the launches
    "many": [(16, 16, 16)] * 120,
    # many levels: the launches for these, clusters for the short ones
    "deep": [(2, 2048, 1)] * 40 + [(50, 1, 1)] * 7,
    # tails of larger domains: clusters of four CTAs, of fewer than their rows, and too many
    "tails_at_once": [(20, 17, 13)] * 30,
    "tails_halved": [(33, 31, 17)] * 20,
    "tails_many": [(20, 17, 13), (70, 70, 1)] * 40,
    # small domains that join the launches of a larger one (FP32), and that do not
    "joined": [(16, 16, 16)] * 9 + [(20, 20, 13)],
    "beside": [(16, 16, 16)] * 9 + [(20, 20, 13)] + [(300, 1, 1)] * 3,
}


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(BATCHES))
def test_members_equal_themselves_alone(name, precision):
    from paper_2003_08374_gb300 import mdbs
    from paper_2003_08374_gb300 import workloads as W
    shapes = BATCHES[name]
    cases = [W.darcy_domain(s, seed=1 + i % 3, precision=precision, p_tol=1e-9, max_cg=300)
             for i, s in enumerate(shapes)]
    alone = {}
    for i, (s, c) in enumerate(zip(shapes, cases)):
        if (s, i % 3) not in alone:
            one = mdbs.Simulation(c)
            one.step(2)
            alone[s, i % 3] = one.fields(), one.stats()["cg_iters"]
            one.close()
    sims = [mdbs.Simulation(c) for c in cases]
    batch = mdbs.Batch(sims)
    batch.step(2)
    for i, (s, sim) in enumerate(zip(shapes, sims)):
        fields, iters = alone[s, i % 3]
        assert sim.stats()["cg_iters"] == iters, (s, i)
        got = sim.fields()
        for k in got:
            assert np.array_equal(got[k], fields[k]), (s, i, k)
    batch.close()
    for sim in sims:
        sim.close()

"""Grids solved in thread-block clusters where the device has no cluster of the planned size:
smaller ones, or the launches, take their place and give the same values bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


def _case(shape, precision, seed=11):
    from paper_2003_08374_gb300 import workloads as W
    return W.darcy_domain(shape, seed=seed, precision=precision, p_tol=1e-10, max_cg=300)


def _run(case, limit):
    from paper_2003_08374_gb300 import mdbs
    s = mdbs.Simulation(case)
    if limit is not None:
        s.cluster_limit(limit)
    s.step(2)
    out = s.fields(), s.stats()["cg_iters"]
    s.profile()
    s.step(1)
    kernels = set(s.profile_read())
    s.close()
    return out, kernels


def _same(a, b, what):
    assert a[1] == b[1], what
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), (what, k)


# one, two and sixteen CTAs planned; the last three: only the tail in a cluster
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 1, 1), (200, 1, 1), (2047, 1, 1), (64, 64, 1), (16, 15, 17), (6001, 1, 1),
                                   (33, 31, 17), (130, 97, 1)])
def test_any_limit_gives_the_same_values(shape, precision):
    case = _case(shape, precision)
    want, kernels = _run(case, None)
    small = np.prod(shape) <= 4096
    assert ("cg_cluster" in kernels) == small  # what this device plans
    for limit in (0, 1, 2, 4, 8, 16):
        got, kernels = _run(case, limit)
        _same(got, want, (shape, limit))
        assert limit > 0 or "cg_cluster" not in kernels
        assert limit < 16 or ("cg_cluster" in kernels) == small


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("limit", [0, 1, 2, 8])
def test_a_batch_takes_its_members_limit(limit, precision):
    from paper_2003_08374_gb300 import mdbs
    shapes = [(1800, 1, 1), (45, 80, 1), (9, 20, 11), (250, 1, 1), (24, 20, 22)]
    cases = [_case(s, precision, seed=i) for i, s in enumerate(shapes)]
    alone = [_run(c, None)[0] for c in cases]
    sims = [mdbs.Simulation(c) for c in cases]
    sims[1].cluster_limit(limit)
    batch = mdbs.Batch(sims)
    batch.step(2)
    for s, a in zip(sims, alone):
        f, it = s.fields(), s.stats()["cg_iters"]
        _same((f, it), a, (s.n, limit))
    batch.close()
    for s in sims:
        s.close()


def test_limit_is_refused_in_a_batch_and_below_zero():
    from paper_2003_08374_gb300 import mdbs
    s = mdbs.Simulation(_case((50, 1, 1), 0))
    with pytest.raises(mdbs.MdbsError):
        s.cluster_limit(-1)
    batch = mdbs.Batch([s])
    with pytest.raises(mdbs.MdbsError):
        s.cluster_limit(4)
    batch.close()
    s.cluster_limit(4)
    s.step(1)
    s.close()

"""Small grids solved inside a thread-block cluster (levels of at most 4096 cells; a grid
that fits wholly runs its CG solve there) against the per-level launches: the same values
bit for bit, whatever the grid's shape, the cluster's size and the V-cycle's options."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LAUNCHES = {"smooth_rows": 1, "tail_cells": 0, "snake": 0, "sweep_kz": 0, "tail_ctas": 1}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


def _case(shape, precision, **kw):
    from paper_2003_08374_gb300 import workloads as W
    return W.darcy_domain(shape, seed=11, precision=precision, **{"p_tol": 1e-10, "max_cg": 60, **kw})


def _run(case, schedule, steps=2):
    from paper_2003_08374_gb300 import mdbs
    s = mdbs.Simulation(case)
    if schedule:
        s.set_tuning(schedule)
    try:
        s.step(steps)
    except mdbs.MdbsError as e:  # a cycle that is not symmetric may stall; the steps are taken
        assert e.code == mdbs.ERR_NOT_CONVERGED
    out = s.fields(), s.stats()["cg_iters"]
    s.close()
    return out


def _same(a, b, what):
    assert a[1] == b[1], what
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), (what, k)


# one CTA (up to 256 cells), one partial sum (up to 2048), two (up to 4096); unfilled last rows,
# odd sizes, levels that leave CTA 0 and levels of one warp; the last three: only the tail
SHAPES = [(1, 1, 1), (3, 2, 1), (256, 1, 1), (257, 1, 1), (2047, 1, 1), (2049, 1, 1), (4096, 1, 1), (1, 300, 1),
          (64, 64, 1), (61, 67, 1), (16, 16, 16), (13, 9, 11), (5, 4, 60), (4, 4, 256), (256, 4, 4),
          (4097, 1, 1), (33, 31, 17), (4, 70, 90)]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_equals_launches(shape, precision):
    case = _case(shape, precision)
    _same(_run(case, None), _run(case, LAUNCHES), shape)


@pytest.mark.parametrize("options", [dict(mg_nu1=0, mg_nu2=1), dict(mg_nu1=1, mg_nu2=0, max_cg=2),
                                     dict(mg_nu1=1, mg_nu2=3),
                                     dict(mg_coarse_sweeps=2)])
@pytest.mark.parametrize("shape", [(700, 1, 1), (50, 41, 1), (14, 15, 16), (33, 31, 17)])
def test_cluster_with_other_cycles(shape, options):
    case = _case(shape, 0, **options)
    _same(_run(case, None), _run(case, LAUNCHES), (shape, options))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count", [3, 40, 90])
def test_members_of_a_batch_equal_themselves_alone(count, precision):
    """With many members a CTA holds more of a domain (two, then four cells a thread)."""
    from paper_2003_08374_gb300 import mdbs
    shapes = [(1800, 1, 1), (250, 1, 1), (45, 80, 1), (9, 20, 11), (2500, 1, 1), (30, 20, 18)]
    cases = [_case(shapes[i % len(shapes)], precision) for i in range(count)]
    alone = [_run(c, None) for c in cases[: len(shapes)]]
    sims = [mdbs.Simulation(c) for c in cases]
    batch = mdbs.Batch(sims)
    batch.step(2)
    for i, s in enumerate(sims):
        _same((s.fields(), s.stats()["cg_iters"]), alone[i % len(shapes)], (i, s.n))
    batch.close()
    for s in sims:
        s.close()


@pytest.mark.parametrize("shape", [(2000, 1, 1), (63, 64, 1), (16, 15, 17)])
def test_cap_and_zero_right_hand_side(shape):
    """A solve that stops at max_cg, and one whose right-hand side is zero."""
    from paper_2003_08374_gb300 import mdbs
    got = []
    for schedule in (None, LAUNCHES):
        s = mdbs.Simulation(_case(shape, 0).replace(max_cg=2, p_tol=1e-14))
        if schedule:
            s.set_tuning(schedule)
        with pytest.raises(mdbs.MdbsError) as e:
            s.step(1)
        assert e.value.code == mdbs.ERR_NOT_CONVERGED
        got.append((s.fields(), s.stats()["cg_iters"]))
        s.close()
    _same(got[0], got[1], shape)
    still = _case(shape, 0, inlet_u=0.0, sat=0.5).replace(bc=(0, 2, 0, 0, 0, 0))
    still.permeability[:] = still.permeability[0]
    still.porosity[:] = 0.5
    f, iters = _run(still, None)
    assert iters == [0] * still.n_corr and not f["p"].any() and not f["ux"].any()

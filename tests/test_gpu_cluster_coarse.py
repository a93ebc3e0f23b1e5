"""The cluster kernels' coarsest solve and coarsest sweeps against code that is not theirs: the
cooperative kernel's tail on several levels, the one-CTA tail, and a dense solve of one level."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# levels between the finest and the tail in the cooperative kernel, which runs the tail itself
COOP = {"smooth_rows": 1, "tail_cells": 0, "snake": 0, "sweep_kz": 0, "tail_ctas": 1, "coarse_coop": 1}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_08374_gb300.build import build_library
    build_library()


def _case(shape, precision, **kw):
    from paper_2003_08374_gb300 import workloads as W
    return W.darcy_domain(shape, seed=7, precision=precision, **{"p_tol": 1e-10, "max_cg": 300, **kw})


def _run(case, tuning=None, limit=None, steps=2):
    from paper_2003_08374_gb300 import mdbs
    s = mdbs.Simulation(case)
    if limit is not None:
        s.cluster_limit(limit)
    if tuning:
        s.set_tuning(tuning)
    s.step(steps)
    s.profile()
    s.step(1)
    kernels = set(s.profile_read())
    out = s.fields(), s.stats()["cg_iters"], kernels
    s.close()
    return out


def _same(a, b, what):
    assert a[1] == b[1], what
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), (what, k)


# at least three levels, so that the cooperative kernel has one; coarsest levels of 4 to 64 cells
SHAPES = [(700, 1, 1), (4096, 1, 1), (61, 67, 1), (16, 16, 16), (13, 20, 11), (5, 4, 60), (33, 31, 17), (130, 70, 1)]


@pytest.mark.parametrize("options", [{}, {"mg_coarse_sweeps": 2}])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_equals_the_cooperative_kernel(shape, precision, options):
    case = _case(shape, precision, **options)
    a, b = _run(case), _run(case, COOP)
    assert "cg_cluster" not in b[2] and "coarse_coop" in b[2] and "tail_vcycle" not in b[2]
    _same(a, b, (shape, options))


# one level (each axis at most four cells) and several: the tail kernel of one CTA
@pytest.mark.parametrize("options", [{}, {"mg_coarse_sweeps": 2}])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 2, 1), (4, 4, 4), (4, 1, 1), (5, 1, 1), (64, 1, 1)] + SHAPES[:5])
def test_cluster_equals_the_one_cta_tail(shape, precision, options):
    case = _case(shape, precision, **options)
    a, b = _run(case), _run(case, limit=0)
    assert "cg_cluster" in a[2] and "cg_cluster" not in b[2] and "tail_vcycle" in b[2]
    _same(a, b, (shape, options))


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 1), (3, 2, 1), (4, 4, 1), (4, 3, 2), (4, 4, 4)])
def test_one_level_solves_the_dense_system(shape):
    """On one level the preconditioner is the exact inverse: a solve takes one iteration, and the
    pressure is the dense host solution of the assembled system A p = b."""
    tol = 1e-9
    case = _case(shape, 0, p_tol=tol, max_cg=3)
    from paper_2003_08374_gb300 import mdbs
    s = mdbs.Simulation(case)
    s.step(1)
    iters, p = s.stats()["cg_iters"], s.fields()["p"]
    nx, ny, nz = shape
    n = nx * ny * nz
    order = [(i, j, k) for k in range(nz) for j in range(ny) for i in range(nx)]
    pos = {c: q for q, c in enumerate(order)}
    T = [s.array(nm) if ax < 2 or nz > 1 else np.zeros(n) for ax, nm in enumerate(("Tx", "Ty", "Tz"))]
    A = np.diag(s.array("Dd").copy())
    for (i, j, k), q in pos.items():
        for ax, nb in enumerate(((i + 1, j, k), (i, j + 1, k), (i, j, k + 1))):
            if nb in pos:
                r, t = pos[nb], T[ax][q]
                A[q, q] += t
                A[r, r] += t
                A[q, r] -= t
                A[r, q] -= t
    want = np.linalg.solve(A, s.array("b"))
    s.close()
    assert iters[0] == 1 and max(iters) == 1  # (a later corrector may start below the tolerance)
    # the solve's tolerance and the dense solve's own error, both times the condition number
    bound = np.linalg.cond(A) * (tol + 8 * n * 2.0 ** -53)
    assert np.linalg.norm(p - want) <= bound * np.linalg.norm(want)

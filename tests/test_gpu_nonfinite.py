"""Matrices with an entry that is not a number: the call ends, and X does not come back finite (a
status other than OK does as well).  The entries of a column that is no number anywhere give no
pivot to choose, so every pivot search has to fall back to a row or column inside its block."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _solution(P, **kw):
    """X, or None where the library reports the factorization as failed."""
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection, SpaluError
    dev = torch.device("cuda:0")
    f = Factor(NestedDissection(P.nx, P.ny), symmetric=1 if P.symmetric else 0, **kw)
    try:
        f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    except SpaluError:
        return None
    return f.solve(torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)).cpu().numpy()


def _entry(A, i, j):
    p = A.indptr[i] + np.flatnonzero(A.indices[A.indptr[i]:A.indptr[i + 1]] == j)
    assert p.size == 1
    return int(p[0])


# eps 0: separators of 127 unknowns at the root; the others: the infected segments keep every
# unknown, so that the coarse levels have segments of more than 64
@pytest.mark.parametrize("kind,nx,ny,eps,precision", [
    ("convdiff", 255, 127, 0.0, 0), ("convdiff", 255, 127, 0.0, 1), ("diffusion", 255, 255, 4e-7, 1),
    ("convdiff", 255, 255, 4e-7, 1), ("diffusion", 255, 255, 1e-8, 0), ("convdiff", 511, 255, 1e-8, 0)])
def test_pivot_searches_stay_inside_large_blocks(kind, nx, ny, eps, precision):
    P = W.make_problem(kind, nx, seed=101, nrhs=1, ny=ny)
    node = (nx // 2 + 8) + nx * (ny // 2 + 8)      # inside a leaf at the centre of the grid
    P.A.data[_entry(P.A, node, node)] = np.nan
    X = _solution(P, eps_id=eps, precision=precision)
    assert X is None or not np.isfinite(X).all()


# The coupling of a segment's end node to its junction lies in no other block than the neighbour
# block that the segment's ID samples: an ID that takes its column for zero loses it.  At the first
# cut of the finest level, and where the two coarsest cuts meet: there the segment keeps every
# unknown on the finer levels and meets the junction again in the forms of the coarse ones.
@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf])
@pytest.mark.parametrize("coarse", [False, True])
@pytest.mark.parametrize("kind,nx,ny,precision", [("convdiff", 63, 63, 0), ("aniso", 255, 127, 0),
                                                  ("convdiff", 127, 63, 1)])
def test_neighbour_coupling_is_not_lost(kind, nx, ny, precision, coarse, value):
    if precision == 1 and np.isinf(value):
        pytest.skip("in FP32 an infinite norm also stands for finite entries whose squares overflow")
    P = W.make_problem(kind, nx, seed=102, nrhs=1, ny=ny)
    x, y = (nx // 2, ny // 2) if coarse else (15, 15)
    i, j = x - 1 + nx * y, x + nx * y
    P.A.data[_entry(P.A, i, j)] = value
    X = _solution(P, eps_id=4e-7 if precision else 1e-8, precision=precision)
    assert X is None or not np.isfinite(X).all()

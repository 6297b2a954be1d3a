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

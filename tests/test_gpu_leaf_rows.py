"""FP64 leaf sweeps over the band rows (few right-hand sides or few leaves): against dense
solves where no sparsification happens (eps = 0), and against themselves with the right-hand
sides taken one at a time (another count per warp).  Tolerances: 1e-11 as for every eps = 0
solve of these sizes (condition numbers up to 1e4); 1e-12 between groupings, whose columns
see the same operations up to the order of the atomic separator updates (1e-9 for the indefinite
Helmholtz operator, whose interchange-widened factors amplify that rounding)."""
import numpy as np
import pytest

import workloads as W
from parity import assert_close

pytestmark = pytest.mark.gpu


def _solve(P, eps, nrhs_at_once=None):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    f = Factor(NestedDissection(P.nx, P.ny), eps_id=eps, symmetric=1 if P.symmetric else 0)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
    step = nrhs_at_once or B.shape[0]
    X = torch.cat([f.solve(B[c:c + step].contiguous()) for c in range(0, B.shape[0], step)])
    return X.cpu().numpy().T


# one leaf, an odd count of leaves per warp, both cut directions, a second chunk of right-hand
# sides, and interchanges (Helmholtz: the wide upper sweep)
@pytest.mark.parametrize("kind,nx,ny,nrhs", [("diffusion", 15, 15, 1), ("diffusion", 15, 15, 3),
                                             ("convdiff", 31, 15, 5), ("laplace", 15, 31, 17),
                                             ("diffusion", 63, 31, 16), ("helmholtz", 63, 31, 1),
                                             ("helmholtz", 63, 63, 8)])
def test_against_dense(kind, nx, ny, nrhs):
    P = W.make_problem(kind, nx, seed=51, nrhs=nrhs, ny=ny)
    assert_close(_solve(P, 0.0), np.linalg.solve(P.A.to_dense(), P.B), 1e-11, f"{kind} {nx}x{ny}")


# 255 x 255 with 15 right-hand sides runs two per warp (the last warp one), alone one per warp;
# 511 x 511 with 16 by columns (a thread per leaf and right-hand side)
@pytest.mark.parametrize("kind,nx,ny,nrhs", [("diffusion", 255, 255, 15), ("helmholtz", 255, 255, 15),
                                             ("diffusion", 511, 511, 16)])
def test_groupings_agree(kind, nx, ny, nrhs):
    P = W.make_problem(kind, nx, seed=52, nrhs=nrhs, ny=ny)
    eps = 1e-8
    X, X1 = _solve(P, eps), _solve(P, eps, 1)
    assert_close(X, X1, 1e-9 if kind == "helmholtz" else 1e-12, f"{kind} {nx}x{ny}")

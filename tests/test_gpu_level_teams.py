"""Level solves whose right-hand sides move in groups of 16 bytes: every count of them around the
groups and the chunk of 16 against one at a time, on square and ragged grids, with the segment and
separator widths and groups of the tuner.  Bars: FP64 1e-12 (same factors, sums in another order);
mixed 1e-3 as for every pair of FP32 direct solves."""
import numpy as np
import pytest

import workloads as W
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,nx,ny,precision", [("diffusion", 127, 63, 0), ("convdiff", 63, 127, 0),
                                                  ("diffusion", 255, 63, 1), ("aniso", 127, 127, 1)])
@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 15, 16, 17])
def test_counts_of_right_hand_sides(kind, nx, ny, precision, nrhs):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    P = W.make_problem(kind, nx, seed=81, nrhs=nrhs, ny=ny)
    f = Factor(NestedDissection(nx, ny), eps_id=4e-7 if precision else 1e-8, symmetric=1 if P.symmetric else 0,
               precision=precision)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
    one = torch.stack([f.solve(B[c].contiguous()) for c in range(nrhs)]).cpu().numpy().T
    tol = 1e-3 if precision else 1e-12
    assert_close(f.solve(B).cpu().numpy().T, one, tol, f"{kind} {nx}x{ny} {nrhs}")
    f.tune_solve(min(nrhs, 16))
    assert_close(f.solve(B).cpu().numpy().T, one, tol, f"{kind} {nx}x{ny} {nrhs} tuned")

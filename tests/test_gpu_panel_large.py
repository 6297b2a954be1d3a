"""Separators of more than 64 unknowns with a boundary of their own, exact elimination (eps 0):
127 unknowns (LU by a cluster, boundary unknowns in groups of 32) and 255, which do not fit in
shared memory (the form in global memory).  Bars on the backward error
|b - A x| / (|A| |x| + |b|): FP64 the unit roundoff times the number of unknowns; mixed 1e-4, the
FP32 roundoff times the 1279 unknowns of the largest front."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,schur_tc", [(0, 1), (1, 1), (1, 0)])
@pytest.mark.parametrize("kind,nx,ny,kp", [("convdiff", 255, 127, 127), ("convdiff", 127, 255, 127),
                                           ("diffusion", 255, 255, 127), ("convdiff", 511, 255, 255)])
def test_backward_error(kind, nx, ny, kp, precision, schur_tc):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    P = W.make_problem(kind, nx, seed=121, nrhs=2, ny=ny)
    f = Factor(NestedDissection(nx, ny), eps_id=0.0, symmetric=1 if P.symmetric else 0, precision=precision,
               schur_tc=schur_tc)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    levels = f.stats()["levels"]
    assert levels[1]["nseg"] > 1 and levels[1]["sep_k_max"] == kp, levels[1]   # level 2: boundary not empty
    X = f.solve(torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)).cpu().numpy().T
    rows = np.add.reduceat(np.abs(P.A.data), P.A.indptr[:-1]).max()
    R = np.linalg.norm(P.B - P.A.matvec(X), axis=0)
    err = np.max(R / (rows * np.linalg.norm(X, axis=0) + np.linalg.norm(P.B, axis=0)))
    assert err <= (1e-4 if precision else 1.2e-16 * nx * ny)

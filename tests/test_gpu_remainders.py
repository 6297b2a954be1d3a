"""Segments with more than 64 remainders beside a skeleton: lines of unknowns coupled strongly along
themselves, decaying by about exp(-s) per node, and weakly (0.01) across.  A segment across the lines
keeps every unknown as long as its boxes are 64 wide, exp(-64 s) > 0.01 eps, and nearly none once
they are 128 wide (FP64: a cluster per segment, its LU in one CTA; mixed: the block forms).  The
matrix is well conditioned, so the bars on the residual of the direct solve are those of every
factorization at eps 1e-8, 1e-6, and 1e-4 in mixed mode."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,eps,s,tol", [(0, 1e-8, 0.25, 1e-6), (1, 4e-7, 0.15, 1e-4)])
def test_many_remainders(precision, eps, s, tol):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    n = 511
    P = W.make_problem("laplace", n, seed=131, nrhs=2)
    A = P.A
    off = np.abs(A.indices - np.repeat(np.arange(A.n), np.diff(A.indptr)))
    A.data[:] = np.where(off == 0, 2.0 * np.cosh(s) + 0.02, np.where(off == 1, -1.0, -0.01))
    f = Factor(NestedDissection(n), eps_id=eps, symmetric=1, precision=precision)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (A.indptr, A.indices, A.data)])
    t = f.export_level(4)
    assert np.max(np.where(t["kk"] > 0, t["cnt"] - t["kk"], 0)) > 64
    X = f.solve(torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)).cpu().numpy().T
    R = np.linalg.norm(P.B - A.matvec(X), axis=0) / np.linalg.norm(P.B, axis=0)
    assert R.max() <= tol, R

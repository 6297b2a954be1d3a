"""Sparsification by a cluster per segment (FP64, levels of few segments): against the oracle, on
sizes where both forms occur (large and small segments of a level), both symmetries, square and
ragged grids, and segments of more than 64 remainders (the LU dealt out by columns).  Bars: 1e-6
as for every FP64 factorization at eps 1e-8 (Helmholtz through the refined residual, 1e-10)."""
import numpy as np
import pytest

import workloads as W
from oracle.nd import nested_dissection
from oracle.spalu import Options as OOpts, factor as ofactor, solve as osolve
from parity import assert_close

pytestmark = pytest.mark.gpu


def _gpu(P, refine=False):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    f = Factor(NestedDissection(P.nx, P.ny), eps_id=1e-8, symmetric=1 if P.symmetric else 0)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
    X = f.solve(B)
    if refine:
        f.refine(B, X)
    return X.cpu().numpy().T, f.stats()


@pytest.mark.parametrize("kind,nx,ny", [("diffusion", 255, 127), ("convdiff", 127, 255), ("aniso", 255, 127)])
def test_against_oracle(kind, nx, ny):
    P = W.make_problem(kind, nx, seed=91, nrhs=2, ny=ny)
    X, st = _gpu(P)
    F = ofactor(P.A, nested_dissection(nx, ny), OOpts(eps=1e-8, symmetric=P.symmetric))
    assert_close(X, osolve(F, P.B), 1e-6, f"{kind} {nx}x{ny}")
    for lv in st["levels"]:
        assert abs(lv["k_max"] - F.stats["levels"][lv["level"]]["k_max"]) <= 2


@pytest.mark.parametrize("nx,ny", [(255, 255), (511, 127)])
def test_helmholtz_refined(nx, ny):
    P = W.make_problem("helmholtz", nx, seed=92, nrhs=2, ny=ny)
    X, st = _gpu(P, refine=True)
    assert max(lv["e_max"] for lv in st["levels"]) > 64
    R = P.B - P.A.matvec(X)
    assert np.max(np.linalg.norm(R, axis=0) / np.linalg.norm(P.B, axis=0)) <= 1.01e-10

"""The ID of a segment in its forms: up to 32 and up to 64 unknowns (lanes over columns), above 64
(block form); the sketch continued from the previous pass (working set in shared memory)
against the sketch redone (global scratch).  Bars: 1e-6 against the oracle as for every FP64
factorization at eps 1e-8; 1e-9 between the two places of the working set, which differ in
rounding only, amplified by the indefinite operator."""
import numpy as np
import pytest

import workloads as W
from oracle.nd import nested_dissection
from oracle.spalu import Options as OOpts, factor as ofactor, solve as osolve
from parity import assert_close

pytestmark = pytest.mark.gpu


def _solve(P, **kw):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    f = Factor(NestedDissection(P.nx, P.ny), eps_id=1e-8, symmetric=1 if P.symmetric else 0, **kw)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    X = f.solve(torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)).cpu().numpy().T
    return X, max(lv["e_max"] for lv in f.stats()["levels"])


@pytest.mark.parametrize("kind,nx,ny,emax", [("convdiff", 63, 31, 32), ("aniso", 127, 63, 64),
                                             ("diffusion", 255, 63, 64)])
def test_against_oracle(kind, nx, ny, emax):
    P = W.make_problem(kind, nx, seed=61, nrhs=2, ny=ny)
    X, e = _solve(P)
    assert e <= emax
    F = ofactor(P.A, nested_dissection(nx, ny), OOpts(eps=1e-8, symmetric=P.symmetric))
    assert_close(X, osolve(F, P.B), 1e-6, f"{kind} {nx}x{ny}")


# 255 x 255 Helmholtz has segments above 64 unknowns; 16 CTAs per SM leave no segment its place
@pytest.mark.parametrize("kind,nx,ny", [("helmholtz", 255, 255), ("aniso", 255, 127), ("diffusion", 255, 255)])
def test_places_agree(kind, nx, ny):
    P = W.make_problem(kind, nx, seed=62, nrhs=2, ny=ny)
    X, _ = _solve(P)
    Xg, _ = _solve(P, spars_ctas=16)
    assert_close(Xg, X, 1e-9, f"{kind} {nx}x{ny}")

"""Separator elimination (LU of the block, W, Z and the stored inverses, 32 boundary unknowns at a
time over the CTAs of a parent) and the CUDA-core Schur tiles, where no rank is decided (eps = 0):
separators of 15 .. 127 unknowns (one and two row sets, and the form for more than 64) against a
dense solve.  Bar: 1e-11 as for every eps = 0 solve of these condition numbers; mixed 1e-4 (FP32
factors, condition numbers up to 1e3)."""
import numpy as np
import pytest

import workloads as W
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,schur_tc,tol", [(0, 1, 1e-11), (1, 1, 1e-4), (1, 0, 1e-4)])
@pytest.mark.parametrize("kind,nx,ny", [("convdiff", 31, 15), ("convdiff", 63, 63), ("convdiff", 127, 31),
                                        ("convdiff", 63, 127)])
def test_exact_elimination(kind, nx, ny, precision, schur_tc, tol):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    P = W.make_problem(kind, nx, seed=71, nrhs=2, ny=ny)
    f = Factor(NestedDissection(nx, ny), eps_id=0.0, symmetric=0, precision=precision, schur_tc=schur_tc)
    csr = [torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)]
    B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
    f.factor(*csr)
    X = f.solve(B)
    A = torch.sparse_csr_tensor(csr[0].long(), csr[1].long(), csr[2], size=(B.shape[1],) * 2).to_dense()
    Xd = torch.linalg.solve(A, B.T)
    assert_close(X.cpu().numpy().T, Xd.cpu().numpy(), tol, f"{kind} {nx}x{ny} precision {precision}")

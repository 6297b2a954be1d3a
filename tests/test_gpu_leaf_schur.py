"""FP64 leaf Schur complements over the band rows: exact elimination (eps 0) on grids at the edges of
the forms with 2 and 5 columns per half-warp, without and with interchanges in the leaves.  Bar on the
backward error |b - A x| / (|A| |x| + |b|): 1e-11, above the unit roundoff times the number of
unknowns, 7e-12 at the largest grid."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["convdiff", "helmholtz"])
@pytest.mark.parametrize("nx,ny", [(31, 15), (127, 127), (255, 127), (255, 255)])
def test_backward_error(kind, nx, ny):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    P = W.make_problem(kind, nx, seed=93, nrhs=2, ny=ny)
    f = Factor(NestedDissection(nx, ny), eps_id=0.0, symmetric=1 if P.symmetric else 0)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    X = f.solve(torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)).cpu().numpy().T
    rows = np.add.reduceat(np.abs(P.A.data), P.A.indptr[:-1]).max()
    R = np.linalg.norm(P.B - P.A.matvec(X), axis=0)
    assert np.max(R / (rows * np.linalg.norm(X, axis=0) + np.linalg.norm(P.B, axis=0))) <= 1e-11

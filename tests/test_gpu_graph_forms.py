"""Solve kernels that a captured step takes: the headroom of its capacities leaves a level in the form
that the plain solve uses (segments and separators of at most 64 unknowns) wherever 4 unknowns of
headroom stay below that line, and a level that does change form takes that form's CTA width."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


# levels of 52 to 64 unknowns, at the geometric bound of their segments (63) and below it (127); the last
# with separators of 56
@pytest.mark.parametrize("kind,nx,ny,eps,precision", [
    ("helmholtz", 255, 255, 4e-7, 1), ("aniso", 127, 127, 1e-10, 0), ("convdiff", 255, 127, 1e-10, 0),
    ("helmholtz", 255, 127, 1e-10, 0)])
def test_captured_step_keeps_the_forms(kind, nx, ny, eps, precision):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    P = W.make_problem(kind, nx, seed=62, nrhs=2, ny=ny)
    csr = [torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)]
    B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
    nd = NestedDissection(nx, ny)
    kw = dict(eps_id=eps, symmetric=1 if P.symmetric else 0, precision=precision)
    f = Factor(nd, **kw)
    f.factor(*csr)
    plain = f.stats()["levels"]
    g = Factor(nd, **kw)
    X = torch.empty_like(B)
    for _ in range(2):                             # plain calls and capture, then a replay
        g.factor_solve_graph(*csr, B, X)
    st = g.stats()
    assert st["step_graph"]["replays"] == 1 and st["step_graph"]["refits"] == 0, st["step_graph"]
    R = P.B - P.A.matvec(X.cpu().numpy().T)
    assert np.max(np.linalg.norm(R, axis=0) / np.linalg.norm(P.B, axis=0)) <= 1.01e-10
    forms = st["step_graph"]["solve_forms"]        # per level: segments' form, separators', CTA widths
    assert len(forms) == len(plain)
    near = 0
    for p, c in zip(plain, forms):
        near += 52 <= p["e_max"] <= 60
        for q, v in enumerate((p["e_max"], p["sep_k_max"])):
            if p["solve_form"][q] and v <= 60:
                assert c[q] == 1, (p, c)
            if c[q] != p["solve_form"][q]:
                assert c[2 + q] == 256, (p, c)
    assert near > 0                                # the sizes that the test is about occur

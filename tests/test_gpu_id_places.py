"""Segments of 33 to 64 unknowns whose working set lies in shared memory against the same segments in
global scratch, where a larger sketch is formed anew instead of continued: boxes of 64 x 64 on a
1023 x 511 grid, 472 segments, several of which share an SM by default and get one SM each with
spars_ctas = 1.  The counter of spalu_stats says where they worked.  Both places run the same
operations in the same order, so the ranks are equal; bars on X: FP64 1e-9, mixed 1e-3 (the atomic
sums of two direct solves)."""
import numpy as np
import pytest

import workloads as W
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,eps,precision,tol", [("aniso", 1e-10, 0, 1e-9), ("aniso", 1e-7, 1, 1e-3)])
def test_scratch_agrees_with_shared_memory(kind, eps, precision, tol):
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    nx, ny, lev = 1023, 511, 8
    P = W.make_problem(kind, nx, seed=62, nrhs=2, ny=ny)
    csr = [torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)]
    B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
    X, level = {}, {}
    for ctas in (1, 4):
        f = Factor(NestedDissection(nx, ny), eps_id=eps, symmetric=1 if P.symmetric else 0, precision=precision,
                   spars_ctas=ctas)
        f.factor(*csr)
        X[ctas] = f.solve(B).cpu().numpy().T
        level[ctas] = f.stats()["levels"]
        del f
    one, four = level[1][lev - 1], level[4][lev - 1]
    assert one["nseg"] == 472 and 52 < one["e_max"] <= 64 and one["passes"] > one["nseg"]
    assert one["scratch"] == 0 and four["scratch"] > 0, (one, four)
    for a, b in zip(level[1], level[4]):
        assert (a["k_max"], a["k_sum"], a["e_sum"], a["passes"]) == (b["k_max"], b["k_sum"], b["e_sum"], b["passes"]), (a, b)
    assert_close(X[4], X[1], tol, f"{kind} precision {precision}")


def test_segments_of_up_to_40_unknowns_keep_their_place():
    """However many segments per SM are asked for (1984 at the finest level, 976 of up to 31 unknowns)."""
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    P = W.make_problem("diffusion", 511, seed=63, nrhs=1)
    f = Factor(NestedDissection(511), eps_id=1e-8, symmetric=1, spars_ctas=16)
    f.factor(*[torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)])
    few = [lv for lv in f.stats()["levels"] if lv["e_max"] <= 40]
    assert max(lv["nseg"] for lv in few) == 1984 and all(lv["scratch"] == 0 for lv in few), few

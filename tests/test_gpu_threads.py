"""Several host threads, each with a handle and a stream of its own: grids whose kernels ask for
different amounts of shared memory, factored and solved at the same time, against the same calls
one after the other.  Bars: FP64 1e-9, mixed 1e-3 (two FP32 direct solves)."""
import threading

import numpy as np
import pytest

import workloads as W
from parity import assert_close

pytestmark = pytest.mark.gpu


def test_handles_in_threads():
    import torch
    from paper_2408_14193_gb300 import Factor, NestedDissection
    dev = torch.device("cuda:0")
    jobs = []
    for kind, nx, ny, precision in [("diffusion", 63, 63, 0), ("helmholtz", 255, 127, 0), ("convdiff", 127, 127, 1),
                                    ("aniso", 255, 127, 1)]:
        P = W.make_problem(kind, nx, seed=111, nrhs=3, ny=ny)
        f = Factor(NestedDissection(nx, ny), eps_id=4e-7 if precision else 1e-8, symmetric=1 if P.symmetric else 0,
                   precision=precision)
        csr = [torch.from_numpy(a).to(dev) for a in (P.A.indptr, P.A.indices, P.A.data)]
        B = torch.from_numpy(np.ascontiguousarray(P.B.T)).to(dev)
        f.factor(*csr)
        ref = f.solve(B)
        jobs.append((f, csr, B, torch.zeros_like(B), ref, precision, f"{kind} {nx}x{ny}"))
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            f, csr, B, X = jobs[i][:4]
            s = torch.cuda.Stream(dev)
            for _ in range(25):
                f.factor(*csr, stream=s)
                f.solve(B, X, stream=s)
            s.synchronize()
        except Exception as exc:                   # reported by the main thread
            errors.append((jobs[i][6], exc))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for _, _, _, X, ref, precision, name in jobs:
        assert_close(X.cpu().numpy(), ref.cpu().numpy(), 1e-3 if precision else 1e-9, name)

"""CSR applies of the fixed-point kernels with 8 and 16 threads per row (32 and 64 or
more stored entries per operator row in the mean), dimensions whose last groups of
threads are ragged, against the CPU oracle; 1e-10 as in test_gpu_csr_split.py."""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,per_row,mean", [(257, 24, 32), (3001, 24, 32), (259, 48, 64), (1537, 48, 64)])
@pytest.mark.parametrize("form", ["krylov", "chebyshev"])
def test_csr_lanes(dim, per_row, mean, form):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    H0 = W.random_hermitian_csr(5, dim, per_row, True)
    V = W.random_hermitian_csr(6, dim, per_row, False, band=max(40, per_row))
    assert mean <= (H0[0][-1] + V[0][-1]) / (2 * dim) < 2 * mean  # entries per operator row: 8 or 16 threads
    drives = [lambda t: 0.7 * math.cos(1.1 * t)]
    psi0 = W.random_state(9, dim)
    dt, m = 0.2 / per_row, 16
    ref, log, _ = OC.propagate(O.Sparse(H0, [V]), psi0, 0.0, dt, 1, 4, drives, 1e-11, m, return_log=True)
    prop = P.Propagator(P.CSR(*H0), [P.CSR(*V)], drives, m_max=m, precision="fx", expm=form)
    t = torch.from_numpy(psi0).cuda()
    if form == "chebyshev":
        prop.propagate(t, 0.0, dt, 1, order=4, tol=1e-13)
    else:
        prop.propagate(t, 0.0, dt, 1, order=4, tol=1e-11, forced=log)
    assert np.linalg.norm(t.cpu().numpy() - ref) <= 1e-10
    prop.close()

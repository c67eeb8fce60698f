"""Row split and shared rows of the CSR applies: 1 to 8 threads per row (by the
mean number of entries), rows of uneven length split over 1 to many CTAs by
their work, real and complex operators side by side, against the CPU oracle.

Tolerances as in test_gpu_csr.py: 1e-10 for the fixed-point vectors with the
oracle's Krylov decisions replayed and for the Chebyshev exponentials; for
complex64 n_substeps * (4 sqrt(m_max) + 1) * 2^-24.
"""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,per_row,form", [
    (257, 2, "fx"), (257, 18, "fx"), (769, 4, "fx"), (769, 18, "fx"), (3001, 9, "fx"), (20011, 4, "fx"),
    (257, 9, "c64"), (3001, 18, "c64"), (769, 4, "cheb"), (3001, 9, "cheb")])
def test_csr_split(dim, per_row, form):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    H0 = W.random_hermitian_csr(5, dim, per_row, True)
    V = W.random_hermitian_csr(6, dim, max(1, per_row // 2), False, band=30)
    drives = [lambda t: 0.7 * math.cos(1.1 * t)]
    psi0 = W.random_state(9, dim)
    dt, m = 0.2 / per_row, 16
    ref, log, _ = OC.propagate(O.Sparse(H0, [V]), psi0, 0.0, dt, 2, 4, drives, 1e-11, m, return_log=True)
    prop = P.Propagator(P.CSR(*H0), [P.CSR(*V)], drives, m_max=m, precision="c64" if form == "c64" else "fx",
                        expm="chebyshev" if form == "cheb" else "krylov")
    t = torch.from_numpy(psi0).cuda()
    if form == "cheb":
        prop.propagate(t, 0.0, dt, 2, order=4, tol=1e-13)
        tol = 1e-10
    else:
        prop.propagate(t, 0.0, dt, 2, order=4, tol=1e-11, forced=log)
        tol = sum(map(len, log)) * (4 * math.sqrt(m) + 1) * 2.0 ** -24 if form == "c64" else 1e-10
    assert np.linalg.norm(t.cpu().numpy() - ref) <= tol

"""FP64 kernel over the sizes where its split changes: one CTA up to 256 elements,
128 elements per CTA above (ragged last CTAs), one CTA per SM from about 2^14,
several elements per thread from 2^17; explicit block and grid sizes beside the
default, and the full re-orthogonalisation, against the CPU oracle with its Krylov
decisions replayed (1e-10, as in test_gpu_parity.py)."""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,opts", [(2, {}), (6, {}), (8, {}), (9, {}), (9, dict(block_size=256)), (11, dict(block_size=32)),
                                    (12, {}), (12, dict(grid_size=3)), (12, dict(reorth=1)), (15, {}), (18, {})])
def test_f64_chain(N, opts):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    pr = W.spin_chain(N)
    psi0 = W.random_state(4, 1 << N)
    nsteps = 3 if N < 15 else 1
    ref, log, _ = OC.propagate(O.SpinChain(N, pr.J, pr.Delta, pr.h, [np.ones(N)]), psi0, 0.0, 0.02, nsteps, 4,
                               [pr.drive], 1e-11, 16, return_log=True, reorth=bool(opts.get("reorth")))
    prop = P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, np.ones(N))], [pr.drive], m_max=16,
                        precision="f64", **opts)
    for _ in range(2):  # the second call continues the exchange's tags over cleared records
        t = torch.from_numpy(psi0).cuda()
        prop.propagate(t, 0.0, 0.02, nsteps, order=4, tol=1e-11, forced=log)
        assert np.linalg.norm(t.cpu().numpy() - ref) <= 1e-10
    prop.close()


@pytest.mark.parametrize("dim", [255, 257, 300, 1025, 19001])
def test_f64_csr(dim):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    H0 = W.random_hermitian_csr(5, dim, 5, True)
    V = W.random_hermitian_csr(6, dim, 2, False, band=30)
    drives = [lambda t: 0.7 * math.cos(1.1 * t)]
    psi0 = W.random_state(9, dim)
    ref, log, _ = OC.propagate(O.Sparse(H0, [V]), psi0, 0.0, 0.04, 2, 4, drives, 1e-11, 16, return_log=True)
    prop = P.Propagator(P.CSR(*H0), [P.CSR(*V)], drives, m_max=16, precision="f64")
    t = torch.from_numpy(psi0).cuda()
    prop.propagate(t, 0.0, 0.04, 2, order=4, tol=1e-11, forced=log)
    assert np.linalg.norm(t.cpu().numpy() - ref) <= 1e-10
    prop.close()

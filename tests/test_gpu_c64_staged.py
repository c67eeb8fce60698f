"""Complex64 chains staged in the shared memory of 128 CTAs (17 to 21 sites):
against the CPU oracle at 17 and 18 sites with its Krylov decisions replayed,
within n_substeps * (4 sqrt(m_max) + 1) * 2^-24 (test_gpu_c64.py), and against
the element-wise form at every size of the range: the sums run in the same
order, so with the same decisions only the partition of the compensated
reductions differs (below 1e-12)."""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu
M = 16


def _budget(nsub):
    return nsub * (4 * math.sqrt(M) + 1) * 2.0 ** -24


def _prop(N, a, form):
    import paper_1102_5071_gb300 as P
    pr = W.spin_chain(N)
    return P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, a)], [pr.drive], m_max=M, precision="c64",
                        apply_form=form)


def _field(N, uniform):
    return np.ones(N) if uniform else W.uniform(3, N, 0.5, 1.5)


@pytest.mark.parametrize("N,uniform", [(17, True), (18, False)])
def test_staged_matches_oracle(N, uniform):
    torch = pytest.importorskip("torch")
    pr, a = W.spin_chain(N), _field(N, uniform)
    psi0 = W.random_state(4, 1 << N)
    ref, log, _ = OC.propagate(O.SpinChain(N, pr.J, pr.Delta, pr.h, [a]), psi0, 0.0, 0.02, 1, 4, [pr.drive], 1e-9, M,
                               return_log=True)
    t = torch.from_numpy(psi0).cuda()
    prop = _prop(N, a, "auto")
    prop.propagate(t, 0.0, 0.02, 1, order=4, tol=1e-9, forced=log)
    assert np.linalg.norm(t.cpu().numpy() - ref) <= _budget(sum(map(len, log)))
    prop.close()


@pytest.mark.parametrize("N,uniform", [(17, False), (19, True), (20, False), (21, True), (21, False)])
def test_staged_matches_elementwise(N, uniform):
    torch = pytest.importorskip("torch")
    a = _field(N, uniform)
    psi0 = torch.from_numpy(W.random_state(5, 1 << N)).cuda()
    out, log = [], None
    for form in ("elementwise", "auto"):
        prop = _prop(N, a, form)
        t = psi0.clone()
        if log is None:
            _, log = prop.propagate(t, 0.0, 0.02, 2, order=4, tol=1e-9, record=True)
        else:
            prop.propagate(t, 0.0, 0.02, 2, order=4, tol=1e-9, forced=log)
        out.append(t)
        prop.close()
    assert torch.linalg.vector_norm(out[0] - out[1]).item() <= 1e-12

"""Re-orthogonalised FP64 propagation over many launches with one Lanczos iteration
each (replayed decisions of dimension 1): every launch then crosses the grid barrier
exactly once, and each has to wait there although the launch before ended at the same
count.  Against the CPU oracle with the same decisions, 1e-10 as in
test_gpu_reorth.py."""

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [9, 13, 15])
def test_one_iteration_per_launch(N):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    pr = W.spin_chain(N)
    psi0 = W.random_state(4, 1 << N)
    nsteps, log = 6, [[(1, 0)]] * 6  # order 2: one stage exponential per step
    ref = OC.propagate(O.SpinChain(N, pr.J, pr.Delta, pr.h, [np.ones(N)]), psi0, 0.0, 0.02, nsteps, 2, [pr.drive], 1e-11,
                       16, forced_log=log, reorth=True)
    prop = P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, np.ones(N))], [pr.drive], m_max=16,
                        precision="f64", reorth=True, steps_per_launch=1)
    for _ in range(5):
        t = torch.from_numpy(psi0).cuda()
        prop.propagate(t, 0.0, 0.02, nsteps, order=2, tol=1e-11, forced=log)
        assert np.linalg.norm(t.cpu().numpy() - ref) <= 1e-10
    prop.close()

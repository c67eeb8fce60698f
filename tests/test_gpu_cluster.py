"""Fixed-point chains of 10 to 13 sites on one thread-block cluster (the applied
vector staged in the cluster's shared memory, records exchanged there), against
the CPU oracle with its Krylov decisions replayed (1e-10, as in
test_gpu_parity.py), and against the launch over independent CTAs with exact
integer sums in both: identical states."""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,uniform,order,nsteps", [(10, True, 4, 3), (11, False, 4, 2), (12, True, 6, 2),
                                                    (13, False, 6, 1), (13, True, 8, 1)])
def test_cluster_matches_oracle(N, uniform, order, nsteps):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    pr = W.spin_chain(N)
    a = np.ones(N) if uniform else W.uniform(3, N, 0.5, 1.5)
    psi0 = W.random_state(4, 1 << N)
    ref, log, _ = OC.propagate(O.SpinChain(N, pr.J, pr.Delta, pr.h, [a]), psi0, 0.0, 0.02, nsteps, order, [pr.drive],
                               1e-11, 16, return_log=True)
    out = []
    for grid in (0, (1 << N) // 768 + 1):  # the cluster; the same elements over independent CTAs
        prop = P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, a)], [pr.drive], m_max=16,
                            grid_size=grid, steps_per_launch=1)
        for _ in range(2):  # the second call replays the captured launches
            t = torch.from_numpy(psi0).cuda()
            prop.propagate(t, 0.0, 0.02, nsteps, order=order, tol=1e-11, forced=log)
            out.append(t.cpu().numpy())
            assert np.linalg.norm(out[-1] - ref) <= 1e-10
        t = torch.from_numpy(psi0).cuda()
        st = prop.propagate(t, 0.0, 0.02, nsteps, order=order, tol=1e-11)
        assert np.linalg.norm(t.cpu().numpy() - ref) <= 1e-10 and math.isclose(st["n_exp"], len(log))
        prop.close()
    assert all(np.array_equal(out[0], o) for o in out[1:])

"""Batches of small and mixed instances under the default plan and under plans of
every CTA size: sums over one, some or all warps of a CTA, parts that are empty,
the staged and the gathering passes, and both register forms of the kernel (all
items resident at once or not), against the oracle with its Krylov decisions
replayed.  Tolerances as in test_gpu_batch.py."""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "c64"])
@pytest.mark.parametrize("sizes,copies,plan", [
    ([1, 2, 6, 7], 4, None), ([6, 7], 350, None), ([8, 9], 10, None), ([7, 10], 200, (1, 128, 25)),
    ([5, 9, 11], 3, (8, 512, 5)), ([12, 6], 2, (8, 128, 12)), ([11, 13], 3, None), ([10, 12], 120, (4, 256, 12))])
def test_batch_small(sizes, copies, plan, precision):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    u = W.uniform(3, 2 * len(sizes))
    insts = [W.ChainInstance(N, 1.0, 0.5, W.uniform(200 + i, N, -1, 1), 0.5 + 1.5 * u[i], 1.0 + 2.0 * u[len(sizes) + i],
                             300 + i) for i, N in enumerate(sizes)]
    refs, logs, psi = [], [], []
    for c in insts:
        psi.append(W.random_state(c.psi_seed, 1 << c.N))
        r, log, _ = OC.propagate(O.SpinChain(c.N, c.J, c.Delta, c.h, [c.xfield]), psi[-1], 0.0, 0.02, 1, 4, [c.drive],
                                 1e-11, 16, return_log=True, max_substeps=200)
        refs.append(r)
        logs.append(log)
    prop = P.BatchPropagator([P.Chain(c.N, c.J, c.Delta, c.h, c.xfield, None, c.A, c.omega, 0.0) for c in insts] * copies,
                             m_max=16, precision=precision)
    if plan:
        prop.set_plan(*plan)
    states = [torch.from_numpy(p).cuda() for _ in range(copies) for p in psi]
    prop.propagate(states, 0.0, 0.02, 1, order=4, tol=1e-11, forced=logs * copies)
    for i, t in enumerate(states):
        log = logs[i % len(sizes)]
        tol = 1e-10 if precision == "f64" else sum(map(len, log)) * (4 * math.sqrt(16) + 1) * 2.0 ** -24
        assert np.linalg.norm(t.cpu().numpy() - refs[i % len(sizes)]) <= tol, (i, sizes[i % len(sizes)])
    prop.close()

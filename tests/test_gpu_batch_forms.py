"""Batches in which the choice between the two register forms of the kernel and the
room for staged vectors depends on the longest item: one that is too large to be
staged beside many that are not (nothing staged), one that is staged although it
leaves room for one CTA per SM only, more items than CTAs of 128 registers, and
uniform batches that take the other form; against the oracle with its Krylov
decisions replayed.  Tolerances as in test_gpu_batch.py."""

import math

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu

MIXED = [14] + [10, 8, 6] * 14          # a long one and 42 short ones
LARGE = [15] + [9, 11] * 8              # 2^15 elements do not fit one CTA in either format


@pytest.mark.parametrize("precision", ["f64", "c64"])
@pytest.mark.parametrize("sizes,plan", [
    (LARGE, (1, 128, 25)), (LARGE, (1, 512, 25)), (LARGE, (2, 512, 13)), (MIXED, (1, 256, 25)), (MIXED, (8, 512, 8)),
    (MIXED, (4, 512, 10)), (MIXED, None), ([12] * 40, (4, 512, 12)), ([11] * 60, None), ([12, 13] * 30, None)])
def test_batch_forms(sizes, plan, precision):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    ref, log, psi, chain = {}, {}, {}, {}
    for N in sorted(set(sizes)):
        c = chain[N] = W.ChainInstance(N, 1.0, 0.5, W.uniform(200 + N, N, -1, 1), 1.0, 1.7, 300 + N)
        psi[N] = W.random_state(c.psi_seed, 1 << N)
        ref[N], log[N], _ = OC.propagate(O.SpinChain(N, c.J, c.Delta, c.h, [c.xfield]), psi[N], 0.0, 0.02, 1, 2, [c.drive],
                                         1e-10, 16, return_log=True, max_substeps=200)
    prop = P.BatchPropagator([P.Chain(N, chain[N].J, chain[N].Delta, chain[N].h, chain[N].xfield, None, chain[N].A,
                                      chain[N].omega, 0.0) for N in sizes], m_max=16, precision=precision)
    if plan:
        prop.set_plan(*plan)
    states = [torch.from_numpy(psi[N]).cuda() for N in sizes]
    prop.propagate(states, 0.0, 0.02, 1, order=2, tol=1e-10, forced=[log[N] for N in sizes])
    for N, t in zip(sizes, states):
        tol = 1e-10 if precision == "f64" else sum(map(len, log[N])) * (4 * math.sqrt(16) + 1) * 2.0 ** -24
        assert np.linalg.norm(t.cpu().numpy() - ref[N]) <= tol, N
    prop.close()

"""Explicit block and grid sizes of the FP64 kernel: block_size threads per CTA and the
grid that was asked for (one thread per element, or grid_size, up to what is resident
at once), with the counter barrier of large grids in several launches, against the
CPU oracle with its Krylov decisions replayed (1e-10, as in test_gpu_parity.py)."""

import ctypes as C

import numpy as np
import pytest

import workloads as W
from oracle import cfet as OC, operators as O

pytestmark = pytest.mark.gpu


def shape(prop):
    g, b = C.c_int32(), C.c_int32()
    assert prop._lib.cfet_selftest_launch_shape(prop._ctx, C.byref(g), C.byref(b)) == 0
    return g.value, b.value


@pytest.mark.parametrize("N,opts,grid,block", [
    (9, dict(block_size=256), 2, 256), (10, dict(block_size=32), 32, 32), (10, dict(block_size=96), 11, 96),
    (12, dict(block_size=160), 26, 160), (14, dict(block_size=64), 256, 64),
    (15, dict(block_size=64), 512, 64), (15, dict(block_size=32), 1024, 32), (14, dict(block_size=64, grid_size=161), 161, 64),
    (14, dict(block_size=64, grid_size=224), 224, 64), (14, dict(block_size=64, grid_size=225), 225, 64), (14, dict(block_size=128, grid_size=300), 300, 128),
    (12, dict(grid_size=16), 16, 256), (14, dict(block_size=64, reorth=1), 256, 64)])
def test_explicit_sizes(N, opts, grid, block):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    pr = W.spin_chain(N)
    psi0 = W.random_state(4, 1 << N)
    ref, log, _ = OC.propagate(O.SpinChain(N, pr.J, pr.Delta, pr.h, [np.ones(N)]), psi0, 0.0, 0.02, 2, 4, [pr.drive],
                               1e-11, 16, return_log=True, reorth=bool(opts.get("reorth")))
    prop = P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, np.ones(N))], [pr.drive], m_max=16,
                        precision="f64", steps_per_launch=1, **opts)
    assert shape(prop) == (grid, block)
    for _ in range(2):
        t = torch.from_numpy(psi0).cuda()
        prop.propagate(t, 0.0, 0.02, 2, order=4, tol=1e-11, forced=log)
        assert np.linalg.norm(t.cpu().numpy() - ref) <= 1e-10
    prop.close()

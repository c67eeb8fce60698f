"""Explicit block sizes of the fixed-point kernel on chains of 9 to 13 sites: the
thread-block cluster only where its parts are at most two elements per thread,
otherwise as many independent CTAs as there are elements for; exact sums in both, so
the states are those of the default launch, bit for bit."""

import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,block_size,grid,block", [
    (9, 32, 8, 96), (9, 64, 2, 160), (10, 32, 16, 96), (12, 32, 64, 96), (13, 32, 128, 96), (13, 96, 43, 224),
    (13, 128, 16, 288), (13, 384, 16, 544)])
def test_cluster_or_grid_by_block_size(N, block_size, grid, block):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    pr = W.spin_chain(N)
    psi0 = W.random_state(4, 1 << N)
    out = []
    for bs in (0, block_size):
        prop = P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, np.ones(N))], [pr.drive], m_max=16,
                            block_size=bs)
        g, b = C.c_int32(), C.c_int32()
        assert prop._lib.cfet_selftest_launch_shape(prop._ctx, C.byref(g), C.byref(b)) == 0
        t = torch.from_numpy(psi0).cuda()
        prop.propagate(t, 0.0, 0.02, 2, order=4, tol=1e-11)
        out.append(t.cpu().numpy())
        prop.close()
    assert (g.value, b.value) == (grid, block)
    assert np.array_equal(*out)

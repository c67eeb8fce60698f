"""Two propagators of one kernel alive at the same time: a kernel's limit of dynamic
shared memory is one value for the whole process, so making the smaller one must
not take away what the larger one's launches need.  The larger is made first and
run last; its states are those of a run on its own, bit for bit (same launch, sums
in a fixed order)."""

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("large,small,precision", [(9, 8, "fx"), (13, 10, "fx"), (21, 17, "c64")],
                         ids=["fx-one-cta", "fx-cluster", "c64-staged"])
def test_smaller_context_leaves_the_larger_one_usable(large, small, precision):
    torch = pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P

    def make(N):
        pr = W.spin_chain(N)
        return P.Propagator(P.XXZChain(N, pr.J, pr.Delta, pr.h), [P.XField(N, np.ones(N))], [pr.drive], m_max=16,
                            precision=precision)

    def run(prop, N):
        t = torch.from_numpy(W.random_state(4, 1 << N)).cuda()
        prop.propagate(t, 0.0, 0.02, 1, order=4, tol=1e-6)
        return t.cpu().numpy()

    lone = make(large)
    ref = run(lone, large)
    lone.close()
    a = make(large)
    b = make(small)
    assert abs(np.linalg.norm(run(b, small)) - 1.0) <= 1e-4
    assert np.array_equal(run(a, large), ref)
    b.close()
    a.close()

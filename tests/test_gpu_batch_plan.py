"""The plan of a complex64 batch before any tuning: chains that one CTA can stage are
spread over a cluster only while the chip has CTAs for them."""

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,spread_from", [
    ([11] * 16, None), ([11] * 256, None), ([12] * 16, 12), ([12] * 48, 12), ([12] * 100, None),
    ([10, 11, 12] * 85, None), ([8, 13] * 20, 13), ([12, 13] * 128, None), ([14] * 100, 13), ([10, 16] * 50, 14)])
def test_default_plan(sizes, spread_from):
    pytest.importorskip("torch")
    import paper_1102_5071_gb300 as P
    b = P.BatchPropagator([P.Chain(N, 1.0, 0.5, W.uniform(1, N), np.ones(N), None, 1.0, 2.0, 0.0) for N in sizes],
                          precision="c64")
    plan = b.plan
    b.close()
    spread = [N for N in sizes if N >= plan["coop_min_sites"]]
    assert plan["cluster_size"] == 8
    if spread_from is None:
        assert not spread
    else:
        assert spread and min(spread) >= spread_from and max(sizes) in spread

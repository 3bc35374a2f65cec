"""The measurement product v_b = N g_b at the edges of its row blocks, column
slices and anchor groups, through the measured G.

Tolerances: float64 that of the measurement parity tests; float32 1e-4 of the
largest |G|, that of the mixed form's measurement (float32 positions and sums).
"""
import numpy as np
import pytest

from parity import compare_config, oracle_for
from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


# orders around blocks of 64 rows and slices of 64 and 128 columns; up to 8
# anchors in one group, more in several, the last one partial
@pytest.mark.parametrize("precision", [pk.CTAUX_FP64, pk.CTAUX_MIXED])
@pytest.mark.parametrize("n,anchors", [(1, 1), (31, 2), (33, 3), (64, 4), (65, 8), (129, 5), (513, 6), (600, 7),
                                       (129, 9), (200, 17), (600, 64), (1025, 4)])
def test_edges(n, anchors, precision):
    ch = configs.cube8(K=float(max(16, n)), k_max=4, capacity=n + 64)
    cfg = configs.synthetic_configuration(ch, n, seed=n + anchors)
    oc = oracle_for(ch)
    oc.set_config(cfg["tau"], cfg["site"], cfg["s"], cfg["birth"], cfg["t"])
    with pk.Context([ch], precision=precision, refresh_every=0, n_tau_bins=anchors, n_anchors=anchors) as ctx:
        ctx.set_config(0, **cfg)
        ctx.reset_measurements()
        ctx.sweep(1, measure=True)   # a few proposals: the order stays within 4 of n
        G = ctx.measure_G(0)[0]
        oc.run(ctx.stats(0)["t"] - oc.t)
        compare_config(ctx, 0, oc)
        ref = oc.measure_G(anchors, anchors)
        if precision == pk.CTAUX_FP64:
            np.testing.assert_allclose(G, ref, rtol=1e-9, atol=1e-10 * max(1.0, np.abs(ref).max()))
        else:
            np.testing.assert_allclose(G, ref, rtol=0, atol=1e-4 * max(1.0, np.abs(ref).max()))

"""From-scratch recomputations of several chains together."""
import dataclasses

import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


@pytest.mark.parametrize("sizes", [((300, 400), (900, 1500)), ((500, 960), (500, 961), (40, 64)),
                                   ((60, 200), (150, 13000))])
def test_recomputation_in_a_mixed_set_gives_the_bits_of_the_chain_alone(sizes):
    """(order, capacity) on both sides of the line between panels in one and two levels,
    and of the one between panels of 32 and 16 columns."""
    chains = [configs.cube8(K=256.0, k_max=32, capacity=cap) for _, cap in sizes]
    chains = [dataclasses.replace(c, chain_id=i) for i, c in enumerate(chains)]
    cfgs = [configs.synthetic_configuration(c, n, seed=9 + i) for i, (c, (n, _)) in enumerate(zip(chains, sizes))]

    def state(ctx, i):
        return [ctx.get_N(i, 0), ctx.get_N(i, 1), np.array(ctx.stats(i)["logdet"])]

    with pk.Context(chains) as ctx:
        for i, cfg in enumerate(cfgs):
            ctx.set_config(i, **cfg)
        each = [state(ctx, i) for i in range(len(chains))]
        ctx.recompute()
        together = [state(ctx, i) for i in range(len(chains))]
    for i, cfg in enumerate(cfgs):
        with pk.Context([chains[i]]) as ctx:
            ctx.set_config(0, **cfg)
            alone = state(ctx, 0)
        for a, e, t in zip(alone, each[i], together[i]):
            np.testing.assert_array_equal(e, a)
            np.testing.assert_array_equal(t, a)

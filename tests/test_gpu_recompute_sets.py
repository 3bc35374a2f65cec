"""From-scratch recomputations of several chains together."""
import dataclasses

import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


@pytest.mark.parametrize("sizes", [((300, 400), (900, 1500)), ((767, 1000), (768, 1000), (40, 64)),
                                   ((60, 200), (150, 13000))])
def test_recomputation_in_a_mixed_set_gives_the_bits_of_the_chain_alone(sizes):
    """(order, capacity) on both sides of the line between panels in one and two levels
    (order 768), and of the one between panels of 32 and 16 columns."""
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


@pytest.mark.parametrize("capacity", [600, 6000])
def test_recomputation_is_launched_up_to_the_order(capacity):
    """Launches of the recomputation phase: at most three per 32 columns and three
    more per 128 up to the order and the insertions since it was last known, and
    four around them."""
    k, n = 32, 200
    ch = configs.cube8(K=256.0, k_max=k, capacity=capacity)
    with pk.Context([ch], refresh_every=2) as ctx:
        ctx.set_config(0, **configs.synthetic_configuration(ch, n, seed=1))
        before = ctx.phase_times()
        ctx.sweep(2)
        ctx.synchronize()
        after = ctx.phase_times()
        ctx.recompute()
        last = ctx.phase_times()
    refresh = pk.Context.PHASES.index("refresh")

    def launches(a, b):
        return b[1][refresh] - a[1][refresh]

    def most(order):
        return 4 + 3 * -(-order // 32) + 3 * -(-order // 128)

    assert 0 < launches(before, after) <= most(n + 2 * k)
    assert 0 < launches(after, last) <= most(n + 2 * k)


def test_recomputation_of_a_growing_chain_reaches_its_whole_order():
    """From an empty configuration, many blocks and recomputations in one call: N is the
    inverse of the configuration that was reached, as another context rebuilds it."""
    k = 64
    ch = configs.cube8(K=256.0, k_max=k, capacity=3000)
    with pk.Context([ch], refresh_every=1) as ctx:
        ctx.sweep(40)
        ctx.sweep(1)
        cfg = ctx.get_config(0)
        N = [ctx.get_N(0, spin) for spin in (0, 1)]
    assert len(cfg["tau"]) > 200
    with pk.Context([ch]) as ctx:
        ctx.set_config(0, cfg["tau"], cfg["site"], cfg["s"], cfg["birth"], cfg["t"])
        for spin in (0, 1):
            np.testing.assert_array_equal(ctx.get_N(0, spin), N[spin])


def test_captured_sweeps_replayed_past_the_orders_seen_by_the_host():
    """A caller's graph of a block and a recomputation, replayed while the chain grows
    from an empty configuration, gives the chain of the same calls made directly."""
    torch = pytest.importorskip("torch")
    ch = configs.cube8(K=256.0, k_max=64, capacity=1000)

    def state(ctx):
        return [ctx.get_config(0)["tau"], ctx.get_N(0, 0), ctx.get_N(0, 1)]

    with pk.Context([ch], refresh_every=1) as ctx:
        ctx.sweep(13)
        direct = state(ctx)
    with pk.Context([ch], refresh_every=1) as ctx:
        stream = torch.cuda.Stream()
        ctx.sweep(1, stream=stream.cuda_stream)   # kernels loaded before the capture
        ctx.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            ctx.sweep(1, stream=stream.cuda_stream)
        with torch.cuda.stream(stream):
            for _ in range(11):
                graph.replay()
        stream.synchronize()
        ctx.sweep(1, stream=stream.cuda_stream)
        ctx.synchronize()
        for a, b in zip(state(ctx), direct):
            np.testing.assert_array_equal(a, b)

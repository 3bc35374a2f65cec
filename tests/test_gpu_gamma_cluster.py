"""Proposals with Gamma^{-1} spread over a cluster: the same bits as one CTA per chain.

One chain alone runs on a cluster of 16 CTAs, the same chain among others on
smaller clusters and in a large batch on one CTA: decisions, ratios and N must be
equal bit for bit, in float64 and float32, with slots changed twice (flips and
removals of vertices inserted in the same block) and near-tie stops on the way.
"""
import dataclasses

import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n0,k", [(3, 25), (40, 33), (90, 64), (150, 130)])
def test_cluster_sizes_give_the_same_bits(n0, k, precision):
    base = configs.cube8(K=60.0, k_max=k, capacity=420)
    prec = pk.CTAUX_FP64 if precision == "fp64" else pk.CTAUX_MIXED
    cfg = configs.synthetic_configuration(base, n0, seed=7)
    got = []
    for n_chains in (1, 16, 30, 80):     # clusters of 16, 8, 4 (2 from 39 chains on), one CTA
        chains = [dataclasses.replace(base, chain_id=i) for i in range(n_chains)]
        with pk.Context(chains, precision=prec, trace_capacity=4 * k, p_insert=0.4, p_flip=0.3,
                        refresh_every=0) as ctx:
            for i in range(n_chains):
                ctx.set_config(i, **cfg)
            ctx.sweep(4)
            ctx.synchronize()
            got.append((ctx.trace(0), ctx.get_N(0, 0), ctx.get_N(0, 1), ctx.stats(0)))
    t0, a0, b0, s0 = got[0]
    assert len(t0) > 0 and (t0["accept"] & 1).any()
    for t, a, b, s in got[1:]:
        assert t.tobytes() == t0.tobytes()
        np.testing.assert_array_equal(a, a0)
        np.testing.assert_array_equal(b, b0)
        assert s["accepted"] == s0["accepted"] and s["proposals"] == s0["proposals"]
        assert s["near_ties"] == s0["near_ties"] and s["sign"] == s0["sign"]

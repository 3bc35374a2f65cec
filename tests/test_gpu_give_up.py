"""A bounded wait of the sliced float64 products that runs out (no GPU fault: the
test setting of tc_wait_limit lets one CTA wait on a barrier that nothing completes).
"""
import dataclasses

import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


def _chains(k, n_chains):
    base = configs.cube8(K=256.0, k_max=k, capacity=1024)
    chains = [dataclasses.replace(base, chain_id=i) for i in range(n_chains)]
    return chains, [configs.synthetic_configuration(c, 430 + i, seed=3 + i) for i, c in enumerate(chains)]


def _give_up(ctx, cfgs):
    for i, cfg in enumerate(cfgs):
        ctx.set_config(i, **cfg)
    ctx.sweep(1)
    with pytest.raises(pk.CtauxError) as ei:
        ctx.synchronize()
    assert ei.value.code == 7                      # CTAUX_ETIMEOUT


@pytest.mark.parametrize("k,n_chains", [(64, 1), (64, 8), (160, 2)])
def test_every_chain_of_a_product_that_gave_up_reports_it(k, n_chains):
    """Also those whose items the CTA would have come to later: none goes on with a
    product that is missing a part."""
    chains, cfgs = _chains(k, n_chains)
    with pk.Context(chains, refresh_every=0, trace_capacity=4 * k, tc_wait_limit=-20000) as ctx:
        _give_up(ctx, cfgs)
        assert all(ctx.stats(i)["status"] & 8 for i in range(n_chains))
        assert all(len(ctx.trace(i)) == 0 for i in range(n_chains))


@pytest.mark.parametrize("k,n_chains", [(64, 1), (64, 8), (160, 2)])
def test_chains_recover_from_a_product_that_gave_up(k, n_chains):
    """After ctaux_set_config they go on as in a context where nothing happened: no
    half-arrived split product is left."""
    chains, cfgs = _chains(k, n_chains)
    kw = dict(refresh_every=0, trace_capacity=4 * k)
    with pk.Context(chains, **kw) as ctx:
        for i, cfg in enumerate(cfgs):
            ctx.set_config(i, **cfg)
        ctx.sweep(3)
        ctx.synchronize()
        clean = [ctx.trace(i) for i in range(n_chains)]
    with pk.Context(chains, tc_wait_limit=-20000, **kw) as ctx:
        _give_up(ctx, cfgs)
        for i, cfg in enumerate(cfgs):
            try:
                ctx.set_config(i, **cfg)
            except pk.CtauxError as e:             # reports the chains that still wait
                assert e.code == 7 and i + 1 < n_chains
        ctx.sweep(3)
        ctx.synchronize()
        for i in range(n_chains):
            tr = ctx.trace(i)
            assert len(tr) == len(clean[i])
            for name in tr.dtype.names:
                np.testing.assert_array_equal(tr[name], clean[i][name])


def test_every_chain_of_a_mixed_flush_that_gave_up_reports_it():
    """The same for the tensor-core flush of the mixed form, whose test setting stalls
    every CTA: chains that no CTA begins with stop as well."""
    chains, cfgs = _chains(64, 24)
    with pk.Context(chains, precision=pk.CTAUX_MIXED, refresh_every=0, tc_wait_limit=-2000) as ctx:
        _give_up(ctx, cfgs)
        assert all(ctx.stats(i)["status"] & 8 for i in range(24))

"""Contexts that live side by side, and the chains of one context beside each other."""
import dataclasses

import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


def _start(chains, orders, **kw):
    ctx = pk.Context(chains, **kw)
    for i, (ch, n) in enumerate(zip(chains, orders)):
        ctx.set_config(i, **configs.synthetic_configuration(ch, n, seed=50 + ch.chain_id))
    return ctx


def _same_traces(a, b):
    assert len(a) == len(b) > 0
    for name in a.dtype.names:
        np.testing.assert_array_equal(a[name], b[name], err_msg=name)


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("form,k,other_k", [("inverse", 32, 32), ("lu", 192, 8)])
def test_smaller_context_created_later_leaves_the_first_one_running(use_graph, form, k, other_k):
    """The limits that a context asks for its kernels hold for the process, so a
    second context may not lower them (fewer chains; a shorter block)."""
    from paper_1010_3690_gb300 import ctaux
    base = configs.cube8(K=64.0, k_max=k, capacity=400)
    chains = [dataclasses.replace(base, chain_id=i) for i in range(40 if form == "inverse" else 2)]
    orders = [100 + 3 * i for i in range(len(chains))]
    kw = dict(trace_capacity=4 * k, refresh_every=0, use_graph=use_graph,
              gamma_form=ctaux.CTAUX_GAMMA_LU if form == "lu" else ctaux.CTAUX_GAMMA_INVERSE)
    with _start(chains, orders, **kw) as ctx:
        ctx.sweep(3)
        ctx.synchronize()
        alone = [ctx.trace(i) for i in range(len(chains))]
    with _start(chains, orders, **kw) as ctx:
        other = [dataclasses.replace(base, chain_id=99, k_max=other_k)]
        with _start(other, [120], **dict(kw, trace_capacity=0)) as second:
            for _ in range(3):
                ctx.sweep(1)
                second.sweep(1)
            ctx.synchronize()
            second.synchronize()
        for i in range(len(chains)):
            _same_traces(ctx.trace(i), alone[i])

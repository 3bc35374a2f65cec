"""Float64 products on the float16 tensor cores (sliced operands) at their edges.

The tolerance is the one of the float64 parity tests (1e-10 of the matrix
scale): a sliced product's error is below that of a chain of float64
multiply-adds, and the oracle's N comes from a dense float64 inverse.
"""
import numpy as np
import pytest

from parity import compare_traces, oracle_for
from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


def _check_N(ctx, chains, cfgs):
    for i, (ch, cfg) in enumerate(zip(chains, cfgs)):
        oc = oracle_for(ch)
        oc.set_config(cfg["tau"], cfg["site"], cfg["s"], cfg["birth"], cfg["t"])
        st = ctx.stats(i)
        for spin in (0, 1):
            No = oc.N(spin)
            np.testing.assert_allclose(ctx.get_N(i, spin), No, rtol=1e-10, atol=1e-10 * np.abs(No).max())
            assert st["logdet"][spin] == pytest.approx(oc.slogdet(spin, oc.tau, oc.site, oc.s)[1],
                                                       rel=1e-11, abs=1e-9)


@pytest.mark.parametrize("orders,capacity", [
    ((1, 33, 127, 128), 1500),        # panels in two levels (leading dimension >= 1408), 8 matrices
    ((129, 160, 257, 1030, 96), 1500),  # the same, clusters of 8 CTAs
    ((31, 64, 300) + (17,) * 127, 320),  # one level, clusters of 4 CTAs
])
def test_recomputation_of_uneven_chains_together(orders, capacity):
    base = configs.cube8(K=256.0, k_max=32, capacity=capacity)
    chains = [configs.dataclasses.replace(base, chain_id=i) for i in range(len(orders))]
    cfgs = [configs.synthetic_configuration(c, n, seed=100 + i) for i, (c, n) in enumerate(zip(chains, orders))]
    with pk.Context(chains) as ctx:
        for i, cfg in enumerate(cfgs):
            ctx.set_config(i, **cfg)
        ctx.recompute()   # every chain in one set of launches
        _check_N(ctx, chains[:5], cfgs[:5])


@pytest.mark.parametrize("n0,k", [(40, 256), (100, 32), (127, 64), (128, 64), (129, 160), (257, 256), (511, 24)])
def test_sliced_products_of_a_block_at_tile_edges(n0, k):
    """Prep (tiles of 128 rows x 64 insertions, parts of 128 of the inner index, split
    over it) and flush (ranks up to 256, two parts) against the oracle's ratios and N."""
    ch = configs.cube8(K=256.0, k_max=k, capacity=n0 + 2 * k + 64)
    cfg = configs.synthetic_configuration(ch, n0, seed=n0)
    oc = oracle_for(ch, p_insert=0.45, p_flip=0.1)
    oc.set_config(cfg["tau"], cfg["site"], cfg["s"], cfg["birth"], cfg["t"])
    with pk.Context([ch], trace_capacity=2 * k, refresh_every=0, p_insert=0.45, p_flip=0.1) as ctx:
        ctx.set_config(0, **cfg)
        ctx.sweep(2)
        ctx.synchronize()
        compare_traces(ctx.trace(0), oc.run(2 * k), 1e-10)
        for spin in (0, 1):
            No = oc.N(spin)
            np.testing.assert_allclose(ctx.get_N(0, spin), No, rtol=1e-9, atol=1e-10 * np.abs(No).max())


@pytest.mark.parametrize("K,n0,k", [(1.0, 130, 64), (256.0, 200, 160), (16.0, 257, 256)])
def test_sliced_flush_coefficients_in_the_lu_form(K, n0, k):
    """Y = (G - 1) Gamma^{-1} with Gamma kept as L U, at weak and strong e^V."""
    ch = configs.cube8(K=K, k_max=k, capacity=n0 + 2 * k + 64)
    cfg = configs.synthetic_configuration(ch, n0, seed=n0)
    oc = oracle_for(ch, p_insert=0.45, p_flip=0.1)
    oc.set_config(cfg["tau"], cfg["site"], cfg["s"], cfg["birth"], cfg["t"])
    with pk.Context([ch], trace_capacity=2 * k, refresh_every=0, p_insert=0.45, p_flip=0.1,
                    gamma_form=pk.ctaux.CTAUX_GAMMA_LU) as ctx:
        ctx.set_config(0, **cfg)
        tol = max(1e-10, 64 * 2.0**-52 * max(np.linalg.cond(oc.N(spin)) for spin in (0, 1)))
        ctx.sweep(2)
        ctx.synchronize()
        compare_traces(ctx.trace(0), oc.run(2 * k), tol)
        for spin in (0, 1):
            No = oc.N(spin)
            np.testing.assert_allclose(ctx.get_N(0, spin), No, rtol=tol, atol=tol * np.abs(No).max())

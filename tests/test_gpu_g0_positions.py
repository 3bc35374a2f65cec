"""Fixed-point table positions of the G0 interpolation at their edges.

Times that are equal, differ by less than a position unit, lie on a table
point, at 0 or just below beta, or meet a bin centre; the shortest tables and
one long enough to shorten the positions' fraction.  A position is within
2^-46 of a table step (the float64 position within 2^-42), so the tolerance is
that of the float64 parity tests, or 16 units in the last place times the
condition number of N where that is more (the coarse tables).
"""
import numpy as np
import pytest

from parity import compare_config, compare_traces, oracle_for
from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")


def edge_chain(n_tau, n, k):
    base = configs.cube8(K=64.0, k_max=k, capacity=n + 2 * k)
    grid = np.linspace(0.0, base.beta, base.n_tau)
    to = np.linspace(0.0, base.beta, n_tau)
    table = np.array([[np.interp(to, grid, row) for row in spin] for spin in base.table])
    ch = configs.dataclasses.replace(base, table=np.ascontiguousarray(table))
    cfg = configs.synthetic_configuration(ch, n, seed=n_tau)
    below = np.nextafter(ch.beta, 0.0)
    edges = [0.0, 1e-300, 5e-300, below, np.nextafter(below, 0.0), to[n_tau // 2] if n_tau > 2 else 0.5 * ch.beta,
             3.5 * ch.beta / 8, cfg["tau"][20], np.nextafter(cfg["tau"][21], 0.0)]
    cfg["tau"][:len(edges)] = edges
    cfg["site"][:len(edges)] = np.arange(len(edges)) % ch.n_c
    return ch, cfg


# n * k: panels of up to 4096 pairs, which the gather evaluates directly, and more
@pytest.mark.parametrize("n,k", [(90, 32), (700, 128)])
@pytest.mark.parametrize("n_tau", [2, 5, 1024, 131073])
def test_edge_times(n_tau, n, k):
    ch, cfg = edge_chain(n_tau, n, k)
    oc = oracle_for(ch)
    oc.set_config(cfg["tau"], cfg["site"], cfg["s"], cfg["birth"], cfg["t"])
    tol = max(1e-10, 16 * 2.0**-52 * max(np.linalg.cond(oc.N(spin)) for spin in (0, 1)))
    with pk.Context([ch], trace_capacity=k, refresh_every=0, n_tau_bins=8, n_anchors=1) as ctx:
        ctx.set_config(0, **cfg)
        for spin in (0, 1):
            No = oc.N(spin)
            np.testing.assert_allclose(ctx.get_N(0, spin), No, rtol=tol, atol=tol * np.abs(No).max())
        ctx.reset_measurements()
        ctx.sweep(1, measure=True)
        compare_traces(ctx.trace(0), oc.run(k), tol)
        compare_config(ctx, 0, oc)
        ref = oc.measure_G(8, 1)
        np.testing.assert_allclose(ctx.measure_G(0)[0], ref, rtol=tol, atol=tol * np.abs(ref).max())

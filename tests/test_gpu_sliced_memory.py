"""The sliced float64 products when a context is created with little memory left:
the images are made in smaller groups, and the results keep their bits."""
import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
pk = pytest.importorskip("paper_1010_3690_gb300")


def _free():
    return torch.cuda.mem_get_info()[0]


def _run(ch, cfg):
    before = _free()
    with pk.Context([ch], refresh_every=0, trace_capacity=3 * ch.k_max) as ctx:
        held = before - _free()
        ctx.set_config(0, **cfg)
        ctx.sweep(3)
        ctx.synchronize()
        return held, ctx.trace(0), ctx.get_N(0, 0), ctx.get_N(0, 1)


# bytes left beyond what the context takes when memory is plentiful: of the four images
# of N (39 MB each at this capacity) two, and one, fit in a quarter of what is left when
# they are allocated
@pytest.mark.parametrize("spare_mb", [256, 160])
def test_products_keep_their_bits_when_little_memory_is_left(spare_mb):
    ch = configs.cube8(K=256.0, k_max=64, capacity=1500)
    cfg = configs.synthetic_configuration(ch, 700, seed=5)
    held, *plenty = _run(ch, cfg)
    hold = torch.empty(_free() - held - spare_mb * 2 ** 20, dtype=torch.uint8, device="cuda")
    try:
        scarce = _run(ch, cfg)[1:]
    finally:
        del hold
        torch.cuda.empty_cache()
    for name in plenty[0].dtype.names:
        np.testing.assert_array_equal(scarce[0][name], plenty[0][name])
    np.testing.assert_array_equal(scarce[1], plenty[1])
    np.testing.assert_array_equal(scarce[2], plenty[2])

"""Reading N back: every column at its place for any leading dimension, nothing written
beside them, and no second copy of the matrix on the host."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

from workloads import configs

pytestmark = pytest.mark.gpu

pk = pytest.importorskip("paper_1010_3690_gb300")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _read(ctx, spin, n, pad):
    from paper_1010_3690_gb300 import ctaux
    out = np.full((n, n + pad), -7.0)          # column j in out[j, :n]
    m = C.c_int()
    code = ctaux.lib.ctaux_get_N(ctx.h, 0, spin, out.ctypes.data_as(C.POINTER(C.c_double)), n + pad, C.byref(m))
    assert code == 0 and m.value == n
    assert np.all(out[:, n:] == -7.0)
    return out[:, :n].T


@pytest.mark.parametrize("n", [1, 33, 1448, 1449, 2100])   # 8 MB hold all columns, all, and some
def test_columns_of_the_float32_form(n):
    ch = configs.cube8(K=256.0, k_max=8, capacity=max(64, n))
    cfg = configs.synthetic_configuration(ch, n, seed=n)
    with pk.Context([ch]) as ctx:
        ctx.set_config(0, **cfg)
        ref = [_read(ctx, spin, n, 3) for spin in (0, 1)]
    with pk.Context([ch], precision=pk.CTAUX_MIXED) as ctx:
        ctx.set_config(0, **cfg)
        for spin in (0, 1):
            # a recomputation runs in float64 in both forms: the same numbers, rounded once
            np.testing.assert_array_equal(_read(ctx, spin, n, 0), ref[spin].astype(np.float32).astype(np.float64))
            np.testing.assert_array_equal(_read(ctx, spin, n, 5), _read(ctx, spin, n, 0))


PROGRAM = """
import resource, sys
import numpy as np
import paper_1010_3690_gb300 as pk
from paper_1010_3690_gb300 import ctaux
from workloads import configs
import ctypes as C
n = 4000
ch = configs.cube8(K=256.0, k_max=8, capacity=n)
with pk.Context([ch], precision=pk.CTAUX_MIXED) as ctx:
    ctx.set_config(0, **configs.synthetic_configuration(ch, n, seed=1))
    out, m = np.ones((n, n)), C.c_int()
    ctx.get_config(0)
    before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
    assert ctaux.lib.ctaux_get_N(ctx.h, 0, 0, out.ctypes.data_as(C.POINTER(C.c_double)), n, C.byref(m)) == 0
    print(resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before)
"""


def test_no_second_matrix_on_the_host():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=200)
    assert r.returncode == 0, r.stderr[-500:]
    assert int(r.stdout.split()[-1]) * 1024 < 4000 * 4000 * 4 // 2

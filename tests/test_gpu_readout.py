"""Read-outs: a call that reports an error leaves the caller's arrays as they
were.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2402_04606_gb300 import workloads as wl
from tests.helpers import initial_fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_04606_gb300 import build

    build.build()


@pytest.mark.parametrize("call", ["fields", "populations"])
def test_error_leaves_the_arrays(call):
    from paper_2402_04606_gb300.native import ERR_TIMEOUT, OK, TUNE_SPIN_NS, Domain

    spec = wl.cylinder(D=10, levels=3, block=8, storage=wl.F32, re=100.0)
    g = Domain(spec)
    for l in range(spec.levels):
        g.set_fields(l, *initial_fields(spec, l))
    g.step(1)
    g.set_tuning(TUNE_SPIN_NS, 0)  # the first dependency not yet met stops the launch
    g.step(2)
    nx, ny = g.dims(0)
    out = np.full((9 if call == "populations" else 3, ny, nx), -7.0)
    rows = [p.ctypes.data_as(C.POINTER(C.c_double)) for p in out]
    args = [rows[0]] if call == "populations" else rows
    read = g.L.sbot_get_populations if call == "populations" else g.L.sbot_get_fields
    n = C.c_int64(out.size if call == "populations" else nx * ny)
    assert read(g.h, 0, *args, C.byref(n)) == ERR_TIMEOUT
    assert (out == -7.0).all()
    assert read(g.h, 0, *args, C.byref(n)) == OK and (out != -7.0).all()
    g.close()


@pytest.mark.parametrize("steps", [1, 700, 16000])  # 4, 2800 and 64000 entries: the last exceed the staging memory
def test_long_and_short_force_reads_agree(steps):
    from paper_2402_04606_gb300.native import Domain

    spec = wl.cylinder(D=10, levels=3, block=8, storage=wl.F32, re=100.0)
    whole, parts = [], []
    for parts_of, out in ((steps, whole), (max(1, steps // 7), parts)):
        g = Domain(spec)
        for l in range(spec.levels):
            g.set_fields(l, *initial_fields(spec, l))
        left = steps
        while left:
            n = min(left, parts_of)
            g.step(n)
            out.append(g.forces())
            left -= n
        assert g.forces().shape == (0, 3)
        g.close()
    a, b = np.concatenate(whole), np.concatenate(parts)
    assert a.shape == (4 * steps, 3) and np.array_equal(a, b) and np.abs(a[:, 0]).min() > 0

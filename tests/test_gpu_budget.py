"""Device memory that an instance or a context holds beside its populations:
the table of a solid's links is part of the admission budget, and is kept only
for the blocks at the solid's surface; the device buffer of a read-out is kept
only where the budget leaves room for it.
"""
import numpy as np
import pytest

from paper_2402_04606_gb300 import workloads as wl
from tests.helpers import init_oracle, oracle_from_spec
from tests.test_gpu_parity import TOL64, compare_populations, gpu_domain

pytestmark = pytest.mark.gpu

W, P = wl.BC_WALL, wl.BC_PERIODIC


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_04606_gb300 import build

    build.build()


def channel(nx, ny, block, storage, solid):
    """periodic in x, a moving wall above, the solid below or inside"""
    return wl.DomainSpec("channel", nx, ny, levels=1, block=block, bc=(P, P, W, W), tau_finest=0.7, storage=storage,
                         uwall=(0.0,) * 6 + (0.05, 0.01), solid=solid)


@pytest.mark.parametrize("persistent", [1, 0])
@pytest.mark.parametrize("solid", [(2, 40.3, 0.0, 0.0), (2, 43.3, 0.0, 0.0), (2, 47.6, 0.0, 0.0),
                                   (1, 32.2, 47.1, 24.0)])
def test_blocks_inside_a_solid_against_oracle(solid, persistent):
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT

    spec = channel(64, 96, 8, wl.F64, solid)
    o = init_oracle(oracle_from_spec(spec), spec)
    g = gpu_domain(spec)
    g.set_tuning(TUNE_PERSISTENT, persistent)
    before = g.populations(0)
    o.step(60)
    g.step(60)
    compare_populations(g, o, 1, TOL64)
    full = (g.types(0) == 4).reshape(12, 8, 8, 8).all(axis=(1, 3))
    assert full.any() and np.isfinite(before).all() and np.isfinite(g.populations(0)).all()


def test_solid_table_is_in_the_budget():
    from paper_2402_04606_gb300.native import ERR_OOM, Batch, SbotError

    def admitted_bytes(solid, budget=0):
        b = Batch(1, block=16, storage=wl.F32, budget_bytes=budget)
        try:
            b.admit(channel(256, 256, 16, wl.F32, solid))
            return b.info()["bytes"]
        finally:
            b.close()

    half = (2, 200.3, 0.0, 0.0)
    bytes_ = admitted_bytes(half)
    # the 16 blocks the surface crosses, 64 + 4 bytes per cell; the 192 blocks inside the solid need none
    assert bytes_ - admitted_bytes((0, 0.0, 0.0, 0.0)) == 16 * 256 * 68
    assert admitted_bytes(half, bytes_) == bytes_
    lists = 4 * (256 + 256 // 2 + 16)  # the interior list, which the admission check leaves out
    with pytest.raises(SbotError) as e:
        admitted_bytes(half, bytes_ - lists - 1)
    assert e.value.status == ERR_OOM


def test_kept_read_out_buffer_stays_inside_the_budget():
    import torch

    from paper_2402_04606_gb300.native import Batch

    spec = wl.tgv(n=1024, block=16, storage=wl.F32)
    buffer = 3 * 8 * 1024 * 1024  # what a read of its fields needs on the device
    one = Batch(1, block=16, storage=wl.F32)  # (also loads the kernels)
    i = one.admit(spec)
    want = i.fields(0)
    bytes_ = one.info()["bytes"]
    one.close()

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    b = Batch(1, block=16, storage=wl.F32, budget_bytes=bytes_ + buffer // 2)  # no room beside the instance
    i, before = b.admit(spec), free()
    got = i.fields(0)
    assert before - free() < buffer // 4
    b.close()
    b = Batch(2, block=16, storage=wl.F32, budget_bytes=2 * bytes_ + buffer // 2)  # room until the second one comes
    i = b.admit(spec)
    i.fields(0)
    j = b.admit(spec)
    again = j.fields(0)
    b.close()
    for x, y, z in zip(want, got, again):
        assert np.array_equal(x, y) and np.array_equal(x, z)

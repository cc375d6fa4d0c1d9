"""The largest bodies: the line by which they are admitted, just below it (run,
against the oracle or the graphs) and just above it (refused)."""
import dataclasses

import numpy as np
import pytest

from paper_2402_04606_gb300 import workloads as wl
from tests.helpers import init_oracle, oracle_from_spec
from tests.test_gpu_parity import TOL64, compare_forces, compare_populations, gpu_domain

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_04606_gb300 import build

    build.build()


def circle(a, n, storage):
    s = wl.cylinder(D=58, levels=1, block=8, storage=storage, n_markers=n, lx=4.0, ly=3.0, xc=1.5)
    return dataclasses.replace(s, body=dataclasses.replace(s.body, a=a, b=a))


def test_largest_body_fp64_against_oracle():
    spec = circle(29.0, 238, wl.F64)
    o = init_oracle(oracle_from_spec(spec), spec)
    g = gpu_domain(spec)
    o.step(6)
    g.step(6)
    compare_populations(g, o, 1, TOL64)
    compare_forces(g.forces(), o.forces(), spec.body.a)


def test_largest_body_fp32_in_both_step_forms():
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT

    res = []
    for persistent in (1, 0):
        g = gpu_domain(circle(48.5, 414, wl.F32))
        g.set_tuning(TUNE_PERSISTENT, persistent)
        g.step(6)
        res.append((g.populations(0), g.forces()))
        g.close()
    assert np.isfinite(res[0][1]).all()
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("a,n,storage", [(30.6, 238, wl.F64), (29.0, 239, wl.F64), (48.5, 415, wl.F32)])
def test_next_body_is_refused(a, n, storage):
    from paper_2402_04606_gb300.native import ERR_ARG, SbotError

    with pytest.raises(SbotError) as e:
        gpu_domain(circle(a, n, storage))
    assert e.value.status == ERR_ARG

"""The IBM inside the step: it collides the cells it forces itself, after the
sweep has written them unforced, and in the persistent kernel runs on thread
blocks of its own (IBM servers) where there are few enough bodies.

Each case is compared with the FP64 oracle, and the persistent kernel bit for
bit with the graphs (FP64, blocks of 8 or one cell per thread): one body and
many (more bodies than a quarter of the thread blocks: no servers), lists
longer than a thread's registers hold (markers closer than a cell), more
stencil cells than threads, and stencils on the inlet column's neighbours.
"""
import dataclasses

import numpy as np
import pytest

from paper_2402_04606_gb300 import workloads as wl
from tests.helpers import init_oracle, initial_fields, oracle_from_spec, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_04606_gb300 import build

    build.build()


def dense_markers():
    return wl.cylinder(D=10, levels=2, block=8, storage=wl.F64, n_markers=90)  # 0.35 cells apart: lists of up to 25


def many_cells():
    return wl.cylinder(D=56, levels=1, block=8, storage=wl.F64, n_markers=176, lx=3.0, ly=2.0, xc=1.0)


def near_inlet():
    s = wl.cylinder(D=10, levels=1, block=8, storage=wl.F64, n_markers=31, lx=6.0, ly=4.0)
    return dataclasses.replace(s, body=dataclasses.replace(s.body, x0=(8.0, s.ny0 / 2.0)))


def run(spec, persistent, steps):
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT, TUNE_VECTOR_MIN_CELLS, Domain

    g = Domain(spec)
    g.set_tuning(TUNE_PERSISTENT, persistent)
    g.set_tuning(TUNE_VECTOR_MIN_CELLS, -1)
    for l in range(spec.levels):
        g.set_fields(l, *initial_fields(spec, l))
    g.step(steps)
    out = [g.populations(l) for l in range(spec.levels)], g.forces()
    g.close()
    return out


@pytest.mark.parametrize("make", [dense_markers, many_cells, near_inlet])
def test_ibm_in_the_step_against_oracle_and_graphs(make):
    spec, steps = make(), 9
    pops, forces = run(spec, 1, steps)
    gp, gf = run(spec, 0, steps)
    for a, b in zip(pops, gp):
        assert np.array_equal(a, b)
    assert np.array_equal(forces, gf)
    o = init_oracle(oracle_from_spec(spec), spec)
    o.step(steps)
    for l in range(spec.levels):
        m = o.types(l) == 1
        assert rel_l2(pops[l][:, m], o.populations(l)[:, m]) <= 1e-12
    fo = o.forces()
    np.testing.assert_allclose(forces[:, :2], fo[:, :2], rtol=1e-10, atol=1e-11 * np.abs(fo[:, :2]).max())


@pytest.mark.parametrize("bodies", [3, 130])
def test_servers_and_more_bodies_than_servers(bodies):
    """a batch in the persistent kernel: every body equals itself in the graphs bit for bit"""
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT, Batch

    spec = wl.cylinder(D=10, levels=2, block=8, storage=wl.F32, n_markers=31, lx=14.0, ly=8.0, xc=4.0)
    res = []
    for persistent in (1, 0):
        b = Batch(bodies, block=8, storage=wl.F32)
        b.set_tuning(TUNE_PERSISTENT, persistent)
        members = [b.admit(dataclasses.replace(spec, tau_finest=0.56 + 0.001 * i)) for i in range(bodies)]
        b.step(9)
        res.append([(m.forces(), m.populations(1)) for m in members])
        b.close()
    for (fa, pa), (fb, pb) in zip(*res):
        assert np.array_equal(fa, fb) and np.array_equal(pa, pb)

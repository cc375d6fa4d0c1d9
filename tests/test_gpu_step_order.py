"""Sweeps beside the IBM of a static body: a sweep that pulls from, or
overwrites, the cells the IBM writes and pulls waits for it, wherever its
blocks lie.

Stencils whose last (or first) cell lies on a periodic side (the blocks across
the side pull the forced cells), in a corner of two periodic sides, and stencils
that reach the outermost interior cells of the finest level (the halo blocks
beside it stream from forced cells, and the coarse level merges them): the
persistent kernel equals the per-phase graphs bit for bit, and in FP64 both
equal the oracle to the parity tolerance.
"""
import numpy as np
import pytest

from paper_2402_04606_gb300 import workloads as wl
from tests.helpers import init_oracle, initial_fields, oracle_from_spec, rel_l2

pytestmark = pytest.mark.gpu

P = wl.BC_PERIODIC


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_04606_gb300 import build

    build.build()


def body(x0):
    return wl.BodySpec(a=5.0, b=5.0, n_markers=31, x0=x0)


def seam(x0, block, storage):
    """one level: a circle whose stencils end on a periodic side"""
    return wl.DomainSpec("seam", 64, 64, levels=1, block=block, bc=(P,) * 4, tau_finest=0.6, u_in=(0.05, 0.02),
                         storage=storage, body=body(x0))


def rim(x0, block, storage):
    """two levels, the finer one from cell 32 to 79 (blocks of 8) or 95 (of 16): a circle at its rim"""
    top = 79.0 if block == 8 else 95.0
    return wl.DomainSpec("rim", 64, 64, levels=2, block=block, bc=(P,) * 4, tau_finest=0.6, u_in=(0.05, 0.02),
                         storage=storage, boxes=[(1, 33.0, 33.0, top, top)], body=body(x0))


LAYOUTS = [(seam, (57.0, 32.0)), (seam, (32.0, 57.0)), (seam, (57.0, 57.0)), (seam, (7.6, 32.0)),
           (rim, (39.0, 56.0)), (rim, (56.0, 39.0)), (rim, (39.0, 39.0))]


def run(spec, persistent, steps, vec):
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT, TUNE_VECTOR_MIN_CELLS, Domain

    g = Domain(spec)
    g.set_tuning(TUNE_PERSISTENT, persistent)
    g.set_tuning(TUNE_VECTOR_MIN_CELLS, vec)
    for l in range(spec.levels):
        g.set_fields(l, *initial_fields(spec, l))
    g.step(steps)
    out = [g.populations(l) for l in range(spec.levels)], g.forces()
    g.close()
    return out


@pytest.mark.parametrize("block,storage,vec", [(8, wl.F64, -1), (8, wl.F32, -1), (16, wl.F64, 0), (16, wl.F32, 0)])
@pytest.mark.parametrize("make,x0", LAYOUTS)
def test_sweep_waits_for_the_ibm_whose_cells_it_touches(make, x0, block, storage, vec):
    spec, steps = make(x0, block, storage), 33
    pops, forces = run(spec, 1, steps, vec)
    gp, gf = run(spec, 0, steps, vec)
    for a, b in zip(pops, gp):
        assert np.array_equal(a, b)
    assert np.array_equal(forces, gf)
    if storage != wl.F64:
        return
    o = init_oracle(oracle_from_spec(spec), spec)
    o.step(steps)
    for l in range(spec.levels):
        m = o.types(l) == 1
        assert rel_l2(pops[l][:, m], o.populations(l)[:, m]) <= 1e-12
    fo = o.forces()
    np.testing.assert_allclose(forces[:, :2], fo[:, :2], rtol=1e-10, atol=1e-11 * np.abs(fo[:, :2]).max())


@pytest.mark.parametrize("threads,rounds,crit", [(768, 8, 1), (768, 8, 2), (256, 8, 1), (768, 1, 0), (256, 1, 0),
                                                 (768, 1, 2)])
@pytest.mark.parametrize("make", [
    lambda: wl.cylinder(D=10, levels=3, block=8, storage=wl.F32),                              # 50 level-0 blocks
    lambda: wl.cylinder(D=20, levels=2, block=16, storage=wl.F32, n_markers=63),               # 190
    lambda: wl.cylinder(D=40, levels=2, block=8, storage=wl.F32)], ids=["8 short", "16", "8 long"])  # 2850
def test_task_sizes_do_not_change_results(make, threads, rounds, crit):
    """a list that is cut differently in the first step (bulk tasks) and in the others, several steps per launch:
    each task sweeps its own blocks, whatever its thread block swept before under the same task number"""
    from paper_2402_04606_gb300 import native as nv

    spec, res = make(), []
    for knobs in ((threads, rounds, crit), (0, 8, 0)):
        g = nv.Domain(spec)
        g.set_tuning(nv.TUNE_VECTOR_MIN_CELLS, -1)
        for what, v in zip((nv.TUNE_STEP_THREADS, nv.TUNE_BULK_ROUNDS, nv.TUNE_CRIT_BLOCKS), knobs):
            g.set_tuning(what, v)
        for l in range(spec.levels):
            g.set_fields(l, *initial_fields(spec, l))
        g.step(64)
        res.append(([g.populations(l) for l in range(spec.levels)], g.forces()))
        g.close()
    for a, b in zip(res[0][0], res[1][0]):
        assert np.array_equal(a, b)
    assert np.array_equal(res[0][1], res[1][1])


def test_more_bodies_than_thread_blocks():
    """no thread block is set apart for a body, and every one may hold an IBM task that awaits a sweep: the sweep's
    tasks are taken first, so the step completes and equals the graphs"""
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT, Batch

    spec = wl.cylinder(D=10, levels=2, block=8, storage=wl.F32, n_markers=31, lx=14.0, ly=8.0, xc=4.0)
    n, res = 500, []  # at most 3 thread blocks on each of 152 SMs
    for persistent in (1, 0):
        b = Batch(n, block=8, storage=wl.F32)
        b.set_tuning(TUNE_PERSISTENT, persistent)
        members = [b.admit(spec) for _ in range(n)]
        b.step(40)
        res.append((members[0].populations(1), [m.forces() for m in members[::71]]))
        b.close()
    assert np.array_equal(res[0][0], res[1][0])
    for x, y in zip(res[0][1], res[1][1]):
        assert np.array_equal(x, y) and np.array_equal(x, res[0][1][0])


def wide_ellipse(storage):
    """140 cells long on blocks of 8: 18 blocks, more than the IBM's slot table has a side"""
    spec = wl.wing(c=140, levels=2, re=200.0, n_markers=230, block=8, domain_chords=3.0, storage=storage,
                   thickness=10.0 / 140.0, heave_chords=0.0)
    spec.body.motion = 0
    spec.body.alpha_mean = 0.0
    spec.margin = (0.0, 10.0) + (0.0,) * 6
    spec.retag = 0
    spec.init, spec.tgv_u0 = "tgv", 0.02
    return spec


def small_wing(storage):
    spec = wl.wing(c=16, levels=3, re=100.0, n_markers=50, block=8, domain_chords=8.0, storage=storage,
                   heave_chords=1.0)
    spec.body.period = 400.0
    spec.margin = (0.0, 14.0, 6.0) + (0.0,) * 5
    return spec


FORCED = {"wide": wide_ellipse, "wing": small_wing, "wing mrt": lambda st: wl.with_mrt(small_wing(st)),
          "wing les": lambda st: wl.with_les(small_wing(st)),
          "few cells": lambda st: wl.cylinder(D=10, levels=2, block=8, storage=st, n_markers=3)}


@pytest.mark.parametrize("storage", [wl.F64, wl.F32, wl.BF16DEV])
@pytest.mark.parametrize("name", list(FORCED))
def test_forced_cells_collided_apart(name, storage):
    """the collision of the cells a body forces: a launch of its own in the graphs, a phase of its own in FP64, by the
    IBM's thread block in the other storage kinds"""
    spec, steps = FORCED[name](storage), 20
    pops, forces = run(spec, 1, steps, -1)
    gp, gf = run(spec, 0, steps, -1)
    for a, b in zip(pops, gp):
        assert np.array_equal(a, b)
    assert np.array_equal(forces, gf)
    if storage != wl.F64:
        return
    o = init_oracle(oracle_from_spec(spec), spec)
    o.step(steps)
    for l in range(spec.levels):
        m = o.types(l) == 1
        assert rel_l2(pops[l][:, m], o.populations(l)[:, m]) <= 1e-12
    fo = o.forces()
    np.testing.assert_allclose(forces[:, :2], fo[:, :2], rtol=1e-10, atol=1e-11 * np.abs(fo[:, :2]).max())

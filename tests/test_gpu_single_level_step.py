"""Single-level instances in the persistent kernel: tasks with fixed owners,
sweeps cut into parts of a block, domain sides read from the task's copy of the
block's data, a solid's links from their table.

Equal bit for bit to the per-phase graphs (one cell per thread), which find the
sides through the instance's parameters, and to the FP64 oracle to rounding:
fewer blocks than thread blocks and more, every kind of side and moving walls on
each of them, a solid, a body, launches of one and of several steps.
"""
import numpy as np
import pytest

from paper_2402_04606_gb300 import workloads as wl
from tests.helpers import initial_fields, oracle_from_spec, rel_l2

pytestmark = pytest.mark.gpu

W, I, O, S, P = wl.BC_WALL, wl.BC_INLET, wl.BC_OUTLET, wl.BC_SYMMETRY, wl.BC_PERIODIC
UW = (0.0, 0.01, 0.0, -0.02, 0.03, 0.0, 0.05, 0.0)


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_04606_gb300 import build

    build.build()


def box(nx, ny, block, bc, storage=wl.F64, **kw):
    return wl.DomainSpec("box", nx, ny, levels=1, block=block, bc=bc, tau_finest=0.62, u_in=(0.04, 0.01), uwall=UW,
                         storage=storage, **kw)


CASES = {
    "periodic parts": box(48, 32, 16, (P,) * 4),
    "periodic many": box(200, 248, 8, (P,) * 4),  # 775 blocks: more than one per thread block's share
    "walls": box(64, 48, 16, (W,) * 4),
    "inlet outlet symmetry": box(64, 64, 8, (I, O, S, S)),
    "inlet on all": box(32, 32, 8, (I, I, I, O)),
    "walls y, periodic x": box(32, 96, 32, (P, P, W, W)),
    "symmetry, wall": box(40, 24, 8, (S, W, W, S), storage=wl.F32),
    "bounce cavity": wl.cavity(L=64, mode="bounce", storage=wl.F64),
    "bounce cavity 8": wl.cavity(L=72, mode="bounce", storage=wl.F32, block=8),
    "bounce cavity 16 bit": wl.cavity(L=64, mode="bounce", storage=wl.BF16DEV),
    "bounce cavity mrt": wl.with_mrt(wl.cavity(L=64, mode="bounce", storage=wl.F32)),
    "refined bounce cavity": wl.cavity(L=128, mode="bounce", storage=wl.F64, block=8, levels=2),
    "ibm cavity": wl.cavity(L=64, mode="ibm", storage=wl.F32),
}


def run(spec, persistent, steps):
    from paper_2402_04606_gb300.native import TUNE_PERSISTENT, TUNE_VECTOR_MIN_CELLS, Domain

    g = Domain(spec)
    g.set_tuning(TUNE_PERSISTENT, persistent)
    g.set_tuning(TUNE_VECTOR_MIN_CELLS, -1)
    for l in range(spec.levels):
        rho, ux, uy = initial_fields(spec, l)
        y = np.arange(rho.shape[0])[:, None] / rho.shape[0]
        g.set_fields(l, rho, ux + 0.01 * np.sin(2 * np.pi * y), uy)
    g.step(1)
    g.step(steps - 1)
    out = [g.populations(l) for l in range(spec.levels)], (g.forces() if spec.body is not None else None)
    g.close()
    return out


@pytest.mark.parametrize("name", list(CASES))
def test_single_level_step_equals_graphs_and_oracle(name):
    spec, steps = CASES[name], 19  # 1, then 8 + 8 + 1 + 1
    pops, forces = run(spec, 1, steps)
    gp, gf = run(spec, 0, steps)
    for a, b in zip(pops, gp):
        assert np.array_equal(a, b)
    if forces is not None:
        assert np.array_equal(forces, gf)
    if spec.storage != wl.F64:
        return
    o = oracle_from_spec(spec)
    for l in range(spec.levels):
        rho, ux, uy = initial_fields(spec, l)
        y = np.arange(rho.shape[0])[:, None] / rho.shape[0]
        o.set_fields(l, rho, ux + 0.01 * np.sin(2 * np.pi * y), uy + 0.0 * rho)
    o.finalize_init()
    o.step(steps)
    for l in range(spec.levels):
        m = o.types(l) == 1
        assert rel_l2(pops[l][:, m], o.populations(l)[:, m]) <= 1e-12

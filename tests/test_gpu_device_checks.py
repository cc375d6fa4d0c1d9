"""A check of the device code that no well-formed topology reaches, driven by a
small kernel of its own over hand-made tables: a block away from every domain
side whose neighbour is missing reports it, whatever the shared memory that
holds its data held before.
"""
import ctypes as C
import os
import subprocess

import pytest

from paper_2402_04606_gb300 import build as bld

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_device.cuh"
namespace {
__global__ void k_pull(DevPool P, const float* fin, float* out) {
    __shared__ SlotMeta<float> m;
    if (threadIdx.x < 4) m.kind[threadIdx.x] = BCK_OUTLET;  // what an earlier block on a side left there
    __syncthreads();
    load_meta<float>(P, 0, 0, m);
    __syncthreads();
    if (threadIdx.x == 0)
        out[0] = pull_int<float, float>(P, MetaS<float>{&m}, fin, (const float*)nullptr, false, P.inst[0], 0, 0, 3, 1);
}
template <class T>
T* up(const T* h, size_t n) {
    T* d = nullptr;
    if (cudaMalloc(&d, n * sizeof(T)) == cudaSuccess) cudaMemcpy(d, h, n * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}
}  // namespace
// one block of 8 x 8 cells, flags as given, every neighbour but itself missing: the pull of direction 1 into cell (0, 3)
extern "C" int pull_at_west_end(int flags, int bc_west, float* value, int* err) {
    int nbr[9] = {-1, -1, -1, -1, 0, -1, -1, -1, -1}, child[4] = {-1, -1, -1, -1};
    int zero = 0, type = ST_INT, parent = -1;
    unsigned mask[2] = {~0u, ~0u};
    InstParams ip{};
    ip.m = 1, ip.nx0 = ip.ny0 = 8, ip.tau[0] = 0.6, ip.rho0 = 1.0;
    for (int k = 0; k < 4; k++) ip.bc[k] = bc_west;
    float f[9 * 64];
    for (int i = 0; i < 9 * 64; i++) f[i] = 0.001f * i;
    DevPool P{};
    P.B = 8, P.mask_words = 2;
    P.nbr = up(nbr, 9), P.slot_inst = up(&zero, 1), P.slot_level = up(&zero, 1), P.slot_type = up(&type, 1);
    P.slot_ox = up(&zero, 1), P.slot_oy = up(&zero, 1), P.slot_flags = up(&flags, 1), P.slot_parent = up(&parent, 1);
    P.slot_child = up(child, 4), P.slot_mask = up(mask, 2), P.inst = up(&ip, 1), P.err = up(&zero, 1);
    const float none = -1.0f;
    float *fin = up(f, 9 * 64), *out = up(&none, 1);
    if (!P.nbr || !P.slot_inst || !P.slot_level || !P.slot_type || !P.slot_ox || !P.slot_oy || !P.slot_flags ||
        !P.slot_parent || !P.slot_child || !P.slot_mask || !P.inst || !P.err || !fin || !out)
        return 2;
    k_pull<<<1, 32>>>(P, fin, out);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    cudaMemcpy(value, out, sizeof(float), cudaMemcpyDeviceToHost);
    cudaMemcpy(err, P.err, sizeof(int), cudaMemcpyDeviceToHost);
    const void* all[] = {P.nbr, P.slot_inst, P.slot_level, P.slot_type, P.slot_ox, P.slot_oy, P.slot_flags,
                         P.slot_parent, P.slot_child, P.slot_mask, P.inst, P.err, fin, out};
    for (const void* p : all) cudaFree((void*)p);
    return 0;
}
extern "C" int edge_flag() { return SLOTF_EDGE; }
"""
ERRB_NOSOURCE, BCK_OUTLET = 4, 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("device_checks")
    src, so = d / "checks.cu", d / "checks.so"
    src.write_text(SOURCE)
    subprocess.check_call([bld.NVCC, *bld.ARCH, "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
                           "-I", bld.CSRC, "-I", os.path.join(bld.HERE, "..", "include"), "-o", str(so), str(src)])
    return C.CDLL(str(so))


def pull(lib, flags):
    v, e = C.c_float(), C.c_int()
    assert lib.pull_at_west_end(flags, BCK_OUTLET, C.byref(v), C.byref(e)) == 0
    return v.value, e.value


def test_missing_neighbour_away_from_the_sides_is_reported(lib):
    assert pull(lib, 0) == (0.0, ERRB_NOSOURCE)


def test_outlet_side_repeats_its_cell(lib):
    v, e = pull(lib, lib.edge_flag())
    assert e == 0 and v == pytest.approx(0.001 * (64 + 3 * 8))

"""Where glbm_moments lets its kernel write: the memory of the context's own GPU alone,
by what cudaPointerGetAttributes says of it (a small host program over the rule, no
GPU). On a GPU: managed memory, which takes the copy, and a captured call."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1905_04597_gb300 import build, glbm, inputs

PROGRAM = r"""
#include "glbm_internal.h"
#include <cstdio>
int main()
{
    const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost,
                                    cudaMemoryTypeDevice, cudaMemoryTypeManaged};
    for (cudaError_t e : {cudaSuccess, cudaErrorInvalidValue})
        for (cudaMemoryType t : types)
            for (int dev = 0; dev < 2; ++dev) {
                cudaPointerAttributes a = {};
                a.type = t;
                a.device = dev;
                std::printf("%d", glbm_kernel_may_write(e, a, 0) ? 1 : 0);
            }
    std::printf("\n");
}
"""


def test_rule(tmp_path):
    src = tmp_path / "rule.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "rule")
    subprocess.run([build._nvcc(), "-std=c++17", "-x", "c++", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.strip()
    # device memory of GPU 0 alone, and only when the query succeeded
    assert out == "00001000" + "00000000"


def _lattice():
    lat = glbm.Lattice(dict(dims=2, nx=70, ny=20, k=3, kn=0.1, prec=glbm.FP32_DEV, u_wall_lo=-0.05))
    lat.set_equilibrium(0, *inputs.random_macro(4, 70, 20))
    lat.step(3)
    return lat


@pytest.mark.gpu
def test_managed_memory():
    import __graft_entry__
    __graft_entry__.build_library()
    import torch
    torch.cuda.init()
    lat = _lattice()
    want = lat.moments(0)
    rt = ctypes.CDLL("/usr/local/cuda/lib64/libcudart.so")
    p = ctypes.c_void_p()
    n = 7 * 70 * 20
    assert rt.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(n * 8), ctypes.c_uint(1)) == 0
    glbm.check(glbm.lib().glbm_moments(lat.h, 0, glbm.M_ALL, p, n, 1))
    torch.cuda.synchronize()
    got = np.ctypeslib.as_array(ctypes.cast(p, ctypes.POINTER(ctypes.c_double)), (7, 20, 70)).copy()
    assert rt.cudaFree(p) == 0
    for i, name in enumerate(glbm.FIELDS_2D):
        np.testing.assert_array_equal(got[i], want[name])
    lat.close()


@pytest.mark.gpu
def test_captured_call():
    import __graft_entry__
    __graft_entry__.build_library()
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        lat = _lattice()
        want = lat.moments(0)
        out = torch.zeros((7, 20, 70), dtype=torch.float64, device="cuda")
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.moments(0, out=out)
        g.replay()
        s.synchronize()
    got = out.cpu().numpy()
    for i, name in enumerate(glbm.FIELDS_2D):
        np.testing.assert_array_equal(got[i], want[name])
    lat.close()

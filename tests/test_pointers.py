"""Which of a caller's arrays a kernel reads where they lie and which are copied first: the
decision on the CPU, and on a GPU the arrays that must go through a copy."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import paper_1410_0753_gb300 as pk
from paper_1410_0753_gb300 import CliffsGrid, _build

CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")


@pytest.fixture(scope="module")
def may_read(tmp_path_factory):
    d = tmp_path_factory.mktemp("pointers")
    src = d / "p.cpp"
    src.write_text('#include "pointers.h"\n'
                   'extern "C" int may_read(int type, int owner, int current, unsigned long long p, int size) {\n'
                   '  return cliffs::kernel_may_read((cudaMemoryType)type, owner, current, (const void*)p, size); }\n')
    so = str(d / "p.so")
    # the runtime calls of the header's other function stay unresolved: it is not instantiated
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-I", CUDA_INCLUDE, "-I", _build.CSRC, str(src), "-o", so],
                   check=True)
    return C.CDLL(so).may_read


UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3          # cudaMemoryType


@pytest.mark.parametrize("size", [4, 8])
@pytest.mark.parametrize("kind,owner,current,offset,want", [
    (DEVICE, 0, 0, 0, 1), (DEVICE, 3, 3, 0, 1),
    (DEVICE, 1, 0, 0, 0), (DEVICE, 0, 1, 0, 0),           # another GPU's memory
    (DEVICE, 0, 0, 2, 0), (DEVICE, 0, 0, 1, 0),           # not at a multiple of the element size
    (HOST, 0, 0, 0, 0), (UNREGISTERED, -2, 0, 0, 0), (MANAGED, 0, 0, 0, 0)])
def test_arrays_a_kernel_may_read(may_read, kind, owner, current, offset, want, size):
    assert may_read(kind, owner, current, C.c_ulonglong(0x7F0000000000 + offset), size) == want
    if kind == DEVICE and owner == current and offset == 0:
        assert may_read(kind, owner, current, C.c_ulonglong(0x7F0000000004), size) == (size == 4)


@pytest.mark.gpu
def test_device_arrays_off_their_element_size_are_copied():
    import torch
    nx, ny = 40, 33
    rng = np.random.default_rng(2)
    d = 10.0 * np.exp(rng.normal(0, 1.0, (ny, nx)))
    eta, u = (rng.normal(0, 0.1, (ny, nx)).astype(np.float32) for _ in range(2))

    def shifted(a, by):
        """a in device memory, `by` bytes past an aligned address"""
        raw = torch.zeros(a.nbytes + 16, dtype=torch.uint8, device="cuda")
        raw[by:by + a.nbytes] = torch.as_tensor(np.ascontiguousarray(a).view(np.uint8).reshape(-1), device="cuda")
        return raw, C.c_void_p(raw.data_ptr() + by)

    outs = []
    for by in (0, 4, 2):
        raw, p = shifted(d, by)
        out = torch.empty(ny, nx, dtype=torch.float64, device="cuda")
        n = C.c_int32()
        assert pk.lib().cliffs_depth_filter_noalloc(p, C.c_void_p(out.data_ptr()), nx, ny, 2.0, 0.1, None,
                                                    C.byref(n)) == 0
        g = CliffsGrid(nx, ny, 0.05)
        g.set_bathy(np.arange(nx) * 10.0, np.arange(ny) * 10.0, np.full((ny, nx), 20.0), False)
        (r1, pe), (r2, pu) = shifted(eta, by), shifted(u, by)
        assert pk.lib().cliffs_set_initial(g.h, 0, pe, pu, None, 0) == 0
        outs.append([n.value, out.cpu().numpy(), *g.state(), *g.maxwave()])
        g.close()
    assert np.array_equal(outs[0][2], eta) and np.array_equal(outs[0][3], u)
    for o in outs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(outs[0], o))

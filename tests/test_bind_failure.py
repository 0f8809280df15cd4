"""A bind whose kernel set-up fails leaves the context unbound (CPU: the host part of the library
linked with a CUDA runtime in host memory, its kernel entry points replaced by stubs)."""
import ctypes
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ESTATE, EFAIL = -7, -3

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
static const char* failing = "";
static int status(const char* name) { return *failing && std::strstr(name, failing) ? FAIL : 0; }
extern "C" {
void fail_in(const char* name) { failing = strdup(name); }
int cudaMalloc(void** p, size_t n) { *p = std::calloc(n ? n : 1, 1); return 0; }
int cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
int cudaFree(void* p) { std::free(p); return 0; }
int cudaFreeHost(void* p) { std::free(p); return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int) { std::memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { std::memcpy(d, s, n); return 0; }
int cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n, void*) { std::memset(d, v, n); return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
const char* cudaGetErrorString(int) { return "fake"; }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if shutil.which("g++") is None or shutil.which("nm") is None:
        pytest.skip("no host compiler")
    from paper_2410_17133_gb300 import _build
    _build.build()
    obj = os.path.join(_build.BUILD, "gm_host.o")
    text = subprocess.run(["nm", "-u", obj], capture_output=True, text=True, check=True).stdout
    names = set(re.findall(r"\bU (\S+)", text))
    here = set(re.findall(r"\b(cuda\w+)\(", RUNTIME))
    stubs = sorted(n for n in names if (n.startswith(("cuda", "__cuda")) and n not in here) or re.match(r"_Z\d+gm_", n))
    src = RUNTIME + "".join(f'long {n}() {{ return status("{n}"); }}\n' for n in stubs) + "}\n"
    d = tmp_path_factory.mktemp("host")
    (d / "runtime.cpp").write_text(src)
    so = str(d / "host.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-DFAIL=({EFAIL})", "-o", so, str(d / "runtime.cpp"), obj], check=True)
    return ctypes.CDLL(so)


def make(host):
    d3, vp = ctypes.c_double * 3, ctypes.c_void_p
    h = vp()
    host.fail_in(b"")
    assert host.gm_create(ctypes.byref(h), 0) == 0
    assert host.gm_mesh_structured(h, 2, 2, 2, d3(0, 0, 0), d3(1, 1, 1), (ctypes.c_double * 2)(0, 0)) == 0
    E, k = np.full(8, 1e9), np.full(8, 1e-15)
    host.gm_set_materials.argtypes = [vp, vp, vp, ctypes.c_int64] + [ctypes.c_double] * 4
    assert host.gm_set_materials(h, E.ctypes.data, k.ctypes.data, 8, 0.25, 0.8, 5e10, 1e-3) == 0
    return h


@pytest.mark.parametrize("step", ["gm_prepare_bulk32", "gm_prepare_fx", "gm_launch_diag", "gm_launch_block_jacobi"])
def test_failed_set_up_leaves_the_context_unbound(host, step):
    h = make(host)
    x = np.zeros(4 * 27)
    args = (h, 0, ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(x.ctypes.data), 0, None)
    host.fail_in(step.encode())
    assert host.gm_assemble_or_bind(h) == EFAIL
    assert host.gm_apply_operator(*args) == ESTATE
    host.fail_in(b"")
    assert host.gm_assemble_or_bind(h) == 0
    assert host.gm_apply_operator(*args) == 0

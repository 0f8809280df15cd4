"""Host paths of the tetrahedral library that a GPU does not take by itself (CPU: gm_tet.cu's host
part on a CUDA runtime in host memory whose kernels do nothing)."""
import ctypes
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
#include <map>
static std::map<void*, size_t> blocks;
static size_t used, limit = 1u << 30;
static int refused, device = 7, launches;
extern "C" {
void set_limit(size_t n) { limit = n; }
void refuse_cooperative(int r) { refused = r; }
size_t in_use() { return used; }
int launched() { return launches; }
int cudaMalloc(void** p, size_t n) {
    if (used + n > limit) return 2;
    *p = std::calloc(n, 1);
    blocks[*p] = n;
    used += n;
    return 0;
}
int cudaFree(void* p) {
    if (p) used -= blocks[p];
    blocks.erase(p);
    std::free(p);
    return 0;
}
// kernels do nothing, so what comes back is made up: a solve done in one iteration (its state of
// six doubles and four ints, or done and its count alone), sums of zero, 15 neighbours per node
static void copy(void* d, const void* s, size_t n, int kind) {
    if (kind != 2) { std::memcpy(d, s, n); return; }
    std::memset(d, 0, n);
    int* v = static_cast<int*>(d);
    if (n == 8 || n == 64) { v += n == 64 ? 12 : 0; v[0] = v[1] = 1; }
    else for (size_t i = 0; i < n / 4 && n < 2048; ++i) v[i] = 15;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { copy(d, s, n, kind); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void*) { copy(d, s, n, kind); return 0; }
int cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = limit - used; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return 0; }
int cudaStreamIsCapturing(void* s, int* c) { *c = s == (void*)8; return 0; }     // stream 8 captures
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaSetDevice(int d) { device = d; return 0; }
int cudaLaunchCooperativeKernel() { return refused ? 720 : 0; }
int cudaGraphLaunch() { ++launches; return 0; }
const char* cudaGetErrorString(int) { return "fake"; }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if shutil.which("g++") is None or shutil.which("nm") is None:
        pytest.skip("no host compiler")
    from paper_2410_17133_gb300 import _build
    _build.build()
    obj = os.path.join(_build.BUILD, "gm_tet.o")
    text = subprocess.run(["nm", "-u", obj], capture_output=True, text=True, check=True).stdout
    here = set(re.findall(r"\b(cuda\w+)\(", RUNTIME))
    stubs = sorted(n for n in re.findall(r"\bU ((?:__)?cuda\w+)", text) if n not in here)
    src = RUNTIME + "".join(f"long {n}() {{ return 0; }}\n" for n in stubs) + "}\n"
    d = tmp_path_factory.mktemp("tet")
    (d / "runtime.cpp").write_text(src)
    so = str(d / "tet.so")
    subprocess.run(["g++", "-O1", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", so, str(d / "runtime.cpp"), obj],
                   check=True)
    L = ctypes.CDLL(so)
    L.in_use.restype = ctypes.c_size_t
    L.set_limit.argtypes = [ctypes.c_size_t]
    L.gm_tet_materials.argtypes = [ctypes.c_void_p] + [ctypes.c_double] * 6
    L.gm_tet_step.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double,
                              ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    return L


class Tet:
    """One tetrahedron per four nodes, resting on its first three."""

    def __init__(self, L, n=1):
        self.L, self.n = L, n
        self.h = ctypes.c_void_p()
        L.set_limit(1 << 30)
        L.refuse_cooperative(0)
        assert L.gm_tet_create(ctypes.byref(self.h), 0) == 0
        x = np.tile(np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], float), (n, 1))
        e = np.arange(4 * n, dtype=np.int64)
        assert L.gm_tet_mesh(self.h, x.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(4 * n),
                             e.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(n)) == 0

    def materials(self, E=1e9):
        return self.L.gm_tet_materials(self.h, E, 0.25, 0.8, 5e10, 1e-15, 1e-3)

    def step(self):
        u, p = np.zeros(12 * self.n), np.zeros(4 * self.n)
        return self.L.gm_tet_step(self.h, 1.0, u.ctypes.data, p.ctypes.data, 1e-10, 50, None, None)


def test_a_refused_cooperative_launch_leaves_the_solve_to_the_launches(host):
    t = Tet(host)
    assert t.materials() == 0
    n0 = host.launched()
    assert t.step() == 0
    n1 = host.launched()
    host.refuse_cooperative(1)
    assert t.step() == 0
    assert n1 == n0 and host.launched() > n1            # one launch first, captured iterations then


def test_rows_make_room_for_the_vectors_of_a_step(host):
    """With a byte less than rows and vectors take together, the step still has its vectors."""
    start = host.in_use()
    t = Tet(host, 2)
    assert t.materials() == 0 and t.step() == 0
    whole = host.in_use() - start
    host.gm_tet_destroy(t.h)
    assert host.in_use() == start
    t = Tet(host, 2)
    host.set_limit(start + whole - 1)
    assert t.materials() == 0
    with_rows = host.in_use()
    assert t.step() == 0 and t.step() == 0
    rows = 15 * 8 * 208                                     # 15 entries at 8 nodes
    assert with_rows - start > rows and host.in_use() - start < whole - rows
    assert t.materials(2e9) == 0 and t.step() == 0
    host.gm_tet_destroy(t.h)
    assert host.in_use() == start


def test_rows_that_a_captured_product_holds_stay(host):
    """The same, after a product was captured: the step reports the missing memory, and the rows that
    the caller's graph reads stay until the next mesh."""
    start = host.in_use()
    t = Tet(host, 2)
    assert t.materials() == 0
    with_rows = host.in_use()
    x = np.zeros(4 * 8)
    p = ctypes.c_void_p(x.ctypes.data)
    assert host.gm_tet_apply(t.h, 0, p, p, ctypes.c_double(1.0), 0, ctypes.c_void_p(8)) == 0
    host.set_limit(with_rows + 4096)
    assert t.step() == -2 and host.in_use() >= with_rows
    host.set_limit(1 << 30)
    assert t.step() == 0
    host.gm_tet_destroy(t.h)
    assert host.in_use() == start


def test_materials_leave_the_device_of_the_caller(host):
    t = Tet(host)
    host.cudaSetDevice(5)
    assert t.materials() == 0
    d = ctypes.c_int()
    host.cudaGetDevice(ctypes.byref(d))
    assert d.value == 5

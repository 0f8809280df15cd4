"""Two solvers whose multigrid is set up at the same time take the same route on the coarsest level
(CPU: the host parts of the library on a CUDA runtime in host memory)."""
import ctypes
import os
import re
import shutil
import subprocess
import threading

import numpy as np
import pytest

from test_bind_failure import RUNTIME

QUERY = r"""
#include <atomic>
#include <chrono>
#include <thread>
static std::atomic<int> inside{0}, done{0};
extern "C" {
int asked() { return inside; }
void finished() { done = 1; }
// the first query lasts until the other thread is through, or half a second
int cudaOccupancyMaxActiveClusters(int* n, const void*, const void*) {
    if (inside.exchange(1) == 0)
        for (int i = 0; i < 500 && !done; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    *n = 1;
    return 0;
}
int cudaStreamIsCapturing(void*, int* s) { *s = 0; return 0; }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if shutil.which("g++") is None or shutil.which("nm") is None:
        pytest.skip("no host compiler")
    from paper_2410_17133_gb300 import _build
    _build.build()
    objs = [os.path.join(_build.BUILD, o) for o in ("gm_host.o", "gm_mg.o")]
    nm = lambda flag: set(re.findall(r"\b[UTWV] (\S+)", subprocess.run(
        ["nm", flag] + objs, capture_output=True, text=True, check=True).stdout))
    names = nm("-u") - nm("--defined-only")
    here = set(re.findall(r"\b(cuda\w+)\(", RUNTIME + QUERY))
    stubs = sorted(n for n in names if (n.startswith(("cuda", "__cuda")) and n not in here) or re.match(r"_Z\d+gm_", n))
    src = RUNTIME + "}\n" + QUERY + "".join(f'long {n}() {{ return status("{n}"); }}\n' for n in stubs) + "}\n"
    d = tmp_path_factory.mktemp("mg")
    (d / "runtime.cpp").write_text(src)
    so = str(d / "mg.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-DFAIL=(-3)", "-o", so,
                    str(d / "runtime.cpp")] + objs, check=True)
    return ctypes.CDLL(so)


def solver(L, n=8):
    d3, vp = ctypes.c_double * 3, ctypes.c_void_p
    h = vp()
    assert L.gm_create(ctypes.byref(h), 0) == 0
    assert L.gm_mesh_structured(h, n, n, n, d3(0, 0, 0), d3(1, 1, 1), (ctypes.c_double * 2)(0, 0)) == 0
    E, k = np.full(n ** 3, 1e9), np.full(n ** 3, 1e-15)
    L.gm_set_materials.argtypes = [vp, vp, vp, ctypes.c_int64] + [ctypes.c_double] * 4
    assert L.gm_set_materials(h, E.ctypes.data, k.ctypes.data, n ** 3, 0.25, 0.8, 5e10, 1e-3) == 0
    assert L.gm_assemble_or_bind(h) == 0
    return h


def cycle_launches(L, h):
    x = np.zeros(3 * 9 ** 3)
    p = ctypes.c_void_p(x.ctypes.data)
    n = [ctypes.c_int64(), ctypes.c_int64()]
    L.gm_counters(h, ctypes.byref(n[0]), None)
    assert L._Z12gm_mg_vcycleP6gm_ctxiPKvPvPKiP11CUstream_st(h, 1, p, p, None, None) == 0
    L.gm_counters(h, ctypes.byref(n[1]), None)
    return n[1].value - n[0].value


def test_two_set_ups_at_a_time_take_the_same_route(host):
    a, b = solver(host), solver(host)
    prepare = host._Z13gm_mg_prepareP6gm_ctxiP11CUstream_st
    rc = []
    t = threading.Thread(target=lambda: rc.append(prepare(a, 1, None)))
    t.start()
    while not host.asked():
        assert t.is_alive()
    rc.append(prepare(b, 1, None))
    host.finished()
    t.join()
    assert rc == [0, 0]
    assert cycle_launches(host, a) == cycle_launches(host, b) < 40      # the polynomial is one of them

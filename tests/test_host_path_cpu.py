"""The library's host path on a machine of several GPUs, without one: its
objects linked against a stand-in for the CUDA runtime whose memory is host
memory and whose kernels do nothing.  It keeps the attributes of each device's
kernels, refuses a launch that asks for more dynamic shared memory than they
allow, as the runtime does, and lists what was launched."""
import glob
import os
import shutil
import subprocess
import sys

import pytest

from paper_2404_04994_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#define API extern "C" __attribute__((visibility("default")))
struct dim3 { unsigned x, y, z; };
static int dev = 0, last = 0;
static std::map<std::pair<int, const void*>, int> limit;  // dynamic shared memory
static dim3 grid, block;
static size_t smem;
static void* stream;
static int fail(int e) { return last = e; }
static std::map<const void*, std::string>& names() {  // filled while the library loads
  static auto* m = new std::map<const void*, std::string>;
  return *m;
}
static std::string& log_ = *new std::string;
API const char* launched() {
  static std::string s;
  s.swap(log_);
  log_.clear();
  return s.c_str();
}
static int launch(const void* f, size_t bytes) {
  log_ += names()[f] + " ";
  auto it = limit.find({dev, f});
  return bytes > (it == limit.end() ? 48 * 1024 : (size_t)it->second) ? fail(1) : 0;
}
API int cudaGetDevice(int* d) { *d = dev; return 0; }
API int cudaSetDevice(int d) { dev = d; return 0; }
API int cudaFuncSetAttribute(const void* f, int attr, int v) {
  if (attr == 8) limit[{dev, f}] = v;
  return 0;
}
API unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) {
  grid = g; block = b; smem = s; stream = st;
  return 0;
}
API int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = grid; *b = block; *s = smem; *(void**)st = stream;
  return 0;
}
API int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
API int __cudaLaunchKernel(void* k, dim3, dim3, void**, size_t s, void*) { return launch(k, s); }
struct Config { dim3 g, b; size_t s; };
API int cudaLaunchKernelExC(const Config* c, const void* f, void**) {
  log_ += "overlapped:";
  return launch(f, c->s);
}
API int cudaGetLastError() { int e = last; last = 0; return e; }
API const char* cudaGetErrorString(int) { return "error"; }
API int cudaMalloc(void** p, size_t n) { *p = calloc(n, 1); return 0; }
API int cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(n, 1); return 0; }
API int cudaFree(void* p) { free(p); return 0; }
API int cudaFreeHost(void* p) { free(p); return 0; }
API int cudaMemcpy(void* d, const void* s, size_t n, int) { memcpy(d, s, n); return 0; }
API int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { memcpy(d, s, n); return 0; }
API int cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return 0; }
API int cudaMemsetAsync(void* d, int v, size_t n, void*) { memset(d, v, n); return 0; }
API int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
API int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                               unsigned) { *n = 1; return 0; }
API int cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return 0; }
API int cudaDeviceSynchronize() { return 0; }
API int cudaStreamSynchronize(void*) { return 0; }
API int cudaStreamIsCapturing(void*, int* status) { *status = 0; return 0; }
API int cudaEventCreate(void** e) { *e = &dev; return 0; }
API int cudaEventCreateWithFlags(void** e, unsigned) { *e = &dev; return 0; }
API int cudaEventDestroy(void*) { return 0; }
API int cudaEventRecord(void*, void*) { log_ += "event "; return 0; }
API int cudaEventSynchronize(void*) { return 0; }
API int cudaEventElapsedTime(float* t, void*, void*) { *t = 0.f; return 0; }
API void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
API void __cudaRegisterFatBinaryEnd(void**) {}
API void __cudaUnregisterFatBinary(void**) {}
API void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*,
                                void*, void*, int*) { names()[f] = name; }
API void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    gxx = shutil.which("g++")
    if gxx is None or not objs or build.stale():
        pytest.skip("needs g++ and the objects of an up-to-date build")
    d = tmp_path_factory.mktemp("host_path")
    (d / "runtime.cpp").write_text(RUNTIME)
    lib = str(d / "libqarray_host.so")
    subprocess.check_call([gxx, "-std=c++17", "-shared", "-fPIC", "-o", lib, *objs,
                           str(d / "runtime.cpp")])
    return lib


def _run(library, code):
    env = dict(os.environ, QARRAY_LIB=library, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", code], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split()


@pytest.mark.parametrize("n", [8, 12, 13, 16])
def test_soft_calls_on_each_device(library, n):
    # the backward of 13 to 16 dots needs more than the default limit, on
    # whichever device it runs
    out = _run(library, f"""
import ctypes
import numpy as np
from paper_2404_04994_gb300 import api, inputs
lib, n = api.load(), {n}
r = np.random.Generator(np.random.PCG64(2))
Cdd, Cgd = inputs.chain_cdd(r, n), inputs.dense_cgd(r, n)
ras = api.make_raster(inputs.raster(n, 0, 1, np.ones(n), W=8, H=4), n)
g, d = np.ones((32, n), dtype=np.float32), np.zeros((n, n))
for dev in (0, 1, 0):
    lib.cudaSetDevice(dev)
    m = api.qa_model_create(Cdd, Cgd)
    for rc in (lib.qa_soft_occupation(m, ctypes.byref(ras), 0.05, 1.0, 0, 0, g.ctypes.data, None,
                                      None),
               lib.qa_soft_occupation_backward(m, ctypes.byref(ras), 0.05, 1.0, 0, 0,
                                               g.ctypes.data, d.ctypes.data, d.ctypes.data, None),
               lib.qa_soft_occupation_backward(m, ctypes.byref(ras), 0.05, 1.0, 1, n,
                                               g.ctypes.data, d.ctypes.data, d.ctypes.data, None)):
        print(rc)
    api.qa_model_destroy(m)
""")
    assert out == ["0"] * 9


@pytest.mark.parametrize("team", [0, 1, 4, 8, 32])
def test_batch_item_team_is_the_tile_search(library, team):
    # lanes asked for are lanes of the search by tiles; the library's own
    # choice is a one-pass kernel for arrays of 3 dots and more
    out = _run(library, f"""
import ctypes
import numpy as np
from paper_2404_04994_gb300 import api, inputs
lib = api.load()
lib.launched.restype = ctypes.c_char_p
for n in (3, 5, 8, 11, 12, 16):
    for closed in (0, 1):
        for t in (0.5, 1.0):
            r = np.random.Generator(np.random.PCG64(2))
            item = api.qa_batch_item()
            m = api.qa_model_create(inputs.chain_cdd(r, n), inputs.dense_cgd(r, n))
            out = np.zeros((32, n), dtype=np.int8)
            item.model, item.out_n = m.value, out.ctypes.data
            ras = api.make_raster(inputs.raster(n, 0, 1, np.ones(n), W=8, H=4), n)
            item.raster, item.threshold, item.closed, item.n_charges = ras, t, closed, n
            item.team = {team}
            b = ctypes.c_void_p()
            assert lib.qa_batch_create(ctypes.byref(item), 1, ctypes.byref(b)) == 0
            assert lib.qa_batch_run(b, None) == 0
            names = lib.launched().decode()
            print(int("k_pixels_batch" in names), int("k_search_batch" in names))
""")
    pairs = set(zip(out[::2], out[1::2]))
    assert pairs == {("0", "1")} if team else ("1", "0") in pairs


@pytest.mark.parametrize("n,t,closed,kernel,shape", [
    (2, 1.0, 0, "k_ground_state", (1, 2, 0)), (3, 1.0, 1, "k_pixels", (4, 2, 0)),
    (4, 0.5, 0, "k_pixels", (4, 2, 0)), (8, 1.0, 0, "k_pixels", (8, 4, 0)),
    (9, 0.5, 1, "k_pixels", (16, 4, 0)), (16, 0.5, 0, "k_pixels", (16, 4, 0)),
    (16, 1.0, 1, "k_pixels", (16, 0, 0)), (16, 1.0, 0, "k_pixels", (16, 0, 0))])
def test_stats_describe_the_search_that_ran(library, n, t, closed, kernel, shape):
    # lanes and slots of the kernel of the call, and its time as the search's:
    # the kernel lies between the second and the third of four events
    out = _run(library, f"""
import ctypes
import numpy as np
from paper_2404_04994_gb300 import api, inputs
lib, n = api.load(), {n}
lib.launched.restype = ctypes.c_char_p
r = np.random.Generator(np.random.PCG64(2))
m = api.qa_model_create(inputs.chain_cdd(r, n), inputs.dense_cgd(r, n))
api.qa_model_set_timing(m, True)
ras = api.make_raster(inputs.raster(n, 0, 1, np.ones(n), W=300, H=200), n)
out = np.zeros((60000, n), dtype=np.int8)
if {closed}:
    rc = lib.qa_ground_state_closed(m, ctypes.byref(ras), {t}, n, out.ctypes.data, None, None, None)
else:
    rc = lib.qa_ground_state_open(m, ctypes.byref(ras), {t}, out.ctypes.data, None, None, None)
s = api.qa_model_stats(m, 0)
print(rc, s["team"], s["inner_bits"], s["middle_bits"], lib.launched().decode())
""")
    assert tuple(int(v) for v in out[:4]) == (0, *shape)
    chain = out[4:]
    assert [i for i, v in enumerate(chain) if v == "event"] == [0, 1, 3, 5]
    assert kernel in chain[2] and "k_lists" in chain[4]


def test_grids_of_a_batch_overlap(library):
    # arrays of every kind: after the prep and the first search grid, which
    # waits for it, each grid may start while the one before runs
    out = _run(library, """
import ctypes
import numpy as np
from paper_2404_04994_gb300 import api, inputs
lib = api.load()
lib.launched.restype = ctypes.c_char_p
kinds = [(n, c, t) for n in (2, 3, 8, 9, 11, 12, 16) for c in (0, 1) for t in (0.5, 1.0)]
items, keep = (api.qa_batch_item * len(kinds))(), []
for it, (n, closed, t) in zip(items, kinds):
    r = np.random.Generator(np.random.PCG64(2))
    m = api.qa_model_create(inputs.chain_cdd(r, n), inputs.dense_cgd(r, n))
    out = np.zeros((32, n), dtype=np.int8)
    ras = api.make_raster(inputs.raster(n, 0, 1, np.ones(n), W=8, H=4), n)
    keep += [m, out, ras]
    it.model, it.out_n, it.raster = m.value, out.ctypes.data, ras
    it.threshold, it.closed, it.n_charges = t, closed, n
b = ctypes.c_void_p()
assert lib.qa_batch_create(items, len(kinds), ctypes.byref(b)) == 0
assert lib.qa_batch_run(b, None) == 0
print(lib.launched().decode())
""")
    assert "k_prep_batch" in out[0] and "k_lists" in out[-1]
    assert sum("k_pixels_batch" in v for v in out) >= 8
    assert [v.startswith("overlapped:") for v in out] == [False, False] + [True] * (len(out) - 2)


def test_a_small_raster_of_many_dots_takes_tiles(library):
    # one-pass searches leave close pixels to the list kernel, which an open
    # raster of 64 to 4863 pixels does not hide
    out = _run(library, """
import ctypes
import numpy as np
from paper_2404_04994_gb300 import api, inputs
lib = api.load()
lib.launched.restype = ctypes.c_char_p
for n, closed, t, W in ((14, 0, 1.0, 63), (14, 0, 1.0, 64), (14, 0, 1.0, 4863), (14, 0, 1.0, 4864),
                        (14, 1, 1.0, 64), (14, 1, 1.0, 4863),
                        (16, 0, 1.0, 600), (16, 1, 1.0, 600), (13, 0, 0.25, 600), (13, 0, 0.4, 600),
                        (12, 1, 0.0, 999), (12, 1, 0.0, 9999), (13, 1, 0.0, 9999), (10, 0, 1.0, 4863),
                        (10, 0, 1.0, 4864), (9, 0, 1.0, 99999)):
    r = np.random.Generator(np.random.PCG64(2))
    m = api.qa_model_create(inputs.chain_cdd(r, n), inputs.dense_cgd(r, n))
    ras = api.make_raster(inputs.raster(n, 0, 1, np.ones(n), W=W, H=1), n)
    out = np.zeros((W, n), dtype=np.int8)
    if closed:
        lib.qa_ground_state_closed(m, ctypes.byref(ras), t, n, out.ctypes.data, None, None, None)
    else:
        lib.qa_ground_state_open(m, ctypes.byref(ras), t, out.ctypes.data, None, None, None)
    print(int("k_pixels" in lib.launched().decode()))
""")
    assert "".join(out) == "1001" + "11" + "11" + "10" + "101" + "10" + "1"

"""A call that fails between the sort and the leaf scan (a launch that returns
an error) leaves the sort's state as it is; the next call of the context clears
it before it sorts, and no later one does.  The host code is linked against
launch functions and a CUDA runtime that only record their names, so this
needs no GPU."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1709_04488_gb300 import build as B
from paper_1709_04488_gb300 import sph

FAKE = r"""
#include <cstdio>
#include <cstring>
#include <string>
static std::string g_trace, g_fail;
static int hit(const char *name)
{
    g_trace += std::string(name) + "\n";
    return g_fail == name ? 999 : 0;
}
extern "C" const char *fake_trace() { return g_trace.c_str(); }
extern "C" void fake_reset(const char *fail) { g_trace.clear(); g_fail = fail; }

struct CUstream_st;
namespace sph {
struct BatchView;
typedef const BatchView &V;
typedef CUstream_st *S;
typedef unsigned long long H;
long long leaf_tiles(long long n) { return n / 256 + 1; }
long long sort_words(int, long long n) { return 4096 + n; }
long long leaves_upper_bound(long long n) { return n; }
long long gravity_blocks(long long, double) { return 0; }
int gravity_chunks(long long, double) { return 0; }
#define F(name, ...) int name(__VA_ARGS__) { return hit(#name); }
F(launch_refit, V, S) F(launch_forces, V, int, S) F(launch_gather, V, S) F(launch_density, V, int, int, S)
F(launch_block_dt, V, int, S) F(launch_block_open, V, int, S) F(launch_block_gate, V, int, bool, H, H, S)
F(launch_block_kick, V, int, bool, H, H, S) F(launch_kick_close, V, int, int, S) F(launch_kick_drift, V, double, S)
F(launch_radix_sort, V, S) F(launch_reset_step, V, int, S) F(launch_block_drift, V, S) F(launch_block_tasks, V, int, S)
F(launch_block_finish, V, S) F(launch_block_gather, V, int, S) F(launch_build_leaves, V, int, bool, S)
F(launch_set_sorted_h, V, int, const double *, S) F(launch_update_leaves, V, int, S) F(launch_block_leaf_tick, V, int, S)
F(launch_domain_and_keys, V, S) F(launch_block_tick_begin, V, int, H, S)
F(launch_neighbour_export, V, int, bool, int, long long *, int *, long long, S)
void launch_gravity(V, int, S) { hit("launch_gravity"); }
}
extern "C" {
int cudaMemsetAsync(void *p, int v, size_t n, void *)
{
    char t[96];
    snprintf(t, sizeof t, "memset %p %d %zu", p, v, n);
    return hit(t);
}
static char g_handle;
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *)
{
    // (the flags of a block step: one loop tick, then the last)
    static int tick = 0;
    if (k == 2 && n == 24) {
        ((long long *)d)[0] = tick == 0;
        ((long long *)d)[2] = 1;
        tick = !tick;
    }
    return 0;
}
int cudaMemcpy(void *, const void *, size_t, int) { return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int, int) { *v = 152; return 0; }
const char *cudaGetErrorString(int) { return "fake"; }
int cudaGetLastError() { return 0; }
int cudaGraphInstantiate(void **g, void *, unsigned long long) { *g = &g_handle; return hit("instantiate"); }
int cudaGraphLaunch(void *, void *) { return hit("graph"); }
int cudaGraphGetNodes(void *, void *, size_t *n) { *n = 0; return 0; }
int cudaStreamEndCapture(void *, void **g) { *g = nullptr; return 0; }
#define N(name) int name(...) { return 0; }
N(cudaEventCreate) N(cudaEventDestroy) N(cudaEventElapsedTime) N(cudaEventRecord) N(cudaEventRecordWithFlags)
N(cudaGraphAddNode) N(cudaGraphConditionalHandleCreate) N(cudaGraphDestroy) N(cudaGraphExecDestroy)
N(cudaGraphNodeGetType) N(cudaStreamBeginCapture) N(cudaStreamBeginCaptureToGraph) N(cudaStreamCreateWithFlags)
N(cudaStreamDestroy) N(cudaStreamGetCaptureInfo) N(cudaStreamIsCapturing) N(cudaStreamSynchronize)
N(cudaStreamUpdateCaptureDependencies) N(__cudaRegisterFatBinary) N(__cudaRegisterFatBinaryEnd)
N(__cudaUnregisterFatBinary)
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    B.build()
    d = tmp_path_factory.mktemp("fake")
    src, so = d / "fake.cpp", d / "fake.so"
    src.write_text(FAKE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-w", str(src), os.path.join(B.BUILD, "sph_api.o"),
                    "-Wl,-z,defs", "-Wl,-Bsymbolic", "-o", str(so)], check=True, capture_output=True, text=True)
    lib = C.CDLL(str(so))
    lib.fake_trace.restype = C.c_char_p
    return lib


def _trace(L):
    return L.fake_trace().decode().split("\n")


def _context(L, stream, **kw):
    p = sph.Params()
    L.sph_params_default(C.byref(p))
    for k, v in kw.items():
        setattr(p, k, v)
    n, at = 1000, C.c_void_p(1 << 20)
    st = sph.State(**{f: 1 << 20 for f in sph.STATE_FIELDS})
    ctx = C.c_void_p()
    L.fake_reset(b"")
    assert L.sph_setup(C.byref(ctx), C.byref(p), C.c_int64(n), C.byref(st), at, C.c_size_t(1 << 40), C.c_void_p(stream)) == sph.OK
    # the last region the set-up clears that is not a per-particle array
    zero = [t for t in _trace(L) if t.startswith("memset")][2]
    return ctx, zero


CALLS = {
    "density": (0, {}, lambda L, c: L.sph_density_h(c)),
    "step": (0, {}, lambda L, c: L.sph_step(c, C.c_double(1e-3), None)),
    "step, kept leaves": (0, dict(tree_rebuild_every=4), lambda L, c: L.sph_step(c, C.c_double(1e-3), None)),
    "run": (0, {}, lambda L, c: L.sph_run(c, 1)),
    "run, graph": (1 << 12, {}, lambda L, c: L.sph_run(c, 2)),
    "block step": (0, dict(block_levels=2), lambda L, c: L.sph_block_step(c, None, None)),
    "lists": (0, {}, lambda L, c: L.sph_neighbours(c, 0, None, C.c_void_p(1 << 21), C.c_void_p(1 << 22), C.c_int64(10),
                                                   C.byref(C.c_int64()))),
}


@pytest.mark.parametrize("name", CALLS)
@pytest.mark.parametrize("failing", ["launch_radix_sort", "launch_build_leaves"])
def test_state_is_cleared_after_a_failed_call(L, name, failing):
    stream, kw, call = CALLS[name]
    ctx, zero = _context(L, stream, **kw)
    assert L.sph_density_h(ctx) == sph.OK and L.sph_forces(ctx) == sph.OK
    L.fake_reset(failing.encode())
    if name == "step, kept leaves":  # (keeps them: no sort to fail; a density solve fails instead)
        assert L.sph_density_h(ctx) == sph.ECUDA
    else:
        assert call(L, ctx) == sph.ECUDA
    L.fake_reset(b"")
    assert call(L, ctx) == sph.OK
    t = _trace(L)
    assert t.index(zero) < t.index("launch_radix_sort") < t.index("launch_build_leaves")
    L.fake_reset(b"")
    assert call(L, ctx) == sph.OK
    assert zero not in _trace(L)
    L.sph_destroy(ctx)


def test_batch_state_is_cleared_after_a_failed_call(L):
    ctxs = (C.c_void_p * 2)(*[_context(L, 1 << 12)[0] for _ in range(2)])
    for c in ctxs:
        assert L.sph_density_h(C.c_void_p(c)) == sph.OK and L.sph_forces(C.c_void_p(c)) == sph.OK
    bt = C.c_void_p()
    L.fake_reset(b"")
    assert L.sph_batch_create(C.byref(bt), ctxs, 2, C.c_void_p(1 << 24), C.c_size_t(1 << 40), 0) == sph.OK
    zero = [t for t in _trace(L) if t.startswith("memset")][2]
    L.fake_reset(b"launch_build_leaves")
    assert L.sph_batch_run(bt, 1) == sph.ECUDA
    L.fake_reset(b"")
    assert L.sph_batch_run(bt, 1) == sph.OK
    t = _trace(L)
    assert t.index(zero) < t.index("launch_radix_sort")
    L.fake_reset(b"")
    assert L.sph_batch_run(bt, 1) == sph.OK
    assert zero not in _trace(L)
    L.sph_batch_destroy(bt)


def test_a_first_step_without_a_density_solve_builds_the_leaves(L):
    """With tree reuse a context keeps leaves only once it has some."""
    ctx, _ = _context(L, 0, tree_rebuild_every=4)
    L.fake_reset(b"")
    assert L.sph_step(ctx, C.c_double(1e-3), None) == sph.OK
    t = _trace(L)
    assert t.index("launch_radix_sort") < t.index("launch_build_leaves") < t.index("launch_density")
    L.fake_reset(b"")
    assert L.sph_step(ctx, C.c_double(1e-3), None) == sph.OK
    assert "launch_update_leaves" in _trace(L) and "launch_radix_sort" not in _trace(L)
    L.sph_destroy(ctx)

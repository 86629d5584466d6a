"""The kept scratch (csrc/scratch.cpp) on the host, over a CUDA runtime of this test's own: what is kept, for whom, what
makes room, and that nobody waits for another stream.  The runtime's streams run nothing; the test says which of them are at rest."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1311_0705_gb300", "csrc")

RUNTIME = r"""
#include <cuda_runtime.h>
#include <map>
#include "scratch.h"

namespace {
struct Event { cudaStream_t stream = nullptr; long at = -1; };
std::map<void *, size_t> live;
std::map<cudaStream_t, long> sent, done;
size_t used = 0, limit = (size_t)1 << 40;
int cross = 0, unsafe = 0;
cudaStream_t capture = nullptr;
cudaError_t last = cudaSuccess;
cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;
char *next = (char *)0x1000;
bool complete(const Event *e) { return e->at < 0 || done[e->stream] >= e->at; }
cudaError_t fail(cudaError_t e) { return last = e; }
cudaError_t take(void **p, size_t n) {
    if (used + n > limit) { *p = nullptr; return fail(cudaErrorMemoryAllocation); }
    used += n;
    *p = next;
    next += n;
    live[*p] = n;
    return cudaSuccess;
}
void give(void *p) { used -= live.at(p); live.erase(p); }
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return take(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { give(p); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st) {
    *st = capture && s == capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return capture && !s ? fail(cudaErrorStreamCaptureImplicit) : cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m) { auto o = mode; mode = *m; *m = o; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t) new Event; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (Event *)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { auto v = (Event *)e; v->stream = s; v->at = sent[s]; return cudaSuccess; }
static void check_mode() { if (mode != cudaStreamCaptureModeRelaxed) unsafe++; }
cudaError_t cudaEventQuery(cudaEvent_t e) { check_mode(); return complete((Event *)e) ? cudaSuccess : fail(cudaErrorNotReady); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    auto v = (Event *)e;
    check_mode();
    if (!complete(v)) done[v->stream] = v->at;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    auto v = (Event *)e;
    cross += v->stream != s && !complete(v);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { check_mode(); done[s] = sent[s]; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)0x77; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }

// the test's handles
long t_get(size_t n, long s, void **out) {
    auto v = new hg::Scratch;
    const cudaError_t e = hg::scratch_get(*v, n, (cudaStream_t)s);
    sent[(cudaStream_t)s]++;
    *out = v;
    return e;
}
void t_put(void *v, long s) { hg::scratch_put(*(hg::Scratch *)v, (cudaStream_t)s); delete (hg::Scratch *)v; }
void t_users(int delta) { hg::scratch_users(0, delta); }
void t_rest(long s) { done[(cudaStream_t)s] = sent[(cudaStream_t)s]; }
void t_capture(long s) { capture = (cudaStream_t)s; }
void t_forget() { used = 0; live.clear(); }
void t_limit(size_t n) { limit = n; }
size_t t_used() { return used; }
int t_blocks() { return (int)live.size(); }
int t_cross() { return cross; }
int t_unsafe() { return unsafe; }
long t_last() { return last; }
long t_malloc(size_t n) { void *p; return hg::device_malloc(&p, n); }
size_t t_address(void *v) { return (size_t)((hg::Scratch *)v)->p; }
}
"""

MB = 1 << 20


class Fake:
    def __init__(self, lib):
        self.lib = lib
        for f in ("t_used", "t_address"):
            getattr(lib, f).restype = ctypes.c_size_t
        lib.t_last.restype = lib.t_get.restype = ctypes.c_long
        lib.t_put.argtypes = [ctypes.c_void_p, ctypes.c_long]
        lib.t_address.argtypes = [ctypes.c_void_p]
        lib.t_malloc.argtypes, lib.t_malloc.restype = [ctypes.c_size_t], ctypes.c_long
        lib.t_limit.argtypes = [ctypes.c_size_t]
        lib.t_get.argtypes = [ctypes.c_size_t, ctypes.c_long, ctypes.POINTER(ctypes.c_void_p)]

    def get(self, n, s):
        p = ctypes.c_void_p()
        e = self.lib.t_get(n, s, ctypes.byref(p))
        return e, p

    def call(self, n, s):
        """One call's use of scratch; the block's address."""
        e, p = self.get(n, s)
        assert e == 0
        a = self.lib.t_address(p)
        self.lib.t_put(p, s)
        return a

    def reused(self, n, s):
        return self.call(n, s) == self.call(n, s)


@pytest.fixture()
def fake(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    (tmp_path / "runtime.cpp").write_text(RUNTIME)
    so = str(tmp_path / "scratch.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"), "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(tmp_path / "runtime.cpp"), os.path.join(CSRC, "scratch.cpp"), os.path.join(CSRC, "common.cpp"),
                    "-o", so], check=True)
    f = Fake(ctypes.CDLL(so))
    f.lib.t_users(1)
    yield f
    assert f.lib.t_cross() == 0  # no stream waited for another's work
    assert f.lib.t_unsafe() == 0  # no query or wait that would break a capture of another thread
    f.lib.t_users(-1)
    assert f.lib.t_used() == 0


def test_blocks_are_kept_for_their_stream(fake):
    assert fake.reused(100 * MB, 1)
    assert fake.call(100 * MB, 1) != fake.call(100 * MB, 2)
    assert fake.lib.t_used() == 200 * MB


def test_no_more_than_two_gibibytes_or_64_blocks_are_kept(fake):
    held = [fake.get(300 * MB, 1)[1] for _ in range(10)]
    for p in held:
        fake.lib.t_put(p, 1)
    assert 0 < fake.lib.t_used() <= 2048 * MB
    fake.lib.t_users(-1)
    assert fake.lib.t_used() == 0
    fake.lib.t_users(1)
    held = [fake.get(1000, 3)[1] for _ in range(100)]
    for p in held:
        fake.lib.t_put(p, 3)
    assert fake.lib.t_blocks() == 64
    assert fake.call(3000 * MB, 3) and fake.lib.t_used() <= 2048 * MB  # larger than all that is kept


@pytest.mark.parametrize("size,blocks", [(1000 * MB, 2), (1000, 64)], ids=["bytes", "count"])
def test_blocks_of_a_stream_at_rest_make_room(fake, size, blocks):
    held = [fake.get(size, 1)[1] for _ in range(blocks)]
    for p in held:
        fake.lib.t_put(p, 1)
    # the stream works still: its blocks stay, whatever others do
    for _ in range(300):
        fake.call(size, 2)
    assert fake.lib.t_blocks() == blocks and not fake.reused(size, 2)
    # at rest: others' blocks take their place, in time
    fake.lib.t_rest(1)
    for _ in range(300):
        fake.call(size, 2)
    assert fake.reused(size, 2)
    assert fake.lib.t_used() <= 2048 * MB


def test_streams_in_turn_do_not_displace_each_other(fake):
    # two streams that are waited for after every call, with more scratch than is kept for both: one goes on with its own
    first = fake.call(1500 * MB, 1)
    for _ in range(200):
        fake.lib.t_rest(1)
        assert fake.call(1500 * MB, 1) == first
        fake.call(1500 * MB, 2)
        fake.lib.t_rest(2)


def test_allocations_that_fail_are_tried_again_without_the_kept_blocks(fake):
    fake.call(900 * MB, 1)
    fake.lib.t_rest(1)
    fake.lib.t_limit(1000 * MB)
    assert fake.reused(800 * MB, 2)
    e, _ = fake.get(2000 * MB, 2)
    assert e == 2  # cudaErrorMemoryAllocation


def test_grids_and_models_get_the_kept_memory(fake):
    fake.call(900 * MB, 1)
    fake.lib.t_limit(1000 * MB)
    assert fake.lib.t_malloc(800 * MB) == 0 and fake.lib.t_used() == 800 * MB
    assert fake.lib.t_malloc(800 * MB) == 2 and fake.lib.t_last() == 0
    fake.lib.t_forget()


def test_kept_blocks_are_given_back_on_request(fake):
    for s in (1, 2, 3):
        fake.call(500 * MB, s)
    e, held = fake.get(400 * MB, 2)  # in use: not given back
    assert fake.lib.hg_release_scratch() == 0
    assert fake.lib.t_used() == 500 * MB
    fake.lib.t_put(held, 2)
    assert fake.reused(500 * MB, 2)  # kept as before


def test_no_error_is_left_behind(fake):
    fake.call(1000, 1)
    fake.lib.t_capture(5)  # the legacy stream's state cannot be asked for then
    fake.call(1000, 0)
    fake.lib.t_capture(0)
    assert fake.lib.t_last() == 0
    held = [fake.get(1000, 2)[1] for _ in range(80)]
    for p in held:
        fake.lib.t_put(p, 2)
    for _ in range(300):
        fake.call(2000, 4)
    assert fake.lib.t_last() == 0

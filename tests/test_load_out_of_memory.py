"""Loading a grid on the host, over a CUDA runtime of this test's own, with every single allocation failing in turn: the
call returns out of memory, or does with fewer threads; it never ends the process."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1311_0705_gb300", "csrc")

PROGRAM = r"""
#include <cuda_runtime.h>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include "gbuild.h"
#include "hg_internal.h"
#include "scratch.h"

static std::atomic<long> left{-1};  // allocations until one fails; negative: none does
void *operator new(size_t n) {
    if (left.load() >= 0 && left.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void *p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
}
namespace hg {
cudaError_t device_malloc(void **p, size_t n) { return (*p = std::malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
void scratch_users(int, int) {}
hg_status gpu_build_tree(const ModelView &, const hg_build_params &, void *, GpuTree &) { return HG_ECUDA; }
}  // namespace hg

int main() {
    hg_model m{};
    m.kind = HG_MODEL_CONST;
    m.p[0] = 1.0;
    m.m_tot = 8.0;
    for (int a = 0; a < 3; a++) m.lo[a] = -1.0, m.hi[a] = 1.0;
    hg_build_params p{};
    p.kind = HG_OCTREE;
    p.use_delta = 1;
    p.delta_max = 1.0 / 20000;
    p.max_level = 8;
    p.n_ran = 1;
    hg_host_grid *h = nullptr;
    hg_grid_desc d;
    if (hg_build_grid(&m, &p, 2, &h) != HG_OK || hg_host_grid_desc(h, &d) != HG_OK || d.n_leaves != 32768) return 2;
    long n = 0;
    for (;; n++) {
        hg_grid *g = nullptr;
        left = n;
        const hg_status st = hg_load_grid(&d, 0, &g);
        const bool all = left.load() >= 0;  // no allocation failed
        left = -1;
        if (st != HG_OK && st != HG_ENOMEM) return 3;
        if (st == HG_OK) hg_free_grid(g);
        if (all) break;
    }
    std::printf("%ld allocations\n", n);
    hg_free_host_grid(h);
    return 0;
}
"""


def test_every_allocation_of_a_load_may_fail(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    (tmp_path / "load.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "load")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(tmp_path / "load.cpp")] + [os.path.join(CSRC, f) for f in ("grid.cpp", "build.cpp", "common.cpp")] +
                   ["-o", exe, "-lpthread"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and int(r.stdout.split()[0]) > 10, (r.returncode, r.stdout, r.stderr)

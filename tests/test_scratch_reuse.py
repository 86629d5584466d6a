"""Scratch kept between calls: results on several streams and host threads, under capture and replay, across sizes,
and its release with the last grid.  Results must be those of calls made one at a time, bit for bit."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture()
def hg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_0705_gb300 as m
    return m


def _grid(hg, kind=1):
    model, bp, _, _ = synth.workload_disk_small()
    bp.kind = kind
    return hg.load_grid(hg.build_grid(model, bp))


def _rays(seed, n):
    o, k = synth.emission_rays(seed, n)
    return torch.tensor(o, device="cuda"), torch.tensor(k, device="cuda")


def test_streams_and_threads_share_nothing(hg):
    grid = _grid(hg)
    sizes = [300, 20000, 5000, 60000, 1]
    rays = [_rays(50 + i, n) for i, n in enumerate(sizes)]
    ref = [hg.trace_rays(grid, *r) for r in rays]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for turn in range(12):
                j = (i + turn) % len(rays)
                o, k = rays[j]
                if turn % 3 == 2:
                    R = hg.prepare_rays(grid, o, k)
                    tau, nc, st = R.trace()
                    off = hg.scan_offsets(nc)
                    R.free()
                else:
                    tau, nc, st = hg.trace_rays(grid, o, k)
                stream.synchronize() if turn % 4 == 0 else None
                if not (torch.equal(nc, ref[j][1]) and torch.allclose(tau, ref[j][0], rtol=1e-12, atol=0)):
                    bad.append((i, turn))
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not bad


def test_captured_calls_replay_beside_others(hg):
    grid = _grid(hg, 0)
    o, k = _rays(7, 30000)
    o2, k2 = _rays(8, 30000)
    ref, ref2 = hg.trace_rays(grid, o, k), hg.trace_rays(grid, o2, k2)
    out = tuple(torch.empty_like(t) for t in ref)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        hg.trace_rays(grid, o, k, out=out)
    for _ in range(3):
        for t in out:
            t.zero_()
        graph.replay()
        again = hg.trace_rays(grid, o2, k2)  # scratch of its own
        torch.cuda.synchronize()
        for a, b in list(zip(out, ref)) + list(zip(again, ref2)):
            torch.testing.assert_close(a, b, rtol=1e-12, atol=0)


ALONE = """
import ctypes, sys
sys.path.insert(0, {root!r})
import torch
import synth
import paper_1311_0705_gb300 as hg

def used():
    torch.cuda.synchronize()
    cu, dev, pool, v = ctypes.CDLL("libcuda.so.1"), ctypes.c_int(), ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuCtxGetDevice(ctypes.byref(dev)) == 0
    assert cu.cuDeviceGetMemPool(ctypes.byref(pool), dev) == 0
    assert cu.cuMemPoolGetAttribute(pool, 7, ctypes.byref(v)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT
    return int(v.value)

torch.zeros(1, device="cuda")
model, bp, _, _ = synth.workload_disk_small()
o, k = synth.emission_rays(9, 400000)
O, K = torch.tensor(o, device="cuda"), torch.tensor(k, device="cuda")
assert used() == 0
grids = [hg.load_grid(hg.build_grid(model, bp)) for _ in range(2)]
held = []
for n in (1000, 400000, 50000, 200000, 123456, 400000):
    o, k = O[:n].contiguous(), K[:n].contiguous()
    for g in grids:
        hg.trace_rays(g, o, k)
        R = hg.prepare_rays(g, o, k)
        R.trace_stage()
        R.free()
    held.append(used())
    assert held[-1] <= 2 << 30, held
assert held[-1] > 0, held
grids[0].free()
assert used() > 0
R = hg.prepare_rays(grids[1], O, K)
grids[1].free()
assert used() > 0  # the plan is alive
R.free()
assert used() == 0, used()
"""


def test_kept_scratch_is_bounded_and_given_back(hg):
    # in a process of its own: other tests' grids and plans keep scratch alive
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", ALONE.format(root=root)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr

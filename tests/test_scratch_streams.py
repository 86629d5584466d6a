"""Scratch kept between calls, with several threads and streams at work: every turn of every thread has to end, with
the results of calls made one at a time."""
import threading

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1311_0705_gb300 as m
    return m


def _grid(hg):
    model, bp, _, _ = synth.workload_disk_small()
    return hg.load_grid(hg.build_grid(model, bp))


def test_every_turn_ends_with_the_results_of_single_calls(hg):
    grid = _grid(hg)
    sizes = [300, 20000, 5000, 60000, 1]
    rays = [tuple(torch.tensor(a, device="cuda") for a in synth.emission_rays(50 + i, n)) for i, n in enumerate(sizes)]
    ref = [hg.trace_rays(grid, *r) for r in rays]
    torch.cuda.synchronize()
    turns, errors = [0] * 6, []

    def work(i):
        try:
            for turn in range(30):
                if turn % 10 == 0:  # short-lived streams: their blocks are at rest from then on
                    stream = torch.cuda.Stream()
                j = (i + turn) % len(rays)
                with torch.cuda.stream(stream):
                    R = hg.prepare_rays(grid, *rays[j])
                    tau, nc, st, _ = R.trace_stage()
                    R.free()
                    again = hg.trace_rays(grid, *rays[j])
                stream.synchronize()
                for got in ((tau, nc, st), again):
                    assert torch.equal(got[1], ref[j][1]) and torch.equal(got[2], ref[j][2])
                    torch.testing.assert_close(got[0], ref[j][0], rtol=1e-12, atol=0)
                turns[i] += 1
        except BaseException as e:  # an assertion in a thread fails no test by itself
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(turns))]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not errors and turns == [30] * len(turns)


def test_kept_scratch_is_given_back_on_request(hg):
    grid = _grid(hg)
    o, k = (torch.tensor(a, device="cuda") for a in synth.emission_rays(9, 400_000))

    def step():
        R = hg.prepare_rays(grid, o, k)
        out = R.trace_stage()
        R.free()
        torch.cuda.synchronize()
        return out

    first = step()
    kept = torch.cuda.mem_get_info()[0]
    hg.release_scratch()
    freed = torch.cuda.mem_get_info()[0] - kept
    assert freed > 300 << 20, freed  # 64 staged entries of 16 bytes per ray and more
    hg.release_scratch()  # nothing left: fine
    again = step()
    assert torch.equal(again[1], first[1])
    torch.testing.assert_close(again[0], first[0], rtol=1e-12, atol=0)

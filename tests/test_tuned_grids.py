"""Tuned grids: small batches take the path of untuned ones."""
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


@pytest.mark.parametrize("kind", [0, 1], ids=["octree", "kd"])
def test_small_batches_of_a_tuned_grid(hg, kind):
    # heavy-tailed paths and a thread for every ray: the tuner's samples differ by whether long paths are cut, which only
    # schedule 3 does
    model = synth.make_disk()
    host = hg.build_grid_gpu(model, synth.BuildParams(kind=kind, delta_max=1e-5, max_level=12, seed=3))
    o, k = (torch.tensor(a, device="cuda") for a in synth.emission_rays(4, 2000))
    grid = hg.load_grid(host)

    def call():
        n = hg.launch_count()
        out = hg.trace_rays(grid, o, k)
        return hg.launch_count() - n, out

    call()
    plain, ref = call()
    cfg, _ = hg.autotune(grid, o, k)
    assert cfg["schedule"] == 3
    launches, out = call()
    assert launches == plain
    assert torch.equal(out[1], ref[1]) and torch.equal(out[2], ref[2])
    torch.testing.assert_close(out[0], ref[0], rtol=1e-12, atol=0)
    # an order that is asked for is made
    n = hg.launch_count()
    hg.trace_rays(grid, o, k, schedule=3)
    assert hg.launch_count() - n == plain + 1


def test_only_what_makes_a_difference_is_tried(hg):
    model = synth.make_disk()
    o, k = (torch.tensor(a, device="cuda") for a in synth.emission_rays(4, 500))
    o *= 0.3
    for half, shapes in ((1.0, 3 * 2), (0.3, 3 * 2 * 2 * 4)):  # 64-byte records: schedules, blocks; 96-byte: all
        model = synth.make_disk(half=half)
        grid = hg.load_grid(hg.build_grid(model, synth.BuildParams(kind=0, delta_max=1e-3, max_level=8, seed=3)))
        n = hg.launch_count()
        for s in (1, 2, 3):
            hg.trace_rays(grid, o, k, schedule=s)
        once = (hg.launch_count() - n) / 3
        n = hg.launch_count()
        cfg, _ = hg.autotune(grid, o, k)
        assert hg.launch_count() - n == 4 * shapes * once  # one untimed and three timed calls each
        if half == 1.0:
            assert (cfg["smem_nodes"], cfg["min_blocks"]) == (64, 4)

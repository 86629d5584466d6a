"""Walks of 64-byte records (bounds that are single-precision numbers) for origins next to a wall at zero, down to
components that have no single-precision image but zero, bit for bit against the FP64 oracle."""
import numpy as np
import pytest

import oracle
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
@pytest.mark.parametrize("nav", ["lists", "ropes"])
@pytest.mark.parametrize("low", [-1074, -150, -128, -62], ids=lambda e: f"2^{e}")
def test_origins_next_to_a_wall_at_zero(hg, kind, nav, low):
    model = synth.make_torus(5, n_clumps=15)
    bp = synth.BuildParams(kind=kind, delta_max=2e-4, use_q=True, q_max=0.9, max_level=5, seed=11)
    grid, tree = hg.load_grid(hg.build_grid(model, bp), nav=nav), oracle.build_tree(model, bp)
    rng = np.random.default_rng(-low)
    n = 4000
    o = rng.uniform(-1, 1, (n, 3))
    tiny = rng.choice([-1.0, 1.0], (n, 3)) * np.ldexp(1.0, np.ceil(rng.uniform(low, low + 60, (n, 3))).astype(int))
    near = rng.random((n, 3)) < 0.7
    o = np.where(near, tiny, o)
    k = rng.choice([-1.0, 1.0], (n, 3)) * 2.0 ** rng.uniform(-29.9, 0, (n, 3))
    o[0], k[0] = [2.0 ** -130, 2.0 ** -110, 0.3], [-2.0 ** -29, -1.0, 0.1]
    ref = oracle.trace(tree, o, k, emit=True, max_steps=oracle.default_max_steps(tree.n_leaves))
    for split in ("auto", "force"):
        out = hg.trace_emit(grid, torch.tensor(o, device="cuda"), torch.tensor(k, device="cuda"), split=split)
        torch.cuda.synchronize()
        for key in ("ncross", "status", "seg_off", "seg_cell", "seg_ds"):
            np.testing.assert_array_equal(out[key].cpu().numpy(), ref[key], err_msg=key)

"""Walks of grids whose bounds are single-precision numbers (held as 64-byte records and decided mostly in
single precision) against the FP64 oracle, at the edges of what that path accepts: directions and origins
outside its ranges, nearly parallel and grazing rays, the smallest and largest domains, deep trees, small and
ragged launches, and batches that mix both kinds of record.  Everything is bit-exact but the optical depth,
whose additions may be grouped (a few ulps; 1e-12 relative covers the 4 n u of n crossings)."""
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


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _check(hg, grid, tree, o, k, smax=None, **opt):
    ref = oracle.trace(tree, o, k, smax=smax, emit=True, max_steps=oracle.default_max_steps(tree.n_leaves))
    out = hg.trace_emit(grid, _t(o), _t(k), None if smax is None else _t(smax), **opt)
    torch.cuda.synchronize()
    for key in ("ncross", "status", "seg_off", "seg_cell", "seg_ds"):
        np.testing.assert_array_equal(out[key].cpu().numpy(), ref[key], err_msg=key)
    np.testing.assert_allclose(out["tau"].cpu().numpy(), ref["tau"], rtol=1e-12, atol=0)
    return ref


def _grid(hg, kind, half=1.0, level=6, n_clumps=15, nav="lists"):
    # refined at the torus' edge and in its clumps: walls with one, two, four and many neighbors
    model = synth.make_torus(5, n_clumps=n_clumps)
    model.domain_lo, model.domain_hi = model.domain_lo * half, model.domain_hi * half
    model.params = model.params * np.array([half, half, 1.0])
    model.table = model.table * np.array([half] * 4 + [1.0])
    bp = synth.BuildParams(kind=kind, delta_max=2e-4, use_q=True, q_max=0.9, max_level=level, seed=11)
    model.m_tot *= half ** 3
    return hg.load_grid(hg.build_grid(model, bp), nav=nav), oracle.build_tree(model, bp)


def _rays(form, n, half):
    rng = np.random.default_rng(len(form) + n)
    o = rng.uniform(-half, half, (n, 3))
    k = synth.isotropic_dirs(rng, n)
    if form == "scaled":  # direction components on both sides of the accepted range
        k *= 2.0 ** rng.uniform(-60, 60, (n, 1))
        k *= np.where(rng.random((n, 3)) < 0.3, 2.0 ** rng.uniform(-45, 0, (n, 3)), 1.0)
    elif form == "parallel":  # one or two components zero, denormal or tiny: walls that are never reached
        tiny = rng.choice([0.0, -0.0, 5e-324, -1e-310, 1e-40, -1e-12, 1e-9, 3e-7], size=(n, 3))
        m = rng.random((n, 3)) < 0.5
        m[np.arange(n), rng.integers(0, 3, n)] = False
        k = np.where(m, tiny, k)
    elif form == "walls":  # origins on lattice planes and within an ulp of them, lattice directions
        o = np.round(o / half * 64) / 64 * half
        o = np.where(rng.random((n, 3)) < 0.3, np.nextafter(o, rng.choice([-9e9, 9e9], size=(n, 3))), o)
        m = rng.random(n) < 0.7
        k[m] = rng.choice([-1.0, -0.5, 0.0, 0.5, 1.0, np.nextafter(1.0, 2.0)], size=(m.sum(), 3))
        k[np.all(k == 0, axis=1), 1] = -1.0
    elif form == "outside":  # entering from outside, from near to far beyond the accepted origins
        o = synth.isotropic_dirs(rng, n) * half * 2.0 ** rng.uniform(1, 45, (n, 1))
        k = rng.uniform(-half, half, (n, 3)) - o
        k[::2] /= np.linalg.norm(k[::2], axis=1)[:, None]
    return np.ascontiguousarray(o), np.ascontiguousarray(k)


@pytest.mark.parametrize("kind", [0, 1], ids=["octree", "kd"])
@pytest.mark.parametrize("half", [1.0, 2.0 ** -20, 2.0 ** 20, 2.0 ** 21, 0.3],
                         ids=["unit", "smallest", "largest", "beyond", "not-single"])
@pytest.mark.parametrize("form", ["plain", "scaled", "parallel", "walls", "outside"])
def test_ray_forms_bit_exact(hg, kind, half, form):
    grid, tree = _grid(hg, kind, half)
    o, k = _rays(form, 3001, half)
    ref = _check(hg, grid, tree, o, k)
    assert ref["ncross"].sum() > 3001
    _check(hg, grid, tree, o, k, split="force")


@pytest.mark.parametrize("kind", [0, 1], ids=["octree", "kd"])
def test_path_ends_inside_and_on_walls(hg, kind):
    grid, tree = _grid(hg, kind)
    rng = np.random.default_rng(3)
    o, k = _rays("walls", 4000, 1.0)
    smax = rng.choice([1e-300, 2.0 ** -6, 0.25, 1.0, 100.0], size=4000) * np.where(rng.random(4000) < 0.5, 1.0, rng.random(4000) + 0.1)
    _check(hg, grid, tree, o, k, smax=smax)
    _check(hg, grid, tree, o, k, smax=smax, split="force")


@pytest.mark.parametrize("kind", [0, 1], ids=["octree", "kd"])
@pytest.mark.parametrize("nav", ["lists", "ropes"])
@pytest.mark.parametrize("level", [3, 4, 5], ids=["two-ulps", "last-bit", "beyond"])
def test_cells_of_one_ulp_bit_exact(hg, kind, nav, level):
    # planes at 1 + i 2^-(19 + level): cells a few single-precision ulps wide, where every decision falls back
    # on the exact arithmetic; one level further they are no single-precision numbers
    lo, hi = 1.0, 1.0 + 2.0 ** -19
    model = synth.make_dyadic(4, level=2, lo=lo, hi=hi)
    bp = synth.BuildParams(kind=kind, delta_max=2e-4, max_level=level, seed=2)
    grid, T = hg.load_grid(hg.build_grid(model, bp), nav=nav), oracle.build_tree(model, bp)
    rng = np.random.default_rng(8)
    o = lo + rng.random((2000, 3)) * (hi - lo)
    o[1000:] -= synth.isotropic_dirs(rng, 1000)
    k = synth.isotropic_dirs(rng, 2000)
    k[1000:] = lo + rng.random((1000, 3)) * (hi - lo) - o[1000:]
    ref = _check(hg, grid, T, o, k)
    assert ref["ncross"].sum() > 2000


@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 4865, 40000])
@pytest.mark.parametrize("shape", [dict(), dict(schedule=1, block=32), dict(schedule=2, block=96), dict(schedule=3),
                                   dict(split="force")], ids=lambda s: "-".join(f"{a}{b}" for a, b in s.items()) or "auto")
def test_ragged_launches(hg, n, shape):
    grid, tree = _grid(hg, 1)
    o, k = _rays("plain", n, 1.0)
    _check(hg, grid, tree, o, k, **shape)


def test_batch_of_both_kinds_of_record(hg):
    pairs = [_grid(hg, i % 2, half, nav=nav) for i, (half, nav) in
             enumerate([(1.0, "lists"), (0.3, "lists"), (1.0, "ropes"), (0.7, "ropes"), (4.0, "lists")])]
    sizes = [700, 1300, 0, 33, 2048]
    halves = [1.0, 0.3, 1.0, 0.7, 4.0]
    begin = np.concatenate([[0], np.cumsum(sizes)])
    rays = [_rays("plain", max(n, 1), h) for n, h in zip(sizes, halves)]
    o = np.concatenate([r[0][:n] for r, n in zip(rays, sizes)])
    k = np.concatenate([r[1][:n] for r, n in zip(rays, sizes)])
    batch = hg.Batch([p[0] for p in pairs], begin)
    for _ in range(2):
        tau, nc, st = batch.trace(_t(o), _t(k))
        torch.cuda.synchronize()
        for i, (grid, tree) in enumerate(pairs):
            s = slice(int(begin[i]), int(begin[i + 1]))
            if s.stop > s.start:
                ref = oracle.trace(tree, o[s], k[s])
                np.testing.assert_array_equal(nc[s].cpu().numpy(), ref["ncross"])
                np.testing.assert_array_equal(st[s].cpu().numpy(), ref["status"])
                np.testing.assert_allclose(tau[s].cpu().numpy(), ref["tau"], rtol=1e-12, atol=0)


def test_sampling_on_walls_matches_the_oracle(hg):
    for kind in (0, 1):
        for half in (1.0, 0.3):
            grid, tree = _grid(hg, kind, half)
            pts = _rays("walls", 5000, half)[0]
            cell, rho = hg.sample_density(grid, _t(pts))
            c, r = oracle.sample_density(tree, pts)
            np.testing.assert_array_equal(cell.cpu().numpy(), c)
            np.testing.assert_array_equal(rho.cpu().numpy(), r)

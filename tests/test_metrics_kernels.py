"""The disk model's density and quadrature kernels and the two-pass statistics at their edges, against the FP64
oracle and NumPy.  Densities: 2^-52 (s + 16) relative for an exponent s, whose last rounding may differ by one unit
(2^-52 s at most) beside the few of the root, quotients and exponential; optical depths: 1e-9, two integrators of local tolerance 1e-11; statistics: 1e-13 times
the largest magnitude, the additions being grouped differently."""
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


# scale heights: ordinary, exponents beyond the fast exponential's range, scale lengths beyond the fast path's
DISKS = [(1.0, 0.25, 0.03), (3.0, 0.3, 0.002), (1e-3, 1e-13, 0.1), (2.0, 5.0, 1e13)]


@pytest.mark.parametrize("disk", DISKS, ids=lambda d: "-".join(map(str, d)))
def test_disk_density_edges(hg, disk):
    model = synth.make_disk(rho_c=disk[0], h_R=disk[1], h_z=disk[2])
    pts = synth.sample_points(4, 5000)
    pts[:8] = [[0, 0, 0], [0, 0, 0.5], [1, 1, 1], [-1, 0, 0], [1e-300, 0, 0.1], [0, 1e-19, 0], [0, -0.0, -0.0], [1e-25, 1e-25, 1]]
    got = hg.model_density(hg.load_model(model), _t(pts)).cpu().numpy()
    ref = oracle.rho_true(model, pts)
    normal = ref > 1e-300  # below, the exponential itself runs out of digits
    s = -np.log(ref[normal] / disk[0])
    assert (np.abs(got[normal] - ref[normal]) <= 2.0 ** -52 * (s + 16) * ref[normal]).all()
    np.testing.assert_allclose(got[~normal], ref[~normal], rtol=0, atol=1e-300)


@pytest.mark.parametrize("disk", DISKS[:2], ids=lambda d: "-".join(map(str, d)))
@pytest.mark.parametrize("n", [1, 33, 700])
def test_disk_quadrature_edges(hg, disk, n):
    model = synth.make_disk(rho_c=disk[0], h_R=disk[1], h_z=disk[2])
    a, k, L = synth.endpoint_paths(n, n)
    special = [([0.3, 0.2, -0.7], [0, 0, 1], 1.5),      # parallel to the axis
               ([0, 0, -0.9], [0, 0, 1], 1.8),          # along it
               ([-0.8, 0, 0], [1, 0, 0], 1.6),          # in the midplane through the axis
               ([-0.8, 0.1, 0.05], [1, 0, 0], 1.6),     # parallel to the midplane
               ([-0.5, -0.5, -0.5], [3 ** -0.5] * 3, 1.0),  # through the centre
               ([0.1, 0.1, 0.1], [1, 0, 0], 0.0),       # empty
               ([0.5, 0.1, 0.9], [0, 1, 0], 0.3)]       # far from the midplane
    for i, (o, d, s) in enumerate(special[:n]):
        a[i], k[i], L[i] = o, d, s
    got = hg.model_tau(hg.load_model(model), _t(a), _t(k), _t(L), kappa=1.7).cpu().numpy()
    np.testing.assert_allclose(got, oracle.tau_true(model, a, k, L, kappa=1.7), rtol=1e-9, atol=1e-300)


@pytest.mark.parametrize("n", [1, 2, 255, 1025, 311_297, 1_000_003])
def test_statistics(hg, n):
    rng = np.random.default_rng(n)
    a, b = rng.normal(3.0, 2.0, n), rng.normal(-1.0, 0.5, n)
    out = hg.diff_stats(_t(a), _t(b)).cpu().numpy()
    x = a - b
    assert out[0] == n
    assert abs(out[1] - x.mean()) <= 1e-13 * np.abs(x).max()
    assert abs(out[2] - x.std()) <= 1e-13 * np.abs(x).max()

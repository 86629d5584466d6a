"""The disk model's metrics where a faster evaluation could go wrong."""
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


def _tau(hg, model, o, k, L):
    return hg.model_tau(hg.load_model(model), _t(o), _t(k), _t(L), kappa=1.7).cpu().numpy()


@pytest.mark.parametrize("h", [1e-155, 1e-160, 2e-162, 5e-324])
def test_quadrature_of_nearly_vertical_paths(hg, h):
    # h^2 is subnormal or zero: the path is vertical to all digits, wherever it is.  1e-9: two integrators of local
    # tolerance 1e-11
    model = synth.make_disk()
    o = np.array([[0.0, 0.3, -0.5], [0.3, 0.0, -0.5], [0.2, -0.1, 0.4], [-0.5, 0.5, -0.1]])
    for kx, ky in ((h, 0.0), (0.0, -h), (h, h)):
        k = np.tile([kx, ky, 1.0], (4, 1))
        k[2, 2] = -1.0
        L = np.array([1.0, 0.7, 0.9, 0.2])
        np.testing.assert_allclose(_tau(hg, model, o, k, L), oracle.tau_true(model, o, k, L, kappa=1.7), rtol=1e-9)


@pytest.mark.parametrize("disk", [(1.0, 0.25, 0.03), (1.0, 0.1, 0.3)], ids=lambda d: "-".join(map(str, d)))
def test_quadrature_rounds_no_worse_than_the_oracle(hg, disk):
    # In a plane through the axis the exponent is linear between the cuts: closed form, in extended precision.  Both
    # sides integrate the same intervals; 1.1 covers the other exponential and order of additions (the mean of 4000
    # errors is known to 2 %)
    rho_c, h_R, h_z = disk
    model = synth.make_disk(rho_c=rho_c, h_R=h_R, h_z=h_z)
    rng = np.random.default_rng(5)
    n = 4000
    a, b = rng.uniform(-1, 1, (n, 3)), rng.uniform(-1, 1, (n, 3))
    a[:, 1] = b[:, 1] = 0.0
    L = np.linalg.norm(b - a, axis=1)
    k = (b - a) / L[:, None]
    ld = np.longdouble
    o, d, end = a.astype(ld), k.astype(ld), L.astype(ld)
    cut = np.sort(np.clip(np.stack([-o[:, 0] / d[:, 0], -o[:, 2] / d[:, 2]], 1), 0, end[:, None]), axis=1)
    edge = np.concatenate([np.zeros((n, 1), ld), cut, end[:, None]], axis=1)
    s = lambda t: np.abs(o[:, 0] + d[:, 0] * t) / ld(h_R) + np.abs(o[:, 2] + d[:, 2] * t) / ld(h_z)
    tau = np.zeros(n, ld)
    for j in range(3):
        t0, t1 = edge[:, j], edge[:, j + 1]
        s0, ds = s(t0), s(t1) - s(t0)
        tau += np.where(t1 > t0, -np.exp(-s0) * np.expm1(-ds) * (t1 - t0) / np.where(ds == 0, 1, ds), 0)
    tau *= ld(rho_c) * ld(1.7)
    error = lambda x: float(np.mean(np.abs(x.astype(ld) - tau) / tau))
    assert error(_tau(hg, model, a, k, L)) <= 1.1 * error(oracle.tau_true(model, a, k, L, kappa=1.7))


@pytest.mark.parametrize("n", [1, 9, 300, 2433, 500_000])
def test_quadrature_repeats_itself(hg, n):
    model = synth.make_disk()
    o, k, L = synth.endpoint_paths(3, n)
    dm, args = hg.load_model(model), (_t(o), _t(k), _t(L))
    first = hg.model_tau(dm, *args)
    assert bool((first > 0).all())
    for _ in range(5):
        assert torch.equal(hg.model_tau(dm, *args), first)


def test_densities_are_those_of_the_cuda_functions(hg):
    # with y = 0 the radius is |x| whatever its rounding: torch's division and exponential, bit for bit
    model = synth.make_disk()
    p = _t(synth.sample_points(6, 200_000))
    p[:, 1] = 0.0
    p[100_000:, 2] *= 0.1
    h_R, h_z = (torch.full_like(p[:, 0], float(model.params[j])) for j in (1, 2))
    ref = torch.exp(-(p[:, 0].abs() / h_R + p[:, 2].abs() / h_z))
    assert torch.equal(hg.model_density(hg.load_model(model), p), ref)


@pytest.mark.parametrize("n", [2, 5, 1023])
def test_statistics_whose_sums_overflow(hg, n):
    a = np.full(n, 1.7e308)
    out = hg.diff_stats(_t(a), _t(np.zeros(n))).cpu().numpy()
    np.testing.assert_array_equal(out, [n, np.inf, np.inf])

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

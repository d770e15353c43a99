"""Gradients of densities far from 1 in size: the Coulomb part is quadratic in D, E_K's
in D = C C^T as well, whatever arithmetic a mixed handle picks for its
derivative integrals."""
import numpy as np
import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


@pytest.fixture(scope="module", params=[dfjk.DFJK_FP64, dfjk.DFJK_MIXED])
def case(request):
    m = I.molecule(6, seed=1006)
    h = dfjk.Handle(m, precision=request.param)
    C = torch.from_numpy(np.random.default_rng(6).standard_normal((m.nao, 18))).cuda() / m.nao**0.5
    yield h, C, h.coulomb_gradient(C @ C.T), h.jk_gradient(C, 0.0, 1.0), h.jk_gradient(C, 1.0, -0.5)
    h.close()


def _close(a, b):
    assert (a - b).abs().max().item() <= 1e-8 * b.abs().max().item()


@pytest.mark.parametrize("k", [-120, -70, -41, -39, -10, 10, 29, 45, 70, 120])
def test_coulomb(case, k):
    h, C, gj, _, _ = case
    _close(h.coulomb_gradient(C @ C.T * 2.0**k) * 2.0 ** (-2 * k), gj)


@pytest.mark.parametrize("k", [-60, -35, -13, -8, 8, 15, 30, 60])
def test_exchange(case, k):
    h, C, _, gk, gjk = case
    _close(h.jk_gradient(C * 2.0**k, 0.0, 1.0) * 2.0 ** (-4 * k), gk)
    _close(h.jk_gradient(C * 2.0**k, 1.0, -0.5) * 2.0 ** (-4 * k), gjk)


@pytest.mark.parametrize("k", [-90, -40, 40, 90])
def test_weights(case, k):
    h, C, gj, gk, _ = case
    _close(h.jk_gradient(C, 2.0**k, 0.0) * 2.0**-k, gj)
    _close(h.jk_gradient(C, 0.0, 2.0**k) * 2.0**-k, gk)


def test_zero(case):
    h, C, _, _, _ = case
    assert (h.jk_gradient(C * 0.0, 1.0, -0.5) == 0).all() and (h.coulomb_gradient(torch.zeros_like(C @ C.T)) == 0).all()

"""A density build whose bounded device waits expire says so, and the handle's next
call does not inherit the status.  The handle keeps no pair (Schwarz
threshold), so that its setup has no such waits and one poll per wait reaches
the density build."""
import ctypes

import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


@pytest.mark.parametrize("on_device", [False, True])
def test_expired_wait_is_reported(on_device):
    m = I.molecule(5, seed=1005)
    h = dfjk.Handle(m, precision=dfjk.DFJK_MIXED, schwarz_thresh=1e30, timeout_iters=1)
    D = torch.eye(m.nao, dtype=torch.float64, device="cuda")
    lib, E = dfjk.load_library(), torch.empty(2, dtype=torch.float64, device="cuda" if on_device else "cpu")
    J, K = torch.empty_like(D), torch.empty_like(D)
    at = [ctypes.c_void_p(x) for x in (D.data_ptr(), J.data_ptr(), K.data_ptr(), E.data_ptr(), E.data_ptr() + 8,
                                       torch.cuda.current_stream().cuda_stream)]
    rc = lib.dfjk_build_density(h.h, 1, *at)
    assert rc == 6, lib.dfjk_last_error()  # DFJK_ERR_TIMEOUT
    assert b"density" in lib.dfjk_last_error()
    g = h.coulomb_gradient(D)  # no bounded waits in this call
    assert (g == 0).all()
    h.close()


def test_without_pairs_and_with_the_default_limit():
    m = I.molecule(5, seed=1005)
    h = dfjk.Handle(m, precision=dfjk.DFJK_MIXED, schwarz_thresh=1e30)
    J, K, EJ, EK = h.build_density(torch.eye(m.nao, dtype=torch.float64, device="cuda"))
    assert (J == 0).all() and (K == 0).all() and EJ[0] == 0 and EK[0] == 0
    h.close()

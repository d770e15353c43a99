"""dfjk_estimate_bytes bounds what a first build adds to a handle (batching and
serving admit by it), also where screening makes the build's chunks longer.
The allocator may hand out blocks up to an eighth larger than asked for."""
import ctypes

import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


@pytest.mark.parametrize("precision", [dfjk.DFJK_FP64, dfjk.DFJK_MIXED])
@pytest.mark.parametrize("natom,occ", [(5, 0.2), (25, 0.28), (60, 0.2), (70, 0.05)])
def test_first_build(natom, occ, precision):
    lib = dfjk.load_library()
    lib.dfjk_debug_pool_peak.restype = ctypes.c_size_t
    m = I.molecule(natom, seed=1000 + natom)
    nocc = round(occ * m.nao)
    C = torch.randn(m.nao, nocc, dtype=torch.float64, device="cuda")
    lib.dfjk_trim_cache()
    h = dfjk.Handle(m, precision=precision)
    lib.dfjk_debug_pool_peak()
    held = lib.dfjk_debug_pool_peak()
    h.build(C)
    added = lib.dfjk_debug_pool_peak() - held
    h.close()
    lib.dfjk_trim_cache()
    assert added <= 1.125 * dfjk.estimate_bytes(m.nao, m.naux, nocc, precision)["build_ws"]

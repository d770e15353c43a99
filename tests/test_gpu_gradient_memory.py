"""The exchange gradient's memory: its dense part holds X, C^T X, Z, W and G in FP64,
the slices of the two operands without a batch, and ranges of the others'
within the work-buffer cap; and the ranges leave the gradient as it is."""
import numpy as np
import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


@pytest.mark.parametrize("precision", [dfjk.DFJK_FP64, dfjk.DFJK_MIXED])
def test_peak_and_ranges(precision, tmp_path):
    cap = 64  # MB
    table = tmp_path / "tune.txt"
    table.write_text(f"1 100000 16 8 64 {cap}\n")
    m = I.molecule(24, seed=1024)
    nocc = 72
    C = torch.from_numpy(np.random.default_rng(24).standard_normal((m.nao, nocc))).cuda() / m.nao**0.5
    peak = dfjk.load_library().dfjk_debug_pool_peak
    peak.restype = __import__("ctypes").c_size_t
    h = dfjk.Handle(m, precision=precision)
    ref = h.jk_gradient(C, 1.0, -0.5)
    h.close()
    h = dfjk.Handle(m, precision=precision, tune_table=str(table))
    peak()
    before = peak()  # what the handle holds
    g = h.jk_gradient(C, 1.0, -0.5)
    used = peak() - before
    h.close()
    npad, no2 = (m.naux + 63) // 64 * 64, nocc * nocc
    dense = 8 * (m.nao * npad * nocc + 2 * npad * no2 + npad * npad + npad * m.nao**2)
    slices = 16 * (2 * npad * no2 + npad * npad)
    assert used <= dense + 1.2 * slices + 4 * cap * 2**20
    # regrouped sums of the first product and the order of atomic sums
    assert (g - ref).abs().max().item() <= 1e-9 * ref.abs().max().item()


def test_finished_stages_are_given_back(tmp_path):
    """50 atoms: the first stage's slices pass the size from which they go back early."""
    table = tmp_path / "tune.txt"
    table.write_text("1 100000 16 8 64 1024\n")
    m = I.molecule(50, seed=1050)
    C = torch.from_numpy(np.random.default_rng(50).standard_normal((m.nao, 150))).cuda() / m.nao**0.5
    out = []
    for t in (None, str(table)):
        h = dfjk.Handle(m, precision=dfjk.DFJK_MIXED, tune_table=t)
        out.append(h.jk_gradient(C, 1.0, -0.5))
        h.close()
    assert (out[0] - out[1]).abs().max().item() <= 1e-9 * out[0].abs().max().item()

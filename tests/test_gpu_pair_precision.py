"""fp32_pair_thresh = 0 asks for every pair in FP64: a mixed handle then evaluates
its integrals as an FP64 handle does, bit for bit, and its Coulomb gradient
differs from that handle's by the whitening's slices alone.  With a positive
threshold below every pair's bound the pairs are double-single: the checks of
the double-single kernels run again on such handles."""
import numpy as np
import pytest

import test_gpu_df_integrals as base
from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402

BELOW = 1e-290  # every kept pair's bound is above it


def _integrals(m, precision):
    h = dfjk.Handle(m, precision=precision, fp32_pair_thresh=BELOW, schwarz_thresh=1e-10)
    assert h.npair_fp32 == 0
    T = h.three_center()
    h.close()
    return T


@pytest.fixture(autouse=True)
def double_single(monkeypatch):
    monkeypatch.setattr(base, "_integrals", _integrals)


test_standard_bases = base.test_standard_bases
test_separations_and_offsets = base.test_separations_and_offsets
test_contractions = base.test_contractions
test_exponent_limits = base.test_exponent_limits
test_exponents_beyond_the_range_take_fp64 = base.test_exponents_beyond_the_range_take_fp64


@pytest.mark.parametrize("natom", [3, 6])
def test_zero_threshold_is_fp64(natom):
    m = I.water() if natom == 3 else I.molecule(natom, seed=1000 + natom)
    T = []
    for precision, thresh in ((dfjk.DFJK_FP64, -1.0), (dfjk.DFJK_MIXED, 0.0), (dfjk.DFJK_MIXED, BELOW)):
        h = dfjk.Handle(m, precision=precision, fp32_pair_thresh=thresh, schwarz_thresh=0.0)
        assert h.npair_fp32 == 0 or thresh > 0  # unscreened: some bounds are zero
        T.append(h.three_center())
        h.close()
    assert torch.equal(T[0], T[1]) and not torch.equal(T[0], T[2])


def test_zero_threshold_build_and_gradient():
    m = I.molecule(6, seed=1006)
    C = torch.from_numpy(np.random.default_rng(6).standard_normal((m.nao, 18))).cuda() / m.nao**0.5
    out = []
    for precision in (dfjk.DFJK_FP64, dfjk.DFJK_MIXED):
        h = dfjk.Handle(m, precision=precision, fp32_pair_thresh=0.0)
        J, K, _, _ = h.build(C)
        out.append((J, K, h.coulomb_gradient(C @ C.T), h.jk_gradient(C, 1.0, -0.5)))
        h.close()
    for a, b in zip(*out):
        assert (a - b).abs().max().item() <= 1e-7 * a.abs().max().item()

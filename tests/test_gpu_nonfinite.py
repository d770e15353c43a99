"""Infinities, NaN and the ends of the exponent range in the sliced products: what
FP64 sums would make non-finite is non-finite, nothing else is, and results
down to the subnormals and up to the overflow are those of exact integers
scaled by powers of two."""
import numpy as np
import pytest

from paper_2404_09452_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402


def _gemm(A, B, S):
    return dfjk.sliced_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), S=S).cpu().numpy()


def _integers(M, K, seed):
    return np.random.default_rng(seed).integers(-30, 31, (M, K)).astype(float)


@pytest.mark.parametrize("S", [6, 8])
@pytest.mark.parametrize("ka,kb", [(0, 0), (500, 450), (500, 520), (1000, 1000), (-480, -500), (-530, -525), (-900, -900), (900, -950)])
def test_scaled_integers(S, ka, kb):
    A, B = _integers(130, 600, 1), _integers(70, 600, 2)
    with np.errstate(over="ignore"):
        ref = np.ldexp(A @ B.T, ka + kb)
    assert np.array_equal(_gemm(np.ldexp(A, ka), np.ldexp(B, kb), S), ref)


@pytest.mark.parametrize("S", [6, 8])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_rows(S, bad):
    A, B = _integers(130, 2100, 3), _integers(70, 2100, 4)
    ref = A @ B.T
    A[5, 1500] = A[129, 0] = B[64, 2099] = bad
    out = _gemm(A, B, S)
    rows, cols = np.isin(np.arange(130), [5, 129]), np.arange(70) == 64
    hit = rows[:, None] | cols[None, :]
    assert not np.isfinite(out[hit]).any() and np.array_equal(out[~hit], ref[~hit])


@pytest.mark.parametrize("precision", [dfjk.DFJK_FP64, dfjk.DFJK_MIXED])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_orbitals_and_densities(precision, bad):
    m = I.molecule(5, seed=1005)
    h = dfjk.Handle(m, precision=precision)
    C = torch.from_numpy(np.random.default_rng(1).standard_normal((m.nao, 15))).cuda()
    J0, K0, _, _ = h.build(C)
    shell = np.repeat(np.arange(len(m.orb.shells)), [(s.l + 1) * (s.l + 2) // 2 for s in m.orb.shells])
    kept = h.pair_mask().cpu().numpy()[np.ix_(shell, shell)] != 0  # by AO; screened pairs take no part
    Cb = C.clone()
    Cb[7, 3] = bad
    _, K, _, EK = h.build(Cb)
    assert kept[7].sum() > m.nao // 2
    assert not np.isfinite(K[0].diagonal().cpu().numpy()[kept[7]]).any() and not np.isfinite(EK[0])
    D = C @ C.T
    D[3, 4] = D[4, 3] = bad
    _, K, _, EK = h.build_density(D)
    assert not np.isfinite(K[0].diagonal().cpu().numpy()[kept[3] & kept[4]]).any() and not np.isfinite(EK[0])
    assert not h.jk_gradient(Cb, 1.0, -0.5).isfinite().any()
    J, K, _, _ = h.build(C)
    assert torch.equal(J, J0) and torch.equal(K, K0)
    h.close()


@pytest.mark.parametrize("precision", [dfjk.DFJK_FP64, dfjk.DFJK_MIXED])
@pytest.mark.parametrize("k", [-500, 480])
def test_tiny_and_huge_orbitals(precision, k):
    """K is quadratic in C: C 2^k gives K 2^(2k), but for elements that leave the range."""
    m = I.molecule(5, seed=1005)
    h = dfjk.Handle(m, precision=precision)
    C = torch.from_numpy(np.random.default_rng(2).standard_normal((m.nao, 15))).cuda()
    K0, K = h.build(C)[1][0], h.build(C * 2.0**k)[1][0]
    K = K * 2.0**-k * 2.0**-k
    assert (K - K0).abs().max().item() <= 1e-12 * K0.abs().max().item()
    h.close()

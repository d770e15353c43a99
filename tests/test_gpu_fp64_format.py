"""The slice format of the FP64 path (8 slices of 7 bits, 384 elements under one
exponent) bit for bit against a model in integers: balanced digits of every
element, the level sums of the digits' products, the four upper and the four
lower levels as two exact doubles joined with one rounding, and FP64 sums over
the blocks.  A lost slice, level or block, a wrong digit or a second rounding
changes bits.  Inputs: full mantissas, and digits at the ends of their range
that bring the level sums to theirs (2^24)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2404_09452_gb300 import dfjk  # noqa: E402

S, W, KB = 8, 7, 384


def _fixed(X, e):
    """X 2^(56 - e) to the nearest integer, halves away from zero (exact: |n| <= 2^56)."""
    x = np.ldexp(np.abs(X), S * W - e[:, None])
    n = np.where(x < 2.0**52, np.floor(x + 0.5), x).astype(np.int64)
    return np.where(X < 0, -n, n)


def _digits(X):
    """Digits [S, rows, k] and exponents [rows] of a block."""
    e = np.frexp(np.abs(X).max(1))[1]
    e[np.abs(X).max(1) == 0] = 0
    n = _fixed(X, e)
    d = np.empty((S,) + X.shape, dtype=np.int64)
    for s in range(S - 1, 0, -1):
        d[s] = ((n + 2 ** (W - 1)) & (2**W - 1)) - 2 ** (W - 1)
        n = (n - d[s]) >> W
    d[0] = n
    return d, e


def _model(A, B):
    out = None
    for k in range(0, A.shape[1], KB):
        a, ea = _digits(A[:, k:k + KB])
        b, eb = _digits(B[:, k:k + KB])
        lev = [sum(a[s] @ b[l - s].T for s in range(l + 1)) for l in range(S)]
        assert max(np.abs(x).max() for x in lev) <= 2**24
        total = sum(x.astype(object) * 2 ** (W * (S - 1 - l)) for l, x in enumerate(lev))
        v = np.array([[float(x) for x in row] for row in total])  # correctly rounded
        v = np.ldexp(v, ea[:, None] + eb[None, :] - W * (S + 1))
        out = v if out is None else out + v
    return out


def _check(A, B):
    C = dfjk.sliced_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), S=56).cpu().numpy()
    assert np.array_equal(C, _model(A, B))


SHAPES = [(1, 1, 1), (5, 7, 16), (130, 65, 384), (9, 70, 385), (33, 12, 1200)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_full_mantissas(M, N, K):
    rng = np.random.default_rng(M + K)
    A = rng.standard_normal((M, K)) * 10.0 ** rng.uniform(-6, 6, (M, K))  # elements far below their row's largest
    B = rng.standard_normal((N, K)) * 10.0 ** rng.uniform(-3, 3, (N, 1))
    A[M // 2, : K // 2] = 0.0
    _check(A, B)


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_extreme_digits(M, N, K):
    rng = np.random.default_rng(K)
    top = [2**53 - 1, 2**52, 2**52 + 1, 2**53 - 2**45, sum(64 << (7 * i) for i in range(7)), sum(63 << (7 * i) for i in range(7)) + 2**50]
    V = np.array([float(x) for x in top] + [-float(x) for x in top])
    A = np.repeat(V[np.arange(M) % V.size, None], K, axis=1)  # constant rows: every sum at its largest
    B = np.repeat(V[np.arange(N)[::-1] % V.size, None], K, axis=1)
    A[1::3] = V[rng.integers(0, V.size, A[1::3].shape)]
    B[2::3] = V[rng.integers(0, V.size, B[2::3].shape)]
    _check(A, B)


def test_small_factors_leave_one_rounding():
    """Rows of 7-bit integers against full mantissas: nothing is dropped, so a block's
    result is the correctly rounded exact sum."""
    rng = np.random.default_rng(7)
    A = rng.integers(-127, 128, (20, KB)).astype(float)
    A[:, 0] = 127.0
    B = rng.standard_normal((30, KB))
    for x, y in ((A, B), (B, A)):
        C = dfjk.sliced_gemm(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), S=56).cpu().numpy()
        e = np.frexp(np.abs(B).max(1))[1]
        n = _fixed(B, e).astype(object)
        exact = A.astype(int).astype(object) @ n.T
        ref = np.ldexp(np.array([[float(v) for v in r] for r in exact]), (e - 56)[None, :])
        assert np.array_equal(C, ref if x is A else ref.T)

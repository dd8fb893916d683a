"""The tensor-core complex GEMM of batches (exact products modulo small integers) at the edges of its plans:
contraction lengths at which the modulus set or the number of exact K parts changes, lengths of
each operand kernel, tile remainders, and operands whose sums reach the largest accumulator values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


# Every value of a line is rounded to an integer (error 1/2 for Re and Im) after scaling the line's
# 2-norm to at least 2^(ALPHA - 1.1), so an entry is off by at most
# 2 * sqrt(2 K) / 2 * 2^-(ALPHA - 1.1) |a| |b| per component; the 56-bit tier adds FP64 roundings.
N_ITEMS = 12  # the smallest batch that takes residue products
ALPHA = {negf.PREC_MIXED_40: 39.5, negf.PREC_MIXED: 47.5, negf.PREC_MIXED_56: 56.5}


def _check(A, B, prec):
    got = negf.zgemm(torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda"),
                     precision=prec).cpu().numpy()
    K = A.shape[-1]
    wide = np.clongdouble if K <= 1100 else np.complex128  # the sum's own rounding is in K 2^-52
    ref = A.astype(wide) @ B.astype(wide)
    scale = (np.linalg.norm(A, axis=-1)[..., :, None] * np.linalg.norm(B, axis=-2)[..., None, :])
    tol = (np.sqrt(2.0) * np.sqrt(2.0 * K) * 2.0 ** -(ALPHA[prec] - 1.1) + K * 2.0 ** -52) * scale
    assert np.all(np.abs(got - ref) <= tol), float((np.abs(got - ref) / tol).max())


def _rand(rng, *shape):
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


KS = [1, 15, 16, 17, 63, 65, 256, 257, 400, 401, 512, 513, 640, 641, 800, 801, 1024, 1025, 2300,
      4600, 11400]


@pytest.mark.parametrize("prec", [negf.PREC_MIXED_40, negf.PREC_MIXED, negf.PREC_MIXED_56])
@pytest.mark.parametrize("K", KS)
def test_contraction_lengths(K, prec):
    rng = np.random.default_rng(K)
    _check(_rand(rng, N_ITEMS, 19, K), _rand(rng, N_ITEMS, K, 35), prec)
    # equal entries: every product of a residue plane has the same sign, the largest sums
    a, b = complex(rng.uniform(0.1, 1), rng.uniform(0.1, 1)), complex(rng.uniform(0.1, 1), -0.7)
    _check(np.full((N_ITEMS, 5, K), a), np.full((N_ITEMS, K, 9), b), prec)


@pytest.mark.parametrize("prec", [negf.PREC_MIXED, negf.PREC_MIXED_56])
@pytest.mark.parametrize("M,N", [(1, 1), (127, 31), (128, 32), (129, 33), (257, 65), (64, 97),
                                 (300, 129), (130, 256)])
def test_tile_remainders(M, N, prec):
    rng = np.random.default_rng(1000 * M + N)
    for n in (N_ITEMS, 41):
        _check(_rand(rng, n, M, 70), _rand(rng, n, 70, N), prec)


@pytest.mark.parametrize("prec", [negf.PREC_MIXED_40, negf.PREC_MIXED, negf.PREC_MIXED_56])
def test_graded_zero_and_non_finite_lines(prec):
    """Lines spanning the FP64 range scale by their own norm, zero lines give zeros, and a line that
    holds an infinity or NaN makes its own products NaN and no others."""
    rng = np.random.default_rng(7)
    A, B = _rand(rng, N_ITEMS, 40, 50), _rand(rng, N_ITEMS, 50, 30)
    A *= 10.0 ** np.linspace(-150, 140, 40)[None, :, None]
    B[:, :, 3] = 0.0
    A[:, 5] = 0.0
    _check(A, B, prec)
    A[0, 7, 11] = complex(0.0, np.inf)
    B[0, 2, 9] = np.nan
    got = negf.zgemm(torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda"),
                     precision=prec).cpu().numpy()[0]
    bad = np.zeros((40, 30), bool)
    bad[7], bad[:, 9] = True, True
    assert np.all(np.isnan(got[bad].real)) and np.all(np.isfinite(got[~bad]))

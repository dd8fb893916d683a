"""FP64 products on both sides of the rule between tiles and strips (whole and started waves of tiles,
remainders of tiles and strips), for all operand forms and an accumulated output."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


def _op(X, op):
    return X if op == "N" else (np.swapaxes(X, 1, 2) if op == "T" else np.swapaxes(X, 1, 2).conj())


@pytest.mark.parametrize("n,M,N,K", [(152, 64, 64, 9), (153, 64, 64, 9), (38, 128, 128, 17),
                                     (64, 127, 130, 3), (1, 65, 3, 1), (5, 130, 127, 40),
                                     (3, 4, 8, 8), (2, 320, 200, 5)])
@pytest.mark.parametrize("opA", "NTC")
@pytest.mark.parametrize("opB", "NTC")
def test_tiles_and_strips(n, M, N, K, opA, opB):
    rng = np.random.default_rng(n + M)
    rand = lambda *s: rng.normal(size=s) + 1j * rng.normal(size=s)  # noqa: E731
    A = rand(n, *((M, K) if opA == "N" else (K, M)))
    B = rand(n, *((K, N) if opB == "N" else (N, K)))
    C = rand(n, M, N)
    for beta in (0.0, -0.5):
        got = negf.zgemm(torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda"),
                         torch.as_tensor(C.copy(), device="cuda") if beta else None, alpha=1.0,
                         beta=beta, opA=opA, opB=opB, precision=negf.PREC_FP64).cpu().numpy()
        a, b = _op(A, opA), _op(B, opB)
        # 2 K + 4 roundings of terms and sums, each of at most |A| |B| + |C|
        bound = np.abs(a) @ np.abs(b) * 2 + np.abs(C)
        assert np.all(np.abs(got - (a @ b + beta * C)) <= (4 * K + 8) * 2.0 ** -53 * bound)

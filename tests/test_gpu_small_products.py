"""FP64 block products below the tile size, at the edges of their strips."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


def _rand(rng, *shape):
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def _op(x, op):
    return x if op == "N" else x.swapaxes(-1, -2) if op == "T" else x.conj().swapaxes(-1, -2)


@pytest.mark.parametrize("n", [1, 7, 64])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (3, 5, 2), (4, 24, 7), (5, 25, 40), (40, 40, 40),
                                   (41, 33, 16), (64, 64, 64), (8, 48, 130), (100, 49, 31),
                                   (128, 128, 20), (129, 128, 20)])
def test_small_fp64_products(n, M, N, K):
    """Every option of the block product; a sum of K complex products and one more term is off by at
    most 2 (K + 4) eps of the sum of the moduli per component."""
    rng = np.random.default_rng(100 * M + N)
    for opa, opb in [("N", "N"), ("T", "C"), ("C", "N"), ("N", "T")]:
        A = _rand(rng, n, *((M, K) if opa == "N" else (K, M)))
        B = _rand(rng, n, *((K, N) if opb == "N" else (N, K)))
        C = _rand(rng, n, M, N)
        alpha, beta = 0.7 - 0.2j, -1.1 + 0.3j
        got = negf.zgemm(*(torch.as_tensor(x, device="cuda") for x in (A, B, C)), alpha=alpha,
                         beta=beta, opA=opa, opB=opb).cpu().numpy()
        a, b = _op(A, opa).astype(np.clongdouble), _op(B, opb).astype(np.clongdouble)
        ref = alpha * (a @ b) + beta * C
        size = abs(alpha) * (abs(a) @ abs(b)) + abs(beta) * abs(C)
        tol = 2 * np.sqrt(2.0) * (K + 4) * 2.0 ** -52 * size
        assert np.all(np.abs(got - ref) <= tol)

"""Products of batches (residues) keep the precision that the tiers state, for every shape of line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu
N_ITEMS, FEW, M = 12, 6, 12
BITS = {negf.PREC_MIXED_40: 40, negf.PREC_MIXED: 48, negf.PREC_MIXED_56: 56}
KS = [16, 64, 256, 400, 512, 560, 600, 1024, 2000, 3430]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


def _products(A, B):
    """The 64-bit product, and per tier the error of one batch and of calls of a few items."""
    ref = A.astype(np.clongdouble) @ B.astype(np.clongdouble)
    a, b = (torch.as_tensor(np.ascontiguousarray(x), device="cuda") for x in (A, B))
    for prec, bits in BITS.items():
        batch = negf.zgemm(a, b, precision=prec)
        few = torch.cat([negf.zgemm(a[i:i + FEW], b[i:i + FEW], precision=prec)
                         for i in range(0, N_ITEMS, FEW)])
        yield bits, *(np.abs(x.cpu().numpy() - ref).astype(float) for x in (batch, few))


@pytest.mark.parametrize("K", KS)
def test_normal_entries_are_no_less_accurate_than_in_small_calls(K):
    rng = np.random.default_rng(K)
    A, B = (rng.normal(size=s) + 1j * rng.normal(size=s) for s in ((N_ITEMS, M, K), (N_ITEMS, K, M)))
    for bits, e, f in _products(A, B):
        assert np.linalg.norm(e) <= np.linalg.norm(f), bits


@pytest.mark.parametrize("K", KS)
def test_entries_of_one_size_keep_the_stated_error(K):
    """Such a line's 2-norm, sqrt(K) times an entry, is the largest possible.  The 3456 results' rms error
    is at most 1.2 * 2^-(bits + 2) of the norms, twice that bounds every one beyond 6 sigma of chance
    for random phases (FP64's rounding added); equal entries have equal roundings, whose worst case
    over K terms is 2 sqrt(2 K) 2^-(bits + 2)."""
    rng = np.random.default_rng(K)
    phase = [np.exp(2j * np.pi * rng.uniform(size=s)) for s in ((N_ITEMS, M, K), (N_ITEMS, K, M))]
    for bits, e, _ in _products(*phase):
        assert np.sqrt((e ** 2).mean()) <= (1.2 * 2.0 ** -(bits + 2) + 2.0 ** -53) * K, bits
        assert e.max() <= (8 * 2.0 ** -(bits + 2) + K * 2.0 ** -53) * K, bits
    equal = (0.84 * np.broadcast_to(phase[0][:, :, :1], phase[0].shape),
             0.84 * np.broadcast_to(phase[1][:, :1], phase[1].shape))
    for bits, e, _ in _products(*equal):
        assert e.max() <= (2 * np.sqrt(2.0 * K) * 2.0 ** -(bits + 2) + K * 2.0 ** -53) * K, bits

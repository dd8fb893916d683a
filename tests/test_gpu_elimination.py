"""Sizes at which the blocked FP32 elimination of the mixed block inverse changes its panel width or
the rows a thread holds, and panels narrower than the width at the end of a matrix."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


@pytest.mark.parametrize("n", [149, 150, 161, 223, 224, 225, 447, 448, 449, 685, 690, 899, 1290,
                               1793, 2700])
def test_inverse_over_panel_sizes(n):
    rng = np.random.default_rng(n)
    nb = 2 if n < 1000 else 1
    H = (rng.normal(size=(nb, n, n)) + 1j * rng.normal(size=(nb, n, n))) / np.sqrt(n)
    H = 0.5 * (H + np.swapaxes(H, 1, 2).conj())
    M = np.array([0.2 + 1e-2j, -0.4 + 1e-3j])[:nb, None, None] * np.eye(n) - H
    # a zero in the first pivot's place forces an exchange there
    M[:, 0, 0] = 0.0
    X, st = negf.zinv(torch.as_tensor(M, device="cuda"), precision=negf.PREC_MIXED)
    X = X.cpu().numpy()
    assert np.all(st.cpu().numpy() == 0)
    ref = np.linalg.inv(M)
    for p in range(nb):
        kappa = np.linalg.norm(M[p], 2) * np.linalg.norm(ref[p], 2)
        assert np.abs(X[p] - ref[p]).max() / np.abs(ref[p]).max() < 1e-15 * kappa * n

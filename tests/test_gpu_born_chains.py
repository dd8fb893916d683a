"""The Born update at the edges of its chains of energies, and its largest change out of the ordinary range."""
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


@pytest.mark.parametrize("n_E,n_orb,shift", [(1, 1, 0), (5, 3, 0), (37, 50, 1), (64, 33, 5),
                                             (400, 4001, 12), (400, 4001, 399), (9, 20, 9),
                                             (9, 20, 2 ** 31 - 1), (3000, 1000, 160)])
def test_born_update_chains(n_E, n_orb, shift):
    """Against the update written out; sums of eleven FP64 terms, 1e-14 of the largest entry."""
    rng = np.random.default_rng(n_E + shift % 1000)
    gR, gL = _rand(rng, 2, n_E, n_orb), _rand(rng, 2, n_E, n_orb)
    sR, sL = _rand(rng, n_E, n_orb), _rand(rng, n_E, n_orb)
    w, ac, op, n0, mix = np.array([0.3, 0.7]), 0.02, 0.05, 0.4, 0.6
    R, L = (np.einsum("k,keo->eo", w, g) for g in (gR, gL))

    def at(x, d):  # x at energies shifted by d, 0 beyond the window
        y = np.zeros_like(x)
        if abs(d) < n_E:
            y[max(0, -d):n_E - max(0, d)] = x[max(0, d):n_E - max(0, -d)]
        return y

    Rup, Lup, Rdn, Ldn = at(R, shift), at(L, shift), at(R, -shift), at(L, -shift)
    wR = (1 - mix) * sR + mix * (ac * R + op * ((1 + n0) * Rdn + n0 * Rup + 0.5 * (Ldn - Lup)))
    wL = (1 - mix) * sL + mix * (ac * L + op * ((1 + n0) * Lup + n0 * Ldn))
    want = max(np.abs(wR - sR).max(), np.abs(wL - sL).max())
    cu = lambda x: torch.as_tensor(x, device="cuda")
    tR, tL = cu(sR.copy()), cu(sL.copy())
    d = negf.scba_step(cu(gR), cu(gL), cu(w), tR, tL, ac, op, shift, n0, mix=mix)
    for got, ref in ((tR, wR), (tL, wL)):
        assert np.abs(got.cpu().numpy() - ref).max() <= 1e-14 * np.abs(ref).max()
    assert abs(float(d) - want) <= 1e-14 * max(want, 5.0)


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e200, 1e-200])
def test_born_update_delta_outside_the_range_of_squares(bad):
    z = np.zeros((1, 40, 30), complex)
    g = z.copy()
    g[0, 7, 3] = bad
    cu = lambda x: torch.as_tensor(x, device="cuda")
    sR, sL = cu(z[0].copy()), cu(z[0].copy())
    d = float(negf.scba_step(cu(g), cu(z), cu(np.ones(1)), sR, sL, 1.0, 0.0, 2, 0.0, mix=1.0))
    assert d == (bad if np.isfinite(bad) else np.inf)

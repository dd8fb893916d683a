"""Products that take an operand's converted form over from the product before (decimation and sweeps),
and Newton-Schulz steps whose products have the width that the step needs: the mixed form of a batch
against the FP64 form, which shares none of this, with dense hoppings (operands shared) and with
interface hoppings of unequal extents (operands of other columns and rows, converted again)."""
import pytest

from workloads import make_device

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu

N_ITEMS = 12  # the smallest batch that takes residue products


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


def _solve(dev, E, prec, iface, scat):
    d = negf.Device(torch.as_tensor(dev.D[None], device="cuda"),
                    torch.as_tensor(dev.T[None], device="cuda"), iface=iface)
    st = torch.zeros(len(E), dtype=torch.int32, device="cuda")
    opt = negf.options(precision=prec, eta_lead=1e-2, eta_device=1e-2)
    lead = negf.lead_selfenergy(d, E, st, opt)
    kw = {}
    if scat:
        n = dev.D.shape[0] * dev.D.shape[1]
        g = torch.Generator(device="cuda").manual_seed(5)
        gam = 0.02 + 0.03 * torch.rand((len(E), n), dtype=torch.float64, device="cuda", generator=g)
        kw = dict(scat_R=(-1j * gam).contiguous(), scat_L=(1j * gam).contiguous(), diag=True)
    out = negf.rgf_solve(d, E, st, lead["sigma_R"], lead["sigma_L"], opt, **kw)
    out.update({q: lead[q] for q in ("sigma_R", "sigma_L")})
    return {k: v for k, v in out.items() if isinstance(v, torch.Tensor)}


# A 48-bit product is exact to 2^-46 sqrt(2 K) of its lines' norms (40-bit ones, late decimation steps:
# 2^-38.4, damped by the step); eta = 1e-2 limits what inverses and the decimation's doubling add to
# (norm / eta)^2 = 1e5 each: 1e-7 of the largest value bounds both, where a stale operand is off by
# the value itself.
@pytest.mark.parametrize("iface,scat", [(None, False), (None, True), ((17, 29), False),
                                        ((40, 40), True)])
@pytest.mark.parametrize("n_pts", [3, N_ITEMS])
def test_mixed_batch_matches_fp64(iface, scat, n_pts):
    dev = make_device(4, 70, 77, ge_frac=0.1, iface=iface)
    E = torch.linspace(-0.2, 0.3, n_pts, dtype=torch.float64, device="cuda")
    ref = _solve(dev, E, negf.PREC_FP64, iface, scat)
    for prec in (negf.PREC_MIXED, negf.PREC_MIXED_56):
        got = _solve(dev, E, prec, iface, scat)
        for k, v in ref.items():
            if v.is_floating_point() or v.is_complex():
                assert (got[k] - v).abs().max() <= 1e-7 * v.abs().max(), (k, prec)
            else:
                assert torch.equal(got[k], v), k


@pytest.mark.parametrize("prec", [negf.PREC_MIXED_40, negf.PREC_MIXED, negf.PREC_MIXED_56])
@pytest.mark.parametrize("n,b", [(1, 9), (1, 130), (5, 65), (N_ITEMS, 33), (N_ITEMS, 257)])
@pytest.mark.parametrize("eta", [1e-2, 1e-6])
def test_inverse_widths(prec, n, b, eta):
    """Residual of the inverse at the width of the last step, whatever the earlier steps had."""
    g = torch.Generator(device="cuda").manual_seed(b)
    H = torch.randn((n, b, b), dtype=torch.complex128, device="cuda", generator=g) / (2 * b) ** 0.5
    M = -(H + H.mH) / 2
    M.diagonal(dim1=1, dim2=2).add_(0.05 + 1j * eta)
    X, st = negf.zinv(M.contiguous(), precision=prec)
    assert int(st.abs().sum()) == 0
    norms = torch.linalg.matrix_norm(M, 2) * torch.linalg.matrix_norm(X, 2)
    R = torch.linalg.matrix_norm(M @ X - torch.eye(b, dtype=M.dtype, device="cuda"))
    # the residual product, the last correction (R^2, below 2^-48 b) and X's own rounding
    width = {negf.PREC_MIXED_40: 38.4, negf.PREC_MIXED: 46.4, negf.PREC_MIXED_56: 52.0}[prec]
    assert torch.all(R <= 2 * b * norms * 2.0 ** -width + b * 2.0 ** -46)

"""Interface couplings over nearly the whole block, in batches (residue products): the contraction is
then a little shorter than the block and can take more moduli than the block's own products."""
import numpy as np
import pytest

from workloads import make_device

torch = pytest.importorskip("torch")
negf = pytest.importorskip("paper_1510_04686_gb300")

pytestmark = pytest.mark.gpu
N, P, ETA = 3, 12, 1e-2
TOL = 1e-6  # what the mixed tiers state, of the largest value; eta keeps the blocks well conditioned


@pytest.fixture(scope="module", autouse=True)
def _lib():
    negf._build.build()
    negf.library()


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _run(dev, E, prec, iface, contacts=None):
    d = negf.Device(_t(dev.D[None]), _t(dev.T[None]), iface=iface)
    st = torch.zeros(P, dtype=torch.int32, device="cuda")
    opt = negf.options(precision=prec, eta_lead=ETA, eta_device=ETA)
    lead = negf.lead_selfenergy(d, _t(E), st, opt)
    rng = np.random.default_rng(5)
    V = _t(rng.uniform(-0.2, 0.2, (N, dev.D.shape[1]))).requires_grad_()
    # the sweeps start from the same contacts in every form
    sR, sL = contacts or (lead["sigma_R"], lead["sigma_L"])
    dens, cur = negf.rgf(V, d, _t(E), st, sR, sL, opt)
    torch.autograd.backward([dens, cur], [_t(rng.normal(size=dens.shape)),
                                          _t(rng.normal(size=cur.shape))])
    assert int(lead["status"].abs().sum()) == 0
    return (sR, sL), [x.detach().cpu().numpy() for x in (lead["sigma_R"], dens, cur, V.grad)]


@pytest.mark.parametrize("b,r,c", [(600, 560, 560), (600, 570, 540), (610, 576, 576)])
def test_wide_supports_in_batches(b, r, c):
    dev = make_device(N, b, 77 + r, ge_frac=0.1, iface=(r, c))
    E = np.linspace(-1.5, 1.4, P)
    contacts, ref = _run(dev, E, negf.PREC_FP64, None)
    for prec in (negf.PREC_MIXED, negf.PREC_MIXED_56):
        for name, x, y in zip(("sigma", "density", "current", "gradient"),
                              _run(dev, E, prec, (r, c), contacts)[1], ref):
            assert np.abs(x - y).max() <= TOL * np.abs(y).max(), (prec, name)

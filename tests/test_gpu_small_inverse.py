"""The FP64 block inverse in one CTA (pivots found a column ahead) at the edges of its loops and splits,
the thin trailing update of wide blocks, and operand lines of subnormal numbers."""
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


# Gauss-Jordan with partial pivoting: |X M - I| <= c n u |X||M| with a growth factor of order one
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 47, 48, 49, 63, 64, 65, 96, 97, 105, 106, 107])
def test_fp64_inverse_edges(n):
    rng = np.random.default_rng(n)
    M = _rand(rng, 3, n, n)
    M[1] *= 1e-120
    if n > 2:
        M[2, :, 0] = 0.0  # the pivot of the first column is in its last row
        M[2, -1, 0] = 1e-3
    X, st = negf.zinv(torch.as_tensor(M.copy(), device="cuda"), precision=negf.PREC_FP64)
    X = X.cpu().numpy()
    assert np.all(st.cpu().numpy() == 0)
    for p in range(3):
        R = X[p] @ M[p] - np.eye(n)
        norms = np.linalg.norm(X[p]) * np.linalg.norm(M[p])
        assert np.abs(R).max() <= 8 * n * 2.0 ** -52 * norms


def test_fp64_inverse_of_singular_and_nan_items_leaves_the_others():
    rng = np.random.default_rng(4)
    M = _rand(rng, 4, 40, 40)
    M[1, :, 7] = 0.0
    M[2, 3, 5] = np.nan
    X, st = negf.zinv(torch.as_tensor(M.copy(), device="cuda"), precision=negf.PREC_FP64)
    st = st.cpu().numpy()
    assert st[1] & 2 and st[0] == 0 and st[3] == 0
    X = X.cpu().numpy()
    for p in (0, 3):
        assert np.abs(X[p] @ M[p] - np.eye(40)).max() < 1e-10


# panels of eight columns (tiles), of four (thin update), and a last panel of two
@pytest.mark.parametrize("n", [2420, 2430, 2501])
def test_mixed_inverse_of_wide_blocks(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    H = torch.randn((1, n, n), dtype=torch.complex128, device="cuda", generator=g) / (2 * n) ** 0.5
    M = -(H + H.mH) / 2
    M.diagonal(dim1=1, dim2=2).add_(0.05 + 0.05j)  # |M| <= 1.5, |X| <= 20
    X, st = negf.zinv(M.contiguous(), precision=negf.PREC_MIXED)
    assert int(st.abs().sum()) == 0
    R = M[0] @ X[0] - torch.eye(n, dtype=M.dtype, device="cuda")
    # rows of M and columns of X have 2-norms below 1.5 and 20: products to 2^-46 sqrt(2 n) of both
    assert R.abs().max() <= 30 * (2 * n) ** 0.5 * 2.0 ** -46 + n * 2.0 ** -50


def test_subnormal_operand_lines():
    """Lines of numbers down to 2^-1074 beside ordinary ones: exact to the tier relative to the larger
    of the line's norm and the smallest normal number."""
    rng = np.random.default_rng(2)
    A, B = _rand(rng, 12, 20, 33), _rand(rng, 12, 33, 17)
    A[:, 3] *= 1e-310
    A[:, 4] = 5e-324
    A[:, 5, ::2] *= 1e-309
    B *= 1e300
    got = negf.zgemm(torch.as_tensor(A, device="cuda"), torch.as_tensor(B, device="cuda"),
                     precision=negf.PREC_MIXED).cpu().numpy()
    ref = A.astype(np.clongdouble) @ B.astype(np.clongdouble)
    na = np.maximum(np.linalg.norm(A.astype(np.clongdouble), axis=-1), np.sqrt(2 * 33) * 2.0 ** -1022)
    nb = np.linalg.norm(B.astype(np.clongdouble), axis=-2)
    tol = np.sqrt(4 * 33) * 2.0 ** -46.4 * na[..., :, None] * nb[..., None, :]
    assert np.all(np.abs(got - ref) <= tol + 33 * 2.0 ** -52 * np.abs(ref))


def test_ragged_groups_side_by_side_give_the_same_bits():
    from workloads import make_device
    systems = []
    for j, (N, b) in enumerate([(3, 40), (4, 24), (3, 56), (4, 24), (2, 30)]):
        d = make_device(N, b, 60 + j)
        E = torch.linspace(-0.4, 0.5, 3 + j, dtype=torch.float64, device="cuda")
        systems.append((torch.as_tensor(d.D, device="cuda"), torch.as_tensor(d.T, device="cuda"), E))
    opt = negf.options(precision=negf.PREC_MIXED, eta_lead=1e-3, eta_device=1e-3)
    one = negf.solve_ragged(systems, opt, concurrent=False)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side), torch.no_grad():
        two = negf.solve_ragged(systems, opt)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    for a, b in zip(one, two):
        for k, v in a.items():
            if isinstance(v, torch.Tensor):
                assert torch.equal(v, b[k]) and not b[k].requires_grad
    bad = systems[:2] + [(systems[2][0], systems[2][1], systems[2][2].float())]
    with pytest.raises(Exception):  # a group's error reaches the caller
        negf.solve_ragged(bad, opt)
    torch.cuda.synchronize()

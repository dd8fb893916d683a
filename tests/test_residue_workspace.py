"""The scratch of residue products: the sweeps reserve it for b x b blocks and then also contract over
the support of an interface coupling, any number of terms up to b."""
import pytest

import paper_1510_04686_gb300 as negf


@pytest.mark.parametrize("prec", [negf.PREC_MIXED, negf.PREC_MIXED_56])
@pytest.mark.parametrize("n", [12, 64])
def test_scratch_of_a_block_holds_every_shorter_contraction(prec, n):
    negf._build.build()
    lib = negf.library()
    gemm, inv = lib.negf_zgemm_workspace_size, lib.negf_zinv_workspace_size
    slack = 64 * 1024  # alignment of the pieces
    for b in (*range(8, 520, 37), *range(520, 660), *range(660, 2000, 61), 3430, 9266):
        # what an inverse needs beside its products' operands grows with the number of blocks; eleven
        # blocks take digit slices, whose scratch never grows with fewer terms
        rest = (inv(prec, 11, b) - gemm(prec, 11, b, b, b)) * n // 11
        have = inv(prec, n, b) - rest + slack
        for k in range(b, max(0, b - 200), -1):
            assert gemm(prec, n, b, b, k) <= have, (b, k)

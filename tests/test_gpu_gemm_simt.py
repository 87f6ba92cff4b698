"""The SIMT grouped GEMM at the sizes where its tile forms change and end: every operand layout with
a shape that takes each form (128-, 64- and 32-wide tiles), ragged in M, N and the k slice."""
import numpy as np
import pytest

from _gpu_common import built_package

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a_mn", [False, True])
@pytest.mark.parametrize("b_mn", [False, True])
@pytest.mark.parametrize("M,N,Kd,G", [(296, 520, 24, 13),   # 3 x 5 x 13 tiles of 128: that form
                                      (136, 1032, 40, 3),   # 3 x 17 x 3 tiles of 64
                                      (72, 136, 88, 2),     # fewer: tiles of 32
                                      (8, 264, 200, 40),    # at most 32 rows
                                      (1032, 24, 16, 5)])   # at most 32 columns
def test_simt_forms(M, N, Kd, G, a_mn, b_mn):
    import torch

    P = built_package()
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn(G, M, Kd, generator=g, device="cuda").bfloat16()
    B = torch.randn(G, N, Kd, generator=g, device="cuda").bfloat16()
    C = torch.full((G, M, N), float("nan"), device="cuda")
    P.lsgd_grouped_gemm_bf16(A.transpose(1, 2).contiguous() if a_mn else A, a_mn,
                             B.transpose(1, 2).contiguous() if b_mn else B, b_mn, C, M, N, Kd, G, engine=1)
    a, b = A.double(), B.double()
    want, scale = a @ b.transpose(1, 2), a.abs() @ b.abs().transpose(1, 2)
    # a chain of Kd fp32 multiply-adds: Kd 2^-24 of the sum of absolute products
    assert bool(((C.double() - want).abs() <= Kd * 2.0 ** -24 * scale).all())

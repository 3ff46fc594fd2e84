"""Operands of the tensor-core products split from windows of larger matrices: odd strides, odd starts, ragged columns."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402
from paper_2410_11596_gb300 import _lib as L  # noqa: E402

pytestmark = pytest.mark.gpu

# relative error of a product: 2^-21 (TF32x3) and 2^-16 (BF16x3) from the parts, times 8 for the
# FP32 accumulation over K <= 512, of sum_k |A_ik| |B_jk|
TOL = {L.HS_PREC_TF32X3: 2.0 ** -18, L.HS_PREC_BF16X3: 2.0 ** -13}


@pytest.fixture(scope="module")
def ctx():
    ensure_library()
    from paper_2410_11596_gb300.api import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("prec", sorted(TOL))
@pytest.mark.parametrize("M,N,K,offset,extra", [(1, 1, 1, 0, 0), (3, 2, 4, 1, 0), (33, 17, 31, 0, 1), (130, 70, 64, 1, 2),
                                               (257, 129, 66, 2, 2), (300, 5, 510, 0, 2)])
def test_windows(ctx, prec, M, N, K, offset, extra):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    ld = K + offset + extra
    A = torch.randn(M, ld, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, ld, dtype=torch.float64, device="cuda", generator=g)
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    L.check(L.load().hs_gemm(ctx.handle, prec, M, N, K, ctypes.c_void_p(A.data_ptr() + 8 * offset), ld,
                             ctypes.c_void_p(B.data_ptr() + 8 * offset), ld, ctypes.c_void_p(C.data_ptr()), N))
    ctx.sync()
    a, b = A[:, offset:offset + K], B[:, offset:offset + K]
    assert ((C - a @ b.T).abs() <= TOL[prec] * (a.abs() @ b.abs().T)).all()

"""Workspaces of the FP64 products: allocated by the first product that needs them."""
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402

pytestmark = pytest.mark.gpu


def test_unsplit_product_allocates_nothing():
    """1500 x 1500 x 4 is too short for the digit slices and has tiles enough not to split K: in a fresh context
    it leaves the free memory as it was (the splits' 32 MB workspace comes with a product that splits)."""
    ensure_library()
    from paper_2410_11596_gb300 import _lib as L
    from paper_2410_11596_gb300.api import Context
    g = torch.Generator(device="cuda").manual_seed(1)
    A, B = (torch.randint(-99, 100, (1500, 4), device="cuda", generator=g).double() for _ in range(2))
    P, Q = (torch.randint(-99, 100, (64, 4096), device="cuda", generator=g).double() for _ in range(2))
    C, D = (torch.empty(n, n, dtype=torch.float64, device="cuda") for n in (1500, 64))
    ref, ref2 = A @ B.T, P @ Q.T
    warm = Context(0)       # the kernels' modules are loaded by another context's products
    L.hs_gemm(warm.handle, L.HS_PREC_F64, A, B, C)
    L.hs_gemm(warm.handle, L.HS_PREC_F64, P, Q, D)
    warm.sync()
    c = Context(0)
    before = torch.cuda.mem_get_info()[0]
    L.hs_gemm(c.handle, L.HS_PREC_F64, A, B, C)
    c.sync()
    assert torch.cuda.mem_get_info()[0] == before
    assert torch.equal(C, ref)
    L.hs_gemm(c.handle, L.HS_PREC_F64, P, Q, D)     # splits K: takes the workspace
    c.sync()
    assert before - torch.cuda.mem_get_info()[0] >= 32 << 20
    assert torch.equal(D, ref2)
    c.close()
    warm.close()

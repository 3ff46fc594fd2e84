"""FP64 block GEMM (DFMA kernels) at the edges of its 16 x 16 and 64 x 64 tiles and of its K splits."""
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    ensure_library()
    from paper_2410_11596_gb300.api import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (15, 17, 16), (16, 16, 17), (17, 15, 31), (64, 64, 64), (65, 63, 15),
                                   (33, 200, 5), (110, 97, 2593), (20, 1000, 180), (300, 301, 33), (127, 129, 255)])
def test_integers_are_exact(ctx, M, N, K):
    """Integer operands up to 99: every sum is exact in FP64, whatever its order."""
    from paper_2410_11596_gb300 import _lib as L
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N * 3 + K)
    A = torch.randint(-99, 100, (M, K), device="cuda", generator=g).double()
    B = torch.randint(-99, 100, (N, K), device="cuda", generator=g).double()
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    L.hs_gemm(ctx.handle, L.HS_PREC_F64, A, B, C)
    ctx.sync()
    assert torch.equal(C, A @ B.T)

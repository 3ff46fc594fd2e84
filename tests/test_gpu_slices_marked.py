"""FP64 products on the tensor cores whose rows lie outside the digits' range, hold infinities or NaN, or keep too few
digits, one, some or all of them: the entries come from FP64 FMAs, row by row or, from a third of the work on, as the
whole product."""
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


# 64 x 64 tiles ragged on both sides; K = 600 takes a whole CTA a listed row, 4097 x 70 has too few tiles for the
# whole product (rows of length 700 there)
@pytest.mark.parametrize("M,N,K", [(2100, 1100, 40), (2049, 1111, 160), (1300, 1290, 600), (4097, 70, 700)])
@pytest.mark.parametrize("share", [0.0, 0.01, 0.32, 0.35, 1.0])
def test_rows_out_of_range(ctx, M, N, K, share):
    """Rows of A at 2^600 (their products with rows of B at 2^-600 are ordinary numbers): |C - A B^T| stays below the
    bound of two FP64 products, 2 K 2^-53 sum |A||B|; one NaN and one infinity change their row and column only."""
    from paper_2410_11596_gb300 import _lib as L
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K, dtype=torch.float64, device="cuda", generator=g)
    n = int(share * M)
    A[torch.randperm(M, device="cuda", generator=g)[:n]] *= 2.0 ** 600
    B *= 2.0 ** -300
    A[7, 3] = float("nan")
    B[N - 1, K - 1] = float("inf")
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    L.hs_profile_enable(ctx.handle, False)
    L.hs_gemm(ctx.handle, L.HS_PREC_F64, A, B, C)
    ctx.sync()
    assert L.hs_profile_read(ctx.handle)["launches"] >= 2       # the slices were launched
    ref, S = A @ B.T, A.abs() @ B.abs().T
    fin = torch.isfinite(ref)
    assert torch.equal(torch.isnan(C), torch.isnan(ref))
    assert torch.equal(C[~fin & ~torch.isnan(ref)], ref[~fin & ~torch.isnan(ref)])
    assert fin.sum() == (M - 1) * (N - 1)
    assert ((C - ref).abs()[fin] <= 2 * K * 2.0 ** -53 * (1 + 1e-10) * S[fin]).all()


def test_complex_product_of_marked_rows(ctx):
    """The two-site rho is of degree four in A: at 2^-240 A its edge product's rows lie at 2^-480, outside the digits'
    range, all of them (10000 x 100 x 5000, real and imaginary sources), and rho scales by 2^-960 exactly but for
    rounding (FP64 sums of 5000 terms, far below 1e-12 of the largest entry)."""
    import numpy as np

    from paper_2410_11596_gb300 import inputs
    from paper_2410_11596_gb300.api import CTMRG
    A = inputs.random_ipeps(2, 5, 77, True)
    c = CTMRG(ctx, A, 100)
    c.run(1)
    h = torch.eye(4, dtype=torch.float64, device="cuda")
    Ad = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    rho = c.rdm2_of(Ad, h)[0]
    low = c.rdm2_of(Ad * 2.0 ** -240, h)[0] * 2.0 ** 960
    assert (rho - low).abs().max() <= 1e-12 * rho.abs().max()

"""FP64 products on the tensor cores where large factors meet small ones: every entry keeps the error bound of a
chain of FP64 FMAs, K 2^-53 sum_k |A_mk| |B_nk|, however the operands are graded along the contraction."""
import numpy as np
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


def _operands(kind, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + 7 * K)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K, dtype=torch.float64, device="cuda", generator=g)
    k = torch.arange(K, dtype=torch.float64, device="cuda")
    if kind.startswith("opposite"):
        w = 10.0 ** (-float(kind[8:]) * k / max(K - 1, 1))
        return A * w, B * w.flip(0)
    if kind == "gauge":      # a bond's change of basis, by powers of two in no order
        s = torch.pow(2.0, torch.randint(-40, 41, (K,), device="cuda", generator=g).double())
        return A * s, B / s
    if kind == "halves":     # every second row lives in the first half of the indices, its partner's in the second
        first = (k < K / 2).double()
        big = lambda n: torch.where((torch.arange(n, device="cuda") % 2 == 0)[:, None], first, 1 - first)
        return A * (1e-9 + big(M)), B * (1e-9 + big(N))
    if kind == "outlier":    # equal entries (their roundings add up) under one large one, at different indices
        A = torch.full_like(A, 1.0 / 3.0)
        B = torch.full_like(B, 1.0 / 3.0)
        A[:, 0] = 1.0e3 * torch.randn(M, dtype=torch.float64, device="cuda", generator=g)
        B[:, K - 1] = 1.0e3 * torch.randn(N, dtype=torch.float64, device="cuda", generator=g)
        return A, B
    if kind == "disjoint":   # no term at all in most entries
        A[:, ::2] = 0.0
        B[1:, 1::2] = 0.0
        return A, B
    return A, B


KINDS = ["opposite0", "opposite2", "opposite4", "opposite8", "opposite16", "opposite300", "gauge", "halves", "outlier",
         "disjoint"]


# K steps are 32 wide, two share a piece of magnitudes, 14 a stage; K = 20 and 40 take a lane per column in
# the entries that are summed again, the others lanes over k
@pytest.mark.parametrize("M,N,K", [(4000, 1200, 20), (3000, 1201, 40), (2049, 1041, 128), (1023, 879, 257),
                                   (897, 561, 449), (700, 641, 2000)])
@pytest.mark.parametrize("kind", KINDS)
def test_error_bound_of_a_chain(ctx, M, N, K, kind):
    """On sampled entries against extended precision, and on the whole matrix against another FP64 product
    (whose own error has the same bound). Over random terms the error is also no larger than one rounding of
    sum |A||B|, in the mean: a chain's is a third of that."""
    from paper_2410_11596_gb300 import _lib as L
    A, B = _operands(kind, M, N, K)
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    L.hs_profile_enable(ctx.handle, False)
    L.hs_gemm(ctx.handle, L.HS_PREC_F64, A, B, C)
    ctx.sync()
    assert L.hs_profile_read(ctx.handle)["launches"] >= 2          # the slices ran
    S = A.abs() @ B.abs().T
    assert ((C - A @ B.T).abs() <= 2 * K * 2.0 ** -53 * S * (1 + 1e-10)).all()
    rows = np.unique(np.linspace(0, M - 1, 10).astype(int))
    cols = np.unique(np.linspace(0, N - 1, 40).astype(int))
    a, b = A.cpu().numpy()[rows].astype(np.longdouble), B.cpu().numpy()[cols].astype(np.longdouble)
    s = np.abs(a) @ np.abs(b).T
    err = np.abs(C.cpu().numpy()[np.ix_(rows, cols)].astype(np.longdouble) - a @ b.T)
    assert np.all(err <= K * 2.0 ** -53 * s)
    if kind != "outlier":
        rel = (err[s > 0] / s[s > 0]).astype(float)
        assert np.sqrt(np.mean(rel ** 2)) <= 2.0 ** -53

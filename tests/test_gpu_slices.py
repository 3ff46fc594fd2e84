"""FP64 products by digit slices on the tensor cores (k_gemm_sl.cu) through hs_gemm."""
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


def _gemm(ctx, A, B):
    """C = A B^T; asserts that the slices ran (their two launches are counted, the FP64 kernel's is not)."""
    from paper_2410_11596_gb300 import _lib as L
    C = torch.full((A.shape[0], B.shape[0]), 7.0, dtype=torch.float64, device="cuda")
    L.hs_profile_enable(ctx.handle, False)
    L.hs_gemm(ctx.handle, L.HS_PREC_F64, A, B, C)
    ctx.sync()
    assert L.hs_profile_read(ctx.handle)["launches"] >= 2
    return C


# tiles are 128 x 80, K steps 32 and the sums are drained every 192 columns; rows are read whole up to
# 64, 256 and 768 entries
@pytest.mark.parametrize("M,N,K", [(20001, 401, 17), (4096, 1200, 32), (4097, 1201, 33), (5001, 721, 64),
                                   (5001, 719, 65), (2049, 1041, 128), (2047, 1039, 129), (1920, 960, 192),
                                   (1921, 959, 193), (1025, 881, 256), (1023, 879, 257), (897, 561, 768),
                                   (895, 559, 769), (500, 500, 5000), (640, 640, 40001)])
@pytest.mark.parametrize("kind", ["normal", "decaying", "positive"])
def test_against_extended_precision(ctx, M, N, K, kind):
    """Per entry: an operand entry is off by at most 2^-55 of its row's largest, the pairs left out add
    less than 2^-58 per term (both rows' scales at most twice their largest entry), so
    |error| <= K 2^-51 max|A_m| max|B_n| plus the last rounding, and (checked on the whole matrix) the
    2-norm error is no larger than that of an FP64 chain."""
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K, dtype=torch.float64, device="cuda", generator=g)
    if kind == "decaying":
        w = torch.logspace(0, -6, K, dtype=torch.float64, device="cuda")
        A, B = A * w, B * w
    if kind == "positive":
        A, B = A.abs(), B.abs()
    C = _gemm(ctx, A, B).cpu().numpy()
    rows = np.unique(np.linspace(0, M - 1, 8).astype(int))
    cols = np.unique(np.linspace(0, N - 1, 24).astype(int))
    a, b = A.cpu().numpy()[rows].astype(np.longdouble), B.cpu().numpy()[cols].astype(np.longdouble)
    ref = a @ b.T
    err = np.abs(C[np.ix_(rows, cols)].astype(np.longdouble) - ref)
    bound = K * 2.0 ** -51 * np.abs(a).max(1)[:, None] * np.abs(b).max(1)[None, :] + 2.0 ** -52 * np.abs(ref)
    assert np.all(err <= bound)
    chain = np.abs((A @ B.T).cpu().numpy()[np.ix_(rows, cols)].astype(np.longdouble) - ref)
    assert np.linalg.norm(err.astype(float)) <= max(1.5 * np.linalg.norm(chain.astype(float)),
                                                    2.0 ** -53 * np.linalg.norm(ref.astype(float)))


def test_odd_strides_and_offsets(ctx):
    """Operands and result as windows of larger matrices: odd row strides, odd starts; nothing outside is written."""
    import ctypes

    from paper_2410_11596_gb300 import _lib as L
    M, N, K = 2051, 1043, 167
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn(M, K + 6, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K + 3, dtype=torch.float64, device="cuda", generator=g)
    C = torch.full((M + 2, N + 4), 7.0, dtype=torch.float64, device="cuda")
    L.check(L.load().hs_gemm(ctx.handle, L.HS_PREC_F64, M, N, K, ctypes.c_void_p(A.data_ptr() + 8), K + 6,
                             ctypes.c_void_p(B.data_ptr() + 16), K + 3,
                             ctypes.c_void_p(C[1:, 3:].data_ptr()), N + 4))
    ctx.sync()
    ref = A[:, 1:K + 1] @ B[:, 2:K + 2].T
    assert (C[1:M + 1, 3:N + 3] - ref).abs().max().item() <= K * 2.0 ** -51 * 25.0 * 2
    C[1:M + 1, 3:N + 3] = 7.0
    assert torch.all(C == 7.0)


def test_scales_zeros_and_non_finite_rows(ctx):
    """Rows of any scale, zero rows, and rows that hold infinities or NaN behave as in a chain of FP64 FMAs."""
    M, N, K = 2100, 1100, 160
    g = torch.Generator(device="cuda").manual_seed(6)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K, dtype=torch.float64, device="cuda", generator=g)
    A *= torch.pow(2.0, torch.arange(M, device="cuda", dtype=torch.float64) % 61 * 10 - 300)[:, None]
    A[7] = 0.0
    A[11] *= 2.0 ** -700 / A[11].abs().max()       # below the slices' range, products still normal
    A[13] *= 2.0 ** 900 / A[13].abs().max()        # above it
    A[17, 5] = float("inf")
    A[130, 0] = float("nan")
    B[3] = 0.0
    B[90, 159] = -float("inf")
    B[1099, 31] = float("nan")
    C, R = _gemm(ctx, A, B), A @ B.T
    assert torch.equal(torch.isnan(C), torch.isnan(R))
    assert torch.equal(torch.isinf(C), torch.isinf(R))
    inf = torch.isinf(R)
    assert torch.equal(C[inf], R[inf])
    fin = torch.isfinite(R)
    ra = torch.nan_to_num(A, nan=0.0, posinf=0.0, neginf=0.0).abs().amax(1, keepdim=True)
    rb = torch.nan_to_num(B, nan=0.0, posinf=0.0, neginf=0.0).abs().amax(1, keepdim=True)
    bound = 2.0 * K * 2.0 ** -51 * (ra * rb.T)
    assert torch.all((C - R).abs()[fin] <= bound[fin])
    assert torch.all(C[7][torch.isfinite(B).all(1)] == 0.0)

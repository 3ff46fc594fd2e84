"""FP64 products on the tensor cores in row panels, accumulating and complex, and the ways around them: no workspace,
a stream under capture; and the HOTRG step with two solvers at once."""
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def ctx():
    ensure_library()
    from paper_2410_11596_gb300.api import Context
    c = Context(0)
    yield c
    c.close()


def _rand(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _rows(x, g):
    """Some rows out of the digits' range and some whose first and last entries trade places: listed entries in
    every panel, at its edges too."""
    x[::511] *= 2.0 ** 510
    x[1::257, : x.shape[1] // 2] *= 2.0 ** -40
    return x


# digits take 4.8 KB a row at K = 300: whole; panels of A; of B; of both; no room for one block of each
@pytest.mark.parametrize("M,N,K,cap,pairs", [(3001, 901, 300, 1 << 30, (1, 1)), (3001, 901, 300, 16 * MB, (2, 4)),
                                             (500, 3001, 300, 13 * MB, (2, 4)), (3001, 1901, 300, 8 * MB, (6, 40)),
                                             (3001, 901, 300, MB // 2, (0, 0)), (3001, 901, 300, 0, (0, 0))])
@pytest.mark.parametrize("accumulate", [False, True])
def test_panels(ctx, M, N, K, cap, pairs, accumulate):
    """Every panel edge, with listed entries among them: within the bound of two FP64 products, 2 K 2^-53
    sum |A||B|, and the rounding of the sum with C; repeated, the same bits."""
    from paper_2410_11596_gb300 import _lib as L
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A, B = _rows(_rand(g, M, K), g), _rand(g, N, K) * 2.0 ** -300
    C0 = _rand(g, M, N) * 2.0 ** -300
    C, D = C0.clone(), C0.clone()
    n = L.hs_selftest_gemm_f64(ctx.handle, A, B, C, cap, accumulate=accumulate)
    assert pairs[0] <= n <= pairs[1]
    L.hs_selftest_gemm_f64(ctx.handle, A, B, D, cap, accumulate=accumulate)
    ctx.sync()
    assert torch.equal(C, D)
    ref, S = A @ B.T, A.abs() @ B.abs().T
    if accumulate:
        ref = ref + C0
    tol = 2 * K * 2.0 ** -53 * S + 4 * 2.0 ** -53 * (C0.abs() if accumulate else 0) + 2.0 ** -52 * ref.abs()
    assert ((C - ref).abs() <= tol * (1 + 1e-10)).all()


@pytest.mark.parametrize("cap,pairs", [(1 << 30, (1, 1)), (20 * MB, (2, 12))])
@pytest.mark.parametrize("conj", [False, True])
def test_complex_panels(ctx, cap, pairs, conj):
    """Two sources an operand (300 columns each), ragged segments: as above for each part, sums over both sources."""
    from paper_2410_11596_gb300 import _lib as L
    M, N, K = 2001, 701, 301
    g = torch.Generator(device="cuda").manual_seed(11)
    Ar, Ai, Br, Bi = _rows(_rand(g, M, K), g), _rand(g, M, K), _rand(g, N, K), _rows(_rand(g, N, K), g) * 2.0 ** -300
    Cr, Ci = (torch.full((M, N), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    n = L.hs_selftest_gemm_f64(ctx.handle, (Ar, Ai), (Br, Bi), (Cr, Ci), cap, conj_b=conj)
    ctx.sync()
    assert pairs[0] <= n <= pairs[1]
    s = -1.0 if conj else 1.0
    for c, ref, size in ((Cr, Ar @ Br.T - s * (Ai @ Bi.T), Ar.abs() @ Br.abs().T + Ai.abs() @ Bi.abs().T),
                         (Ci, s * (Ar @ Bi.T) + Ai @ Br.T, Ar.abs() @ Bi.abs().T + Ai.abs() @ Br.abs().T)):
        assert ((c - ref).abs() <= 2 * (2 * K + 1) * 2.0 ** -53 * size * (1 + 1e-10)).all()


def test_largest_panels_of_the_chains(ctx):
    """The bra step of a D = 6, chi = 144 density matrix, 1.34 GB of digits: the workspace's own limit cuts it."""
    from paper_2410_11596_gb300 import _lib as L
    M, N, K = 1492992, 72, 36
    g = torch.Generator(device="cuda").manual_seed(12)
    A, B = _rand(g, M, K), _rand(g, N, K)
    C = torch.empty(M, N, dtype=torch.float64, device="cuda")
    assert L.hs_selftest_gemm_f64(ctx.handle, A, B, C, 1 << 40) > 1
    ctx.sync()
    for r in range(0, M, 1 << 18):
        a = A[r: r + (1 << 18)]
        assert ((C[r: r + (1 << 18)] - a @ B.T).abs() <= 2 * K * 2.0 ** -53 * (a.abs() @ B.abs().T) * (1 + 1e-10)).all()


def test_product_under_capture():
    """A stream under capture gets the FP64 kernel, which needs no workspace that a later call could move: the graph
    gives the product of the operands' values at each replay, also after a larger product on the context."""
    ensure_library()
    from paper_2410_11596_gb300 import _lib as L
    from paper_2410_11596_gb300.api import Context
    ctx = Context(0, torch.cuda.Stream())
    g = torch.Generator(device="cuda").manual_seed(13)
    M, N, K = 1200, 800, 200
    A, B = (torch.randint(-99, 100, (n, K), device="cuda", generator=g).double() for n in (M, N))
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    big, out = _rand(g, 4000, 2000), torch.empty(4000, 4000, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    L.hs_gemm(ctx.handle, L.HS_PREC_F64, A, B, C)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=ctx.stream):
        L.hs_gemm(ctx.handle, L.HS_PREC_F64, A, B, C)
    L.hs_gemm(ctx.handle, L.HS_PREC_F64, big, big, out)
    torch.cuda.synchronize()
    A.copy_(torch.randint(-99, 100, (M, K), device="cuda", generator=g).double())
    C.fill_(7.0)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, A @ B.T)
    ctx.close()


def test_hotrg_with_two_solvers_at_once(ctx):
    """One pair of eigen-decompositions after the other gives what four at once give (the same library call on
    the same blocks): the same sides, sectors and ln Z."""
    from paper_2410_11596_gb300 import _lib as L, inputs
    from paper_2410_11596_gb300.api import HOTRG
    runs = []
    for at_once in (4, 2):
        L.hs_selftest_hotrg_solvers(ctx.handle, at_once)
        h = HOTRG(ctx, inputs.asymmetric_ipeps(2, 3, 5), 12)
        h.run(3)
        runs.append((h.log_z_per_site(), [(i["side"], i["h_even"], i["h_odd"]) for i in h.infos]))
    L.hs_selftest_hotrg_solvers(ctx.handle, 4)
    assert runs[0][1] == runs[1][1]
    assert runs[0][0] == pytest.approx(runs[1][0], rel=1e-12)

"""The two-site chain and its adjoint at physical and bond dimensions where its kernels' index maps differ."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402
from oracle import ctmrg as oc, doublelayer as dl, observables as ob  # noqa: E402
from paper_2410_11596_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    ensure_library()
    from paper_2410_11596_gb300.api import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("d,D,chi,moves", [(1, 2, 3, 2), (3, 2, 5, 3), (2, 3, 10, 2), (3, 3, 7, 2), (2, 4, 33, 1)])
@pytest.mark.parametrize("complex_valued", [False, True])
def test_rho_and_eps_match_the_oracle(ctx, d, D, chi, moves, complex_valued):
    """rho and rho1 up to their common factor (the normalisation of C and T) and eps, 1e-10 as the other
    FP64 observables."""
    from paper_2410_11596_gb300.api import CTMRG
    A = inputs.random_ipeps(d, D, 40 + d + D, complex_valued)
    r = oc.run(dl.double_layer(A), chi, moves)
    c = CTMRG(ctx, A, chi)
    c.run(moves)
    rho = c.rdm2(np.eye(d * d))[0].cpu().numpy()
    ref = ob.two_site_rdm(r.C, r.T, A)
    np.testing.assert_allclose(rho / np.trace(rho), ref / np.trace(ref), atol=1e-10)
    eps, eref = c.one_site_env().cpu().numpy(), ob.one_site_environment(r.C, r.T)
    np.testing.assert_allclose(eps / np.abs(eps).max(), eref / np.abs(eref).max(), atol=1e-10)


@pytest.mark.parametrize("d,D,moves,complex_valued", [(1, 2, 1, False), (2, 3, 1, False), (3, 2, 1, True),
                                                      (2, 3, 1, True), (3, 3, 1, False), (1, 11, 0, True)])
def test_adjoint_is_the_transpose_of_the_derivative(ctx, d, D, moves, complex_valued):
    """rho is a polynomial of degree four in A (with its conjugate), so the five-point formula
    (8 (f(1) - f(-1)) - (f(2) - f(-2))) / 12 is its exact derivative along a direction; paired with a random
    cotangent it equals the pairing of the direction with the adjoint. FP64 on both sides: the formula's
    differences lose at most three digits of sums of the size of rho. A is not C4v-symmetric here. The last
    case is the one whose rows of the open double layer do not fit in shared memory."""
    from paper_2410_11596_gb300.api import CTMRG
    A0 = inputs.random_ipeps(d, D, 60 + d + D, complex_valued)
    c = CTMRG(ctx, A0, D * D if moves == 0 else 6, complex_valued=complex_valued)
    c.run(moves)
    dt = torch.complex128 if complex_valued else torch.float64
    g = torch.Generator(device="cuda").manual_seed(9)
    A, v = (torch.randn((d, D, D, D, D), dtype=dt, device="cuda", generator=g) for _ in range(2))
    n = d * d
    w = torch.randn((n, n), dtype=dt, device="cuda", generator=g)
    h = torch.eye(n, dtype=torch.float64, device="cuda")

    def f(t):
        # the mirrored triangle of the real Hermitian-basis rho is left out by pairing with the upper one only
        rho = c.rdm2_of(A + t * v, h)[0]
        return rho if complex_valued else torch.triu(rho)

    def pair(x, y):
        return torch.real((x.conj() * y).sum()).item()

    wt = w if complex_valued else torch.triu(w)
    want = pair(wt, (8 * (f(1) - f(-1)) - (f(2) - f(-2))) / 12)
    got = pair(c.rdm2_vjp(A, wt), v)
    scale = pair(wt.abs(), f(2).abs() + f(-2).abs())
    assert abs(got - want) <= 1e-12 * scale

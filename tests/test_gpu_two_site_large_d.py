"""The two-site density matrix and its adjoint at a large physical dimension, where the chain's largest intermediates
are made in ranges of their leading index."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402
from paper_2410_11596_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("complex_valued,chi", [(False, 256), (True, 225)])
def test_isometry_on_the_physical_leg(complex_valued, chi):
    """A' = W A with an isometry W from d = 2 to d' = 26 has the environment of A, rho' = (W x W) rho (W x W)^+ and
    W^+ dA' = dA for the cotangent (W x W)^+ w' (W x W). c^2 d'^2 q^2 is 6 to 7 e8 entries: two ranges. Sums of at
    most 1e5 terms on both sides: 1e-12 of the largest entry."""
    ensure_library()
    from paper_2410_11596_gb300.api import CTMRG, Context
    ctx = Context(0)
    A = inputs.random_ipeps(2, 2, 91, complex_valued)
    c = CTMRG(ctx, A, chi, complex_valued=complex_valued)
    c.run(4)
    assert c.env.chi_even + c.env.chi_odd == chi
    dt = torch.complex128 if complex_valued else torch.float64
    g = torch.Generator(device="cuda").manual_seed(92)
    d = 26 if not complex_valued else 30
    W = torch.linalg.qr(torch.randn(d, 2, dtype=dt, device="cuda", generator=g))[0]
    A2 = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    Ad = torch.tensordot(W, A2, dims=([1], [0])).contiguous()
    W2 = torch.kron(W, W)

    def eye(n):
        return torch.eye(n, dtype=torch.float64, device="cuda")

    def large(call, *args):     # the environment does not depend on d
        c.d = d
        try:
            return call(*args)
        finally:
            c.d = 2

    rho, rhod = c.rdm2_of(A2, eye(4))[0], large(c.rdm2_of, Ad, eye(d * d))[0]
    want = W2 @ rho.to(dt) @ W2.mH
    assert (rhod - want).abs().max() <= 1e-12 * want.abs().max()
    w = torch.randn(d * d, d * d, dtype=dt, device="cuda", generator=g)
    small = W2.mH @ w @ W2
    got = torch.tensordot(W.mH, large(c.rdm2_vjp, Ad, w), dims=([1], [0]))
    ref = c.rdm2_vjp(A2, small.contiguous())
    assert (got - ref).abs().max() <= 1e-12 * ref.abs().max()
    ctx.close()

"""HOTRG steps whose tensors fall off by many decades (FP64 products held to their rows' scale)."""
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library  # noqa: E402
from oracle import doublelayer as dl, hotrg as oh  # noqa: E402
from paper_2410_11596_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,chi,steps", [(2, 16, 12), (4, 16, 9)])
@pytest.mark.parametrize("basis", ["hermitian", "dense"])
def test_log_z_of_late_steps(D, chi, steps, basis):
    """ln Z per site against the oracle: steps of orthogonal transformations and sums of up to chi^4 terms, 1e-11
    leaves room for 2^-53 chi^2 a step and the truncations' first-order change."""
    ensure_library()
    from paper_2410_11596_gb300.api import Context, HOTRG
    ctx = Context(0)
    A = inputs.random_ipeps(2, D, inputs.SEED_BASE + 40 + D)
    h = HOTRG(ctx, A, chi, basis=basis)
    h.run(steps)
    r = oh.run(dl.double_layer(A), chi, steps)
    assert h.log_z_per_site() == pytest.approx(oh.log_z_per_site(r), rel=1e-11)
    ctx.close()

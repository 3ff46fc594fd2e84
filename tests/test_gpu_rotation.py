"""Rotation of a dense double layer into the Hermitian basis: every bond dimension from 1, odd and even, and
what the call does with blocks that may not exist."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ensure_library, fso_pack  # noqa: E402
from oracle import basis as ba  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    ensure_library()
    from paper_2410_11596_gb300.api import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7])
def test_rotation_of_any_dense_tensor(ctx, D):
    """A dense tensor with no symmetry: the even-total blocks are the oracle's rotation (sums of 16 terms,
    2e-15 of the largest), the tolerance decides about the odd ones."""
    from paper_2410_11596_gb300 import _lib as L
    q = D * D
    rng = np.random.default_rng(70 + D)
    a = rng.standard_normal((q, q, q, q))
    U = ba.hermitian_basis(D)
    t = a
    for ax in range(4):
        t = np.moveaxis(np.tensordot(U.T, t, axes=([1], [ax])), 0, ax)
    s = ba.sector_dims(D)
    ad = torch.from_numpy(a).cuda()
    out = torch.full((L.hs_z2_tensor_bytes(D, L.HS_BASIS_HERMITIAN, L.HS_F64) // 8,), 7.0, dtype=torch.float64,
                     device="cuda")
    L.hs_to_hermitian_basis(ctx.handle, ad, D, L.HS_F64, 2.0, out)
    ref = fso_pack(t, [s, s], [s, s])
    np.testing.assert_allclose(out.cpu().numpy()[:ref.size], ref, atol=2e-15 * np.abs(t).max() * 4)
    if D > 1:
        p = ba.sector_parities(D)
        odd = (p[:, None, None, None] + p[:, None, None] + p[:, None] + p) % 2 == 1
        ratio = np.abs(t[odd]).max() / np.abs(t).max()
        L.hs_to_hermitian_basis(ctx.handle, ad, D, L.HS_F64, ratio * (1 + 1e-12), out)
        with pytest.raises(L.HsError):
            L.hs_to_hermitian_basis(ctx.handle, ad, D, L.HS_F64, ratio * (1 - 1e-12), out)

"""The gradient of A is g times a sum over the slots: a large (small) cotangent with
a small (large) sum leaves the range of the dtype nowhere on the way.

Powers of two throughout and U, V (the columns of B) on entries that A^{-1} does not
couple, so R = 1 (M = C^{-1}) and every entry of the gradient is exact.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [torch.float32, torch.complex64, torch.float64, torch.complex128])
@pytest.mark.parametrize("kind", ["det", "pf"])
@pytest.mark.parametrize("exps", [(100, 32, -75), (-100, -60, 50), (0, 1, -2)])
def test_cotangent_and_factor_of_opposite_size(dt, kind, exps):
    """A^{-1} = 1 / a: the factors A^{-1} u = X and v A^{-1} = Y (B: X and Y)."""
    L = lrugb()
    n, h = 34, 17
    g, X, Y = (2.0 ** (e * (8 if dt in (torch.float64, torch.complex128) else 1)) for e in exps)
    a = 1.0 / X
    u, v = np.zeros(n), np.zeros(n)
    u[:8], v[8:h] = 1.0, Y / X
    st = L.LowRankState(kind, 1, n, dtype=dt)
    gv = tdev(np.array([g]), dt)
    if kind == "det":
        st.init(tdev(a * np.eye(n)[None], dt))
        st.propose_det(L.Operand(dense=tdev(u[None, None], dt)), L.Operand(dense=tdev(v[None, None], dt)))
        _, _, gA = st.backward_det(gv, want_U=False, want_V=False)
        # gA_ij = -g X_j Y_i
        want = -g * np.outer(v * X, u * X)
    else:
        J = np.kron(np.array([[0.0, 1.0], [-1.0, 0.0]]), np.eye(h))
        st.init(tdev(a * J[None], dt))
        st.propose_pf(L.Operand(dense=tdev(np.stack([u, v])[None], dt)))
        _, _, gA = st.backward_pf(gv, want_B=False, want_C=False)
        # gA = -(g / 2) X M^{-1} X^T with X = A^{-1} B = -J B / a, M^{-1} = -J_2
        Xb = -J @ np.stack([u, v], 1) * X
        want = -g / 2 * (Xb @ np.array([[0.0, -1.0], [1.0, 0.0]]) @ Xb.T)
    assert np.count_nonzero(want) > 0
    assert np.array_equal(gA[0].cpu().numpy(), want.astype(gA.cpu().numpy().dtype))

"""A Pfaffian proposal whose 2 x 2 core is not a number has ratio 0 and the status of a
singular core, in the closed form (C = -J) as in the general one (C given)."""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [torch.float64, torch.complex128, torch.float32, torch.complex64])
@pytest.mark.parametrize("delay", [0, 4])
def test_core_not_a_number(dt, delay):
    L = lrugb()
    W, n = 4, 6
    J = np.kron(np.array([[0.0, 1.0], [-1.0, 0.0]]), np.eye(n // 2))
    B = np.random.Generator(np.random.PCG64(1)).standard_normal((W, 2, n)) * 0.2
    B[1, 0, 2] = np.nan
    B[2, 1, :] = np.nan
    C = np.tile(np.array([[0.0, -1.0], [1.0, 0.0]]), (W, 1, 1))
    out = []
    for Cm in (None, tdev(C, dt)):
        st = L.LowRankState("pf", W, n, dtype=dt, delay=delay)
        st.init(tdev(np.tile(J, (W, 1, 1)), dt))
        r, s = st.propose_pf(L.Operand(dense=tdev(B, dt)), Cm)
        out.append((r.cpu().numpy(), s.cpu().numpy()))
    for r, s in out:
        assert s.tolist() == [0, 1, 1, 0]
        assert (r[1:3] == 0).all(), r
    np.testing.assert_allclose(out[0][0], out[1][0], rtol=1e-5)

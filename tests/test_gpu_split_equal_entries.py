"""Split products of vectors whose 64 entries are equal: every digit product of a
level has one sign, so the level sums are the largest there are.

An entry is -64 x y (or 1 less 64 x y) of two doubles, which the split
represents exactly; the dropped levels are below 2^-60 of it, so the result is
the correctly rounded one to within an ulp: 2 eps is asked.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16
n = 128


def pairs(W):
    g = np.random.Generator(np.random.PCG64(5))
    x, y = g.uniform(0.5, 1.0, W), g.uniform(0.5, 1.0, W)
    x[0], y[0] = 0.8067569554883454, 0.9431953105245781
    return x, y


@pytest.mark.parametrize("K", [16, 32, 48, 64])
def test_flush_of_equal_slots(K):
    """A_0 = 1, K moves U = x (rows 64 ..), V = y (columns .. 63): nilpotent, so P = x, Q = y exactly."""
    L = lrugb()
    W = 1024
    x, y = pairs(W)
    st = L.LowRankState("det", W, n, delay=K, flush=L.FLUSH_SPLIT)
    st.init(torch.eye(n, dtype=torch.float64, device="cuda").expand(W, n, n).contiguous())
    U, V = np.zeros((W, 1, n)), np.zeros((W, 1, n))
    U[:, 0, 64:] = x[:, None]
    V[:, 0, :64] = y[:, None]
    U, V = L.Operand(dense=tdev(U)), L.Operand(dense=tdev(V))
    for _ in range(K):
        st.propose_det(U, V)
        st.accept()
    assert (st.tau() == 0).all()
    inv = st.inverse()[:, 64:, :64].cpu().numpy()
    want = -(K * (x * y))[:, None, None]
    assert (np.abs(inv / want - 1)).max() <= 2 * EPS, np.abs(inv / want - 1).max()


@pytest.mark.parametrize("dt", [torch.float64, torch.complex128])
def test_elimination_of_equal_blocks(dt):
    """A = [[1, y], [x, D]] with constant 64 x 64 blocks x, y and D = 64 x y + 1/2 on the
    diagonal, 64 x y off it: the first panel (two for complex scalars) leaves D - 64 x y, off
    by one rounding of 64 x y < 64, 2^-48 per entry.  det = (1/2)^64 (1 + 2 sum of the errors / 64 ..),
    so log|det| may be off by 2 * 64 * 2^-48; an entry of the inverse by 4 * 64 * 2^-48 * 64 x y."""
    L = lrugb()
    W = 512
    x, y = pairs(W)
    A = np.tile(np.eye(n), (W, 1, 1))
    A[:, :64, 64:] = y[:, None, None]
    A[:, 64:, :64] = x[:, None, None]
    A[:, 64:, 64:] = 64 * (x * y)[:, None, None] + 0.5 * np.eye(64)
    D = A[:, 64:, 64:].astype(np.longdouble) - 64 * (x.astype(np.longdouble) * y)[:, None, None]
    E = D - 0.5 * np.eye(64)                       # 2^-48: (D)^{-1} = 2 - 4 E to 2^-90
    want = -64 * np.log(2.0) + 2 * np.trace(E, axis1=1, axis2=2)
    _, logabs = L.slogdet_batched(tdev(A, dt))
    assert np.abs(logabs.cpu().numpy() - want.astype(float)).max() <= 2 * 64 * 2.0 ** -48
    st = L.LowRankState("det", W, n, dtype=dt)
    st.init(tdev(A.transpose(0, 2, 1), dt))        # the elimination takes the transpose
    got = st.inverse().cpu().numpy()[:, 64:, 64:].transpose(0, 2, 1)
    inv = (2 * np.eye(64) - 4 * E).astype(float)
    assert np.abs(got - inv).max() <= 4 * 64 * 2.0 ** -48

"""Inverses of many small F64 matrices, just above the counts from which they are
eliminated on padded copies, against numpy and against the FP64 form.

Bound: condition below about 20; 32 n eps of the largest entry.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


@pytest.mark.parametrize("kind", ["det", "pf"])
@pytest.mark.parametrize("n,W", [(56, 160), (58, 700), (62, 160), (72, 310), (78, 700)])
def test_inverse_and_gradient(kind, n, W):
    L = lrugb()
    g = np.random.Generator(np.random.PCG64(n + W))
    A = 0.35 * g.standard_normal((5, n, n)) / np.sqrt(2 * n)
    for w in range(5):
        p = g.permutation(n)
        if kind == "pf":
            A[w] -= A[w].T
            A[w, p[0::2], p[1::2]] += 1.0
            A[w, p[1::2], p[0::2]] -= 1.0
        else:
            A[w, np.arange(n), p] += 1.0
    want = np.linalg.inv(A)
    x = tdev(A).repeat(W // 5, 1, 1).contiguous()
    out = []
    for refresh in (L.REFRESH_AUTO, L.REFRESH_FP64):
        st = L.LowRankState(kind, W, n, refresh=refresh)
        st.init(x)
        inv = st.inverse().cpu().numpy().reshape(W // 5, 5, n, n)
        assert np.abs(inv - want).max() <= 32 * n * EPS * max(1.0, np.abs(want).max())
        out.append(inv)
    assert not np.array_equal(out[0], out[1])     # two forms, one result to rounding
    y = x.clone().requires_grad_()
    (gA,) = torch.autograd.grad((L.slogdet if kind == "det" else L.slogpf)(y)[1].sum(), y)
    scale = 1.0 if kind == "det" else 0.5
    got = gA.cpu().numpy().reshape(W // 5, 5, n, n)
    assert np.abs(got - scale * want.transpose(0, 2, 1)).max() <= 32 * n * EPS * max(1.0, np.abs(want).max())

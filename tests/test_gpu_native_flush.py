"""The native delayed flush of large handles (exact split products) against the
FP64 tiles that a handle of few walkers of the same matrices takes: sizes that
no tile divides, both kinds and scalars, ranks, forced partial flushes under a
mask, slots of very different and of extreme size.

Both round an FP64 update of K k products, and the second window of slots starts
from that difference, amplified by at most the condition number (below 10): entries
may differ by 64 K k eps of the largest entry
of the walker's inverse.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


def setup(kind, cplx, n, W, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.complex128 if cplx else torch.float64
    A = 0.3 * torch.randn(W, n, n, generator=g, device="cuda", dtype=dt) / n ** 0.5
    if kind == "pf":
        A = A - A.transpose(1, 2)
        A[:, torch.arange(0, n, 2), torch.arange(1, n, 2)] += 1.0
        A[:, torch.arange(1, n, 2), torch.arange(0, n, 2)] -= 1.0
    else:
        A = A + torch.eye(n, device="cuda", dtype=dt)
    vec = lambda *sh: torch.randn(*sh, generator=g, device="cuda", dtype=dt) / n ** 0.5  # noqa: E731
    return dt, A.contiguous(), vec


@pytest.mark.parametrize("kind,cplx,n,k,K", [("det", False, 128, 1, 4), ("det", False, 130, 2, 8), ("det", False, 191, 1, 2),
                                             ("det", False, 257, 4, 16), ("det", True, 129, 1, 4), ("det", True, 192, 2, 16),
                                             ("pf", False, 128, 1, 8), ("pf", False, 146, 2, 4), ("pf", True, 130, 1, 16)])
def test_split_against_fp64_tiles(kind, cplx, n, k, K):
    L = lrugb()
    few, kk = 5, 2 * k if kind == "pf" else k
    W = (1 << 24) // (n * n * kk * (4 if cplx else 1)) + 1
    dt, A, vec = setup(kind, cplx, n, W, n + K)
    sts = [L.LowRankState(kind, w, n, k=k, dtype=dt, delay=K) for w in (W, few)]
    for st, w in zip(sts, (W, few)):
        st.init(A[:w].contiguous())
    steps = K + K // 2
    for t in range(steps):
        U, V = vec(W, kk, n), vec(W, kk, n)
        U[1] *= 1e-4                       # a walker whose slots are of very different size
        if t % 2:
            V[1] *= 1e3
        for st, w in zip(sts, (W, few)):
            if kind == "pf":
                st.propose_pf(L.Operand(dense=U[:w].contiguous()))
            else:
                st.propose_det(L.Operand(dense=U[:w].contiguous()), L.Operand(dense=V[:w].contiguous()))
            st.accept()
    for forced in (False, True):
        if forced:
            mask = torch.tensor([1, 0, 1, 1, 0], dtype=torch.uint8, device="cuda")
            sts[0].flush(torch.cat([mask, torch.zeros(W - few, dtype=torch.uint8, device="cuda")]))
            sts[1].flush(mask)
        assert torch.equal(sts[0].tau()[:few], sts[1].tau())
        a, b = sts[0].inverse()[:few], sts[1].inverse()
        for w in range(few):
            # both start from the same elimination, so the chains differ by the flushes alone
            tol = 64 * K * kk * EPS * b[w].abs().max()
            assert (a[w] - b[w]).abs().max() <= tol, (w, (a[w] - b[w]).abs().max(), tol)
        if kind == "pf" and forced:
            on = mask.bool()    # the others still have pending slots
            assert torch.equal(a[on], -a[on].transpose(1, 2))
    sts[0].check_device_error()


def test_slots_beyond_the_scale_range():
    """A = 1e-150 B: slots near 1e150 take the FP64 fold inside the slicing kernel."""
    L = lrugb()
    n, K = 128, 4
    W = (1 << 24) // (n * n) + 1
    dt, A, vec = setup("det", False, n, W, 1)
    A[2] *= 1e-150
    st = L.LowRankState("det", W, n, dtype=dt, delay=K)
    st.init(A)
    cur = A[:3].cpu().numpy().copy()
    for _ in range(K):
        U, V = vec(W, 1, n), vec(W, 1, n)
        V[2] *= 1e-150
        st.propose_det(L.Operand(dense=U), L.Operand(dense=V))
        st.accept()
        cur += U[:3].cpu().numpy().transpose(0, 2, 1) @ V[:3].cpu().numpy()
    assert (st.tau() == 0).all()
    want = np.stack([np.linalg.inv(cur[0]), np.linalg.inv(cur[1]), np.linalg.inv(cur[2] * 1e150) * 1e150])
    got = st.inverse()[:3].cpu().numpy()
    for w in range(3):
        assert np.abs(got[w] - want[w]).max() <= 64 * n * EPS * np.abs(want[w]).max()

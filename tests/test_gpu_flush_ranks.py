"""Uniform n with a rank per walker below the handle's: a flush of partly filled
slots reads the columns its walker has filled and no others, and so does the
drift of a refresh.

The handle of W walkers takes the split-product flush (W n^2 kk cx^2 >= 2^24) and
the padded elimination, the one of a few walkers FP64 tiles and the FP64
elimination.  Both round FP64 updates of K kk products and inverses of condition
number below 10: entries may differ by 64 K kk eps + 32 n eps of the walker's largest.
"""
import pytest

from gpu_common import lrugb, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


def build(kind, cplx, n, k, K):
    g = torch.Generator(device="cuda").manual_seed(n + K)
    dt = torch.complex128 if cplx else torch.float64
    few, kk = 6, 2 * k if kind == "pf" else k
    W = (1 << 24) // (n * n * kk * (4 if cplx else 1)) + 1
    A = 0.3 * torch.randn(W, n, n, generator=g, device="cuda", dtype=dt) / n ** 0.5
    if kind == "pf":
        A = A - A.transpose(1, 2)
        A[:, torch.arange(0, n, 2), torch.arange(1, n, 2)] += 1.0
        A[:, torch.arange(1, n, 2), torch.arange(0, n, 2)] -= 1.0
    else:
        A = A + torch.eye(n, device="cuda", dtype=dt)
    ranks = [w % k + 1 for w in range(W)]
    L = lrugb()
    sts = [L.LowRankState(kind, w, n, k=k, dtype=dt, delay=K, k_per_walker=ranks[:w], refresh=r)
           for w, r in ((W, L.REFRESH_AUTO), (few, L.REFRESH_FP64))]
    for st in sts:
        st.init(A[:st.W].contiguous())

    def step(accept=None):
        U, V = (torch.randn(W, kk, n, generator=g, device="cuda", dtype=dt) / n ** 0.5 for _ in range(2))
        for st in sts:
            u, v = (L.Operand(dense=x[:st.W].contiguous()) for x in (U, V))
            st.propose_pf(u) if kind == "pf" else st.propose_det(u, v)
            st.accept(None if accept is None else accept[:st.W].contiguous())

    return sts, A, step, few, (64 * K * kk + 32 * n) * EPS


def same(sts, few, tol):
    a, b = sts[0].inverse()[:few], sts[1].inverse()
    for w in range(few):
        assert (a[w] - b[w]).abs().max() <= tol * b[w].abs().max(), (w, (a[w] - b[w]).abs().max())


CASES = [("det", False, 128, 2, 4), ("det", False, 130, 4, 8), ("det", True, 129, 2, 4), ("pf", False, 130, 2, 4),
         ("pf", True, 128, 2, 4)]


@pytest.mark.parametrize("kind,cplx,n,k,K", CASES)
def test_partial_flush(kind, cplx, n, k, K):
    sts, _, step, few, tol = build(kind, cplx, n, k, K)
    for _ in range(K):
        step()
    same(sts, few, tol)
    step(torch.tensor([1, 1, 0, 1, 1, 0] + [1] * (sts[0].W - few), dtype=torch.uint8, device="cuda"))
    step()
    mask = torch.tensor([1, 0, 1, 1, 1, 1] + [0] * (sts[0].W - few), dtype=torch.uint8, device="cuda")
    for st in sts:
        st.flush(mask[:st.W].contiguous())
    assert torch.equal(sts[0].tau()[:few], sts[1].tau())
    same(sts, few, tol)
    sts[0].check_device_error()


@pytest.mark.parametrize("kind,cplx,n,k,K", CASES)
def test_drift_of_pending_slots(kind, cplx, n, k, K):
    sts, A, step, few, tol = build(kind, cplx, n, k, K)
    for _ in range(K + K // 2):
        step()
    drift = [st.refresh(A[:st.W].contiguous())[:few] for st in sts]
    assert (drift[0] - drift[1]).abs().max() <= tol * max(1.0, drift[1].abs().max().item()), drift
    same(sts, few, tol)

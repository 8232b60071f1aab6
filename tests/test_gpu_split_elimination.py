"""The split-product elimination on padded copies (Pfaffian and complex handles,
sizes that are no multiple of 128, the standalone slogdet and its backward)
against numpy and the FP64 elimination, at the edges of its padding, and for
the matrices it leaves to the FP64 form.

Bounds: the matrices are signed permutations plus 0.5 / sqrt(n) Gaussian noise
(condition below about 20); every entry of an inverse, and log|det|, may carry
32 n eps of the largest entry.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


def matrices(seed, W, n, cplx, pf=False):
    g = np.random.Generator(np.random.PCG64(seed))
    rnd = lambda *sh: g.standard_normal(sh) + (1j * g.standard_normal(sh) if cplx else 0)  # noqa: E731
    A = 0.35 * rnd(W, n, n) / np.sqrt(2 * n)
    for w in range(W):
        p = g.permutation(n)
        if pf:
            A[w] -= A[w].T
            for a, b in zip(p[0::2], p[1::2]):
                A[w, a, b] += 1.0
                A[w, b, a] -= 1.0
        else:
            A[w, np.arange(n), p] += np.exp(1j * g.uniform(0, 6.28, n)) if cplx else g.choice([-1.0, 1.0], n)
    return A


def close(a, b, n):
    a, b = np.asarray(a), np.asarray(b)
    assert np.abs(a - b).max() <= 32 * n * EPS * max(1.0, np.abs(b).max()), np.abs(a - b).max()


@pytest.mark.parametrize("kind,cplx", [("det", False), ("det", True), ("pf", False), ("pf", True)])
@pytest.mark.parametrize("n", [56, 64, 72, 128, 130, 194, 514, 1028])
def test_init_and_refresh(kind, cplx, n):
    L = lrugb()
    W = 3
    dt = torch.complex128 if cplx else torch.float64
    A, B = (matrices(7 * n + s, W, n, cplx, kind == "pf") for s in (0, 1))
    st = L.LowRankState(kind, W, n, dtype=dt, delay=4)
    ref = L.LowRankState(kind, W, n, dtype=dt, delay=4, refresh=L.REFRESH_FP64)
    la, sg = st.init(tdev(A, dt))
    lr, sr = ref.init(tdev(A, dt))
    close(st.inverse().cpu().numpy(), np.linalg.inv(A), n)
    close(la.cpu().numpy(), lr.cpu().numpy(), n)
    close(sg.cpu().numpy(), sr.cpu().numpy(), n)
    mask = torch.tensor([1, 0, 1], dtype=torch.uint8, device="cuda")
    drift = st.refresh(tdev(B, dt), mask).cpu().numpy()
    dref = ref.refresh(tdev(B, dt), mask).cpu().numpy()
    assert np.isnan(drift[1]) and np.isnan(dref[1])
    close(drift[[0, 2]], dref[[0, 2]], n)
    want = np.linalg.inv(np.stack([B[0], A[1], B[2]]))
    got = st.inverse().cpu().numpy()
    close(got, want, n)
    if kind == "pf":
        assert (got == -got.transpose(0, 2, 1)).all()
    close(st.logvalue()[0].cpu().numpy(), ref.logvalue()[0].cpu().numpy(), n)
    st.check_device_error()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [56, 65, 72, 127, 129, 513])
def test_slogdet_and_backward(cplx, n):
    L = lrugb()
    A = matrices(11 * n, 3, n, cplx)
    dt = torch.complex128 if cplx else torch.float64
    x = tdev(A, dt).requires_grad_()
    sign, logabs = L.slogdet(x)
    s, la = np.linalg.slogdet(A)
    close(logabs.detach().cpu().numpy(), la, n)
    close(sign.detach().cpu().numpy(), s, n)
    g = tdev(np.array([0.5, -1.0, 2.0]))
    (gA,) = torch.autograd.grad(logabs, x, g)
    close(gA.cpu().numpy(), g.cpu().numpy()[:, None, None] * np.linalg.inv(A).conj().transpose(0, 2, 1), n)


def test_slogpf_backward():
    L = lrugb()
    A = matrices(5, 3, 74, False, pf=True)
    x = tdev(A).requires_grad_()
    (gA,) = torch.autograd.grad(L.slogpf(x)[1].sum(), x)
    close(gA.cpu().numpy(), 0.5 * np.linalg.inv(A).transpose(0, 2, 1), 74)


@pytest.mark.parametrize("cplx", [False, True])
def test_matrices_left_to_the_fp64_form(cplx):
    """Badly scaled rows, extreme scales, zero, infinite and NaN entries, a singular matrix: as the FP64 form answers."""
    L = lrugb()
    n, W = 80, 8
    dt = torch.complex128 if cplx else torch.float64
    A = matrices(3, W, n, cplx)
    A[1] = A[1] * np.exp2(np.arange(n) % 11)[None, :]      # columns of A are rows of the working matrix
    A[2] = A[2] * np.exp2(np.arange(n) % 11)[:, None]
    A[3] *= 1e250
    A[4] *= 1e-250
    A[5, 3, 7] = np.inf
    A[6, 9, 2] = np.nan
    A[7, :, 5] = 0
    outs = []
    for refresh in (L.REFRESH_AUTO, L.REFRESH_FP64):
        st = L.LowRankState("det", W, n, dtype=dt, refresh=refresh)
        st.init(tdev(matrices(4, W, n, cplx), dt))
        drift = st.refresh(tdev(A, dt))
        la, sg = st.logvalue()
        outs.append([x.cpu().numpy() for x in (st.inverse(), la, sg, drift)])
    (inv, la, sg, dr), (inv0, la0, sg0, dr0) = outs
    for w in (1, 2, 3, 4):
        # row scales enter through the largest entry of each row and column of the inverse
        scale = np.maximum(np.abs(inv0[w]).max(0)[None, :], 1e-300)
        assert (np.abs(inv[w] - inv0[w]) / scale).max() <= 32 * n * EPS
        assert la[w] == la0[w] or abs(la[w] - la0[w]) <= 32 * n * EPS * max(1, abs(la0[w]))
        assert abs(sg[w] - sg0[w]) <= 32 * n * EPS
    for w in (5, 6, 7):
        assert np.array_equal(inv[w], inv0[w], equal_nan=True)
        assert np.array_equal(la[w], la0[w], equal_nan=True) and np.array_equal(sg[w], sg0[w], equal_nan=True)
    close(inv[0], np.linalg.inv(A[0]), n)
    sign, logabs = L.slogdet_batched(tdev(A, dt))
    s0, l0 = L.slogdet_batched_noalloc(tdev(A, dt))     # the FP64 form
    # here the rows of the working matrix are those of A: walker 1 is one for the split products
    assert torch.equal(logabs[2:].nan_to_num(7.0), l0[2:].nan_to_num(7.0))
    assert torch.equal(torch.view_as_real(sign[2:] + 0j).nan_to_num(7.0), torch.view_as_real(s0[2:] + 0j).nan_to_num(7.0))
    close(logabs[:2].cpu().numpy(), np.linalg.slogdet(A[:2])[1], n)
    close(sign[:2].cpu().numpy(), np.linalg.slogdet(A[:2])[0], n)

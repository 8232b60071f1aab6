"""The passes X = A^{-1} U, Y = V A^{-1} and the products with the delay slots
at the edges of their tiles: sizes around 32 and 64 rows, odd n (no 16-byte
rows), ranks around the vectors taken per pass, mixed one-hot and dense slots.

Bounds: A = 2 I + N(0, 0.16/n) has condition number below 4 and the ratios
stay near one, so every result carries at most a few n eps; 16 n eps is asked
(eps of the dtype).
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu

DT = {"f64": (torch.float64, False, 2.3e-16), "c128": (torch.complex128, True, 2.3e-16),
      "f32": (torch.float32, False, 1.2e-7), "c64": (torch.complex64, True, 1.2e-7)}


def case(dt, n, k, W=3):
    tdt, cplx, eps = DT[dt]
    g = np.random.Generator(np.random.PCG64(1000 * n + 10 * k + len(dt)))
    rnd = lambda *sh: g.standard_normal(sh) + (1j * g.standard_normal(sh) if cplx else 0)  # noqa: E731
    up = lambda x: tdev(x, tdt).cpu().numpy().astype(np.complex128 if cplx else np.float64)  # noqa: E731
    A = up(2 * np.eye(n) + 0.4 * rnd(W, n, n) / np.sqrt(2 * n))
    U, V = ([up(0.3 * rnd(W, k, n) / np.sqrt(n)) for _ in range(3)] for _ in range(2))
    return tdt, 16 * max(n, 8) * eps, A, U, V


def close(a, b, tol):
    assert np.abs(a - b).max() <= tol * max(1.0, np.abs(b).max()), np.abs(a - b).max()


@pytest.mark.parametrize("dt", list(DT))
@pytest.mark.parametrize("n,k", [(2, 1), (31, 2), (32, 3), (33, 1), (64, 5), (65, 4), (127, 8), (130, 2), (256, 1), (321, 9)])
def test_rank_k_chain_and_adjoint(dt, n, k):
    L = lrugb()
    tdt, tol, A, U, V = case(dt, n, k)
    W, delay = A.shape[0], 4 if k <= 8 else 3
    g = np.linspace(0.5, 1.5, W)
    for persistent in (False, True):
        st = L.LowRankState("det", W, n, k=k, dtype=tdt, delay=delay)
        st.init(tdev(A, tdt))
        cur = A.copy()
        for t in range(3):     # the second and third proposal go through filled slots
            ops = L.Operand(dense=tdev(U[t], tdt)), L.Operand(dense=tdev(V[t], tdt))
            if persistent:
                r, s, _ = st.step_persistent(*ops, accept=False)
            else:
                r, s = st.propose_det(*ops)
            assert (s.cpu().numpy() == 0).all()
            X, Y = np.linalg.solve(cur, U[t].transpose(0, 2, 1)), V[t] @ np.linalg.inv(cur)
            R = np.eye(k) + V[t] @ X
            close(r.cpu().numpy(), np.linalg.det(R), tol)
            gU, gV, gA = (x.cpu().numpy() for x in st.backward_det(tdev(g, tdt)))
            T, Z = np.linalg.solve(R, Y), X @ np.linalg.inv(R)
            close(gU, g[:, None, None] * T.conj(), tol)
            close(gV, g[:, None, None] * Z.transpose(0, 2, 1).conj(), tol)
            close(gA, -g[:, None, None] * (X @ T).transpose(0, 2, 1).conj(), tol)
            if persistent:
                st.step_persistent(*ops)
            else:
                st.accept()
            cur = cur + U[t].transpose(0, 2, 1) @ V[t]
        close(st.inverse().cpu().numpy(), np.linalg.inv(cur), tol)
        st.check_device_error()


@pytest.mark.parametrize("dt", list(DT))
@pytest.mark.parametrize("delay", [0, 4])
def test_mixed_onehot_and_dense_slots(dt, delay):
    """Slots 0 and 3 of U and slot 1 of V one-hot, the others dense."""
    L = lrugb()
    n, k = 66, 4
    tdt, tol, A, U, V = case(dt, n, k)
    W = A.shape[0]
    iu, iv = np.zeros((W, k), np.int32), np.zeros((W, k), np.int32)
    iu[:, 0], iu[:, 3], iv[:, 1] = [3, 65, 0], [64, 2, 33], [31, 32, 65]
    Um, Vm = U[0].copy(), V[0].copy()
    for w in range(W):
        Um[w, 0], Um[w, 3], Vm[w, 1] = np.eye(n)[iu[w, 0]], np.eye(n)[iu[w, 3]], np.eye(n)[iv[w, 1]]
    st = L.LowRankState("det", W, n, k=k, dtype=tdt, delay=delay)
    st.init(tdev(A, tdt))
    r, _ = st.propose_det(L.Operand(dense=tdev(Um, tdt), idx=torch.tensor(iu, device="cuda"), onehot_mask=0b1001),
                          L.Operand(dense=tdev(Vm, tdt), idx=torch.tensor(iv, device="cuda"), onehot_mask=0b0010))
    R = np.eye(k) + Vm @ np.linalg.solve(A, Um.transpose(0, 2, 1))
    close(r.cpu().numpy(), np.linalg.det(R), tol)
    st.accept()
    close(st.inverse().cpu().numpy(), np.linalg.inv(A + Um.transpose(0, 2, 1) @ Vm), tol)


@pytest.mark.parametrize("dt", ["f32", "c64"])
def test_single_precision_ratio_bits_do_not_depend_on_the_path(dt):
    """k = 3 dense columns, delayed: separate calls and the persistent step sum in the same order."""
    L = lrugb()
    n, k = 97, 3
    tdt, _, A, U, V = case(dt, n, k)
    sts = [L.LowRankState("det", A.shape[0], n, k=k, dtype=tdt, delay=4) for _ in range(2)]
    for st in sts:
        st.init(tdev(A, tdt))
    for t in range(3):
        ops = L.Operand(dense=tdev(U[t], tdt)), L.Operand(dense=tdev(V[t], tdt))
        a, _ = sts[0].propose_det(*ops)
        sts[0].accept()
        b, _, _ = sts[1].step_persistent(*ops)
        assert torch.equal(a, b)


@pytest.mark.parametrize("dt", list(DT))
@pytest.mark.parametrize("n", [1, 9, 17, 33, 64, 250, 257, 513])
@pytest.mark.parametrize("onehot", [False, True])
def test_plain_rank_one_accept(dt, n, onehot):
    """Pairs of columns per warp, a last column without a partner, one-hot V."""
    L = lrugb()
    tdt, tol, A, U, V = case(dt, n, 1)
    W = A.shape[0]
    st = L.LowRankState("det", W, n, k=1, dtype=tdt)
    st.init(tdev(A, tdt))
    cur = A.copy()
    for t in range(2):
        v, op = V[t].copy(), L.Operand(dense=tdev(V[t], tdt))
        if onehot:
            at = (np.arange(W) * 7 + t) % n
            v = np.eye(n)[at][:, None, :]
            op = L.Operand(idx=torch.tensor(at[:, None].astype(np.int32), device="cuda"), onehot_mask=1)
        st.propose_det(L.Operand(dense=tdev(U[t], tdt)), op)
        st.accept()
        cur = cur + U[t].transpose(0, 2, 1) @ v
    close(st.inverse().cpu().numpy(), np.linalg.inv(cur), tol)

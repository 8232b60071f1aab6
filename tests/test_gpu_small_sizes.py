"""Both sides of the lines by which small sizes choose their form: dense columns summed in
the propose, four-row sums of the pending slots in the inverse, work items of the
adjoint for many walkers, rank-1 accepts in pairs of columns, and the persistent step
with few and with many items.

A = 2 I + N(0, 0.16/n) has condition number below 4: 16 n eps of the largest entry.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu
DT = {"f64": (torch.float64, False, 2.3e-16), "c128": (torch.complex128, True, 2.3e-16),
      "f32": (torch.float32, False, 1.2e-7), "c64": (torch.complex64, True, 1.2e-7)}


def close(a, b, tol):
    assert np.abs(a - b).max() <= tol * max(1.0, np.abs(b).max()), np.abs(a - b).max()


@pytest.mark.parametrize("dt", list(DT))
@pytest.mark.parametrize("n,k,W", [(8, 2, 3), (9, 2, 3), (32, 3, 3), (33, 1, 3), (34, 1, 400), (48, 2, 3), (49, 4, 3), (64, 1, 170),
                                   (65, 2, 3), (128, 1, 3), (129, 1, 3), (200, 1, 400), (255, 1, 3), (257, 4, 3)])
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("delay", [0, 4])
def test_update_pending_inverse_and_adjoint(dt, n, k, W, persistent, delay):
    L = lrugb()
    tdt, cplx, eps = DT[dt]
    tol, some = 16 * max(n, 8) * eps, 3
    g = np.random.Generator(np.random.PCG64(1000 * n + k + len(dt)))
    rnd = lambda *sh: g.standard_normal(sh) + (1j * g.standard_normal(sh) if cplx else 0)  # noqa: E731
    A = 2 * np.eye(n) + 0.4 * rnd(some, n, n) / np.sqrt(2 * n)
    many = lambda x: tdev(x, tdt).repeat((W + some - 1) // some, 1, 1)[:W].contiguous()  # noqa: E731
    st = L.LowRankState("det", W, n, k=k, dtype=tdt, delay=delay)
    st.init(many(A))
    cur = A.copy()
    for _ in range(2):
        U, V = (0.3 * rnd(some, k, n) / np.sqrt(n) for _ in range(2))
        ops = L.Operand(dense=many(U)), L.Operand(dense=many(V))
        if persistent:
            r, _, _ = st.step_persistent(*ops)
        else:
            r, _ = st.propose_det(*ops)
            st.accept()
        R = np.eye(k) + V @ np.linalg.solve(cur, U.transpose(0, 2, 1))
        close(r.cpu().numpy()[:some], np.linalg.det(R), tol)
        cur = cur + U.transpose(0, 2, 1) @ V
    inv = st.inverse().cpu().numpy()
    close(inv[:some], np.linalg.inv(cur), tol)
    close(inv[W - 1], inv[(W - 1) % some], tol)
    U, V = (0.3 * rnd(some, k, n) / np.sqrt(n) for _ in range(2))
    st.propose_det(L.Operand(dense=many(U)), L.Operand(dense=many(V)))
    _, _, gA = st.backward_det(torch.ones(W, dtype=tdt, device="cuda"), want_U=False, want_V=False)
    X, Y = np.linalg.solve(cur, U.transpose(0, 2, 1)), V @ np.linalg.inv(cur)
    want = -(X @ np.linalg.solve(np.eye(k) + V @ X, Y)).transpose(0, 2, 1).conj()
    gA = gA.cpu().numpy()
    close(gA[:some], want, tol)
    close(gA[W - 1], want[(W - 1) % some], tol)
    st.check_device_error()

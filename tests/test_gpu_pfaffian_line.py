"""The Pfaffian on both sides of the sizes and counts where the double types change
between the unblocked and the blocked elimination, and sizes that differ within one call.

Bound: |log pf| may carry 16 n eps (condition below about 20), the sign none.
"""
import numpy as np
import pytest

from gpu_common import lrugb, tdev, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


def matrices(g, W, n, cplx):
    A = g.standard_normal((W, n, n)) + (1j * g.standard_normal((W, n, n)) if cplx else 0)
    A = 0.25 * (A - A.transpose(0, 2, 1)) / np.sqrt(n)
    for w in range(W):
        p = g.permutation(n)
        A[w, p[0::2], p[1::2]] += 1.0
        A[w, p[1::2], p[0::2]] -= 1.0
    return A


def check(A, logabs, sign):
    n = A.shape[-1]
    s, la = np.linalg.slogdet(A)
    assert np.abs(logabs - la / 2).max() <= 16 * n * EPS * max(1, np.abs(la).max())
    assert np.abs(sign * sign - s).max() <= 32 * n * EPS    # pf^2 = det


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [110, 112, 114, 126, 138, 140, 190, 192, 194])
@pytest.mark.parametrize("W", [3, 160])
def test_slogpf(cplx, n, W):
    L = lrugb()
    A = matrices(np.random.Generator(np.random.PCG64(n + W)), 3, n, cplx)
    x = tdev(A, torch.complex128 if cplx else torch.float64).repeat((W + 2) // 3, 1, 1)[:W].contiguous()
    sign, logabs = (t.cpu().numpy() for t in L.slogpf_batched(x))
    check(A, logabs[:3], sign[:3])
    for w in range(W):
        assert logabs[w] == logabs[w % 3] and sign[w] == sign[w % 3]


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n_max", [34, 150, 194])
def test_handle_of_different_sizes(cplx, n_max):
    L = lrugb()
    dt = torch.complex128 if cplx else torch.float64
    g = np.random.Generator(np.random.PCG64(n_max))
    sizes = [n_max, 2, 14, 16, 18, 32]
    As = [matrices(g, 1, n, cplx) for n in sizes]
    st = L.LowRankState("pf", len(sizes), sizes, dtype=dt)
    logabs, sign = st.init(torch.cat([tdev(A, dt).flatten() for A in As]))
    for w, A in enumerate(As):
        check(A, logabs[w:w + 1].cpu().numpy(), sign[w:w + 1].cpu().numpy())

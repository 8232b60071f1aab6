"""The blocked Pfaffian elimination at the edges of its blocks (16 rows a block,
64 x 64 tiles), with pivots everywhere, zero and singular cases, against the
oracle's slogpf (Householder tridiagonalisation) and log|det| / 2.

Bound: |log pf| may carry 16 n eps (condition below about 20), the sign none.
"""
import numpy as np
import pytest

from gpu_common import O, lrugb, tdev, torch

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [2, 4, 14, 16, 18, 30, 34, 64, 66, 80, 82, 146])
def test_slogpf(cplx, n):
    L = lrugb()
    g = np.random.Generator(np.random.PCG64(n + cplx))
    W = 4
    A = g.standard_normal((W, n, n)) + (1j * g.standard_normal((W, n, n)) if cplx else 0)
    A = 0.25 * (A - A.transpose(0, 2, 1)) / np.sqrt(n)
    for w in range(W):
        p = g.permutation(n)
        A[w, p[0::2], p[1::2]] += 1.0
        A[w, p[1::2], p[0::2]] -= 1.0
    A[3, n // 2, :] = 0      # singular: pf = 0
    A[3, :, n // 2] = 0
    sign, logabs = (x.cpu().numpy() for x in L.slogpf_batched(tdev(A, torch.complex128 if cplx else torch.float64)))
    for w in range(3):
        s, la = O.slogpf(A[w])
        assert abs(logabs[w] - la) <= 16 * n * EPS * max(1, abs(la))
        assert abs(logabs[w] - 0.5 * np.linalg.slogdet(A[w])[1]) <= 16 * n * EPS * max(1, abs(la))
        assert abs(sign[w] - s) <= 16 * n * EPS
    assert logabs[3] == -np.inf and sign[3] == 0

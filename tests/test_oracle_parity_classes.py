"""The symmetry behind the block M2L's parity classes, on the FP64 oracle's operators.

Mirroring an axis multiplies every real-packed coefficient (degree n, order m, real or imaginary
part) by a sign and turns the M2L operator of offset o into that of the mirrored offset.  So the
sums and differences of the eight children over each axis couple, between two parents at offset D,
only with those of the same parity along every axis where D is 0.
"""
import itertools

import numpy as np
import pytest

import oracle as O


def signs(p):
    """signs[axis, k] of the real-packed coefficients under a mirror of x, y, z."""
    s = np.ones((3, p * p))
    for n in range(p):
        for r in range(2 * n + 1):
            m, im = (r + 1) // 2, r > 0 and r % 2 == 0
            k = n * n + r
            s[1, k] = -1 if im else 1
            s[0, k] = (-1) ** m * s[1, k]
            s[2, k] = (-1) ** (n + m)
    return s


def operator(p, o):
    """The M2L of a source centre at offset o from the target centre, on real-packed coefficients."""
    T = np.zeros((p * p, p * p))
    for k in range(p * p):
        n = int(np.sqrt(k + 0.5))
        r = k - n * n
        M = np.zeros(O.ntri(p), dtype=complex)
        M[O.tri(n, (r + 1) // 2)] = 1j if (r > 0 and r % 2 == 0) else 1
        L = O.m2l(p, np.asarray(o, float), np.zeros(3), M)
        for a in range(p):
            T[a * a, k] = L[O.tri(a, 0)].real
            for m in range(1, a + 1):
                T[a * a + 2 * m - 1, k] = L[O.tri(a, m)].real
                T[a * a + 2 * m, k] = L[O.tri(a, m)].imag
    return T


def hadamard(s):
    """H[class, child, k] = (-1)^(class . child) signs^child."""
    H = np.ones((8, 8, s.shape[1]))
    for c, q in itertools.product(range(8), repeat=2):
        for d in range(3):
            if q >> d & 1:
                H[c, q] *= s[d] * (-1 if c >> d & 1 else 1)
    return H


@pytest.mark.parametrize("p", [4, 6])
def test_mirrored_operators(p):
    s = signs(p)
    for o in ((2, 1, -3), (0, 2, -1), (3, 2, 2)):
        T = operator(p, o)
        for d in range(3):
            m = list(o)
            m[d] = -m[d]
            assert np.allclose(operator(p, m), s[d][:, None] * T * s[d][None], atol=1e-13 * np.abs(T).max())


@pytest.mark.parametrize("D", [(1, 0, 0), (0, -1, 1), (0, 0, 1), (1, 1, -1)])
def test_classes_of_other_parity_do_not_couple(D):
    p = 4
    pp = p * p
    B = np.zeros((8, pp, 8, pp))
    for tau, sig in itertools.product(range(8), repeat=2):
        o = [2 * D[d] + (sig >> d & 1) - (tau >> d & 1) for d in range(3)]
        if max(map(abs, o)) >= 2:
            B[tau, :, sig] = operator(p, o)
    H = hadamard(signs(p))
    assert np.allclose(np.einsum("cqk,dqk->cdk", H, H), 8 * np.eye(8)[:, :, None])
    Bc = np.einsum("ctn,tnsk,dsk->cndk", H, B, H) / 8
    scale = np.abs(B).max()
    for c, d in itertools.product(range(8), repeat=2):
        if any(D[a] == 0 and (c ^ d) >> a & 1 for a in range(3)):
            assert np.abs(Bc[c, :, d]).max() <= 1e-13 * scale
    # the children's result from the classes'
    M = np.random.default_rng(1).standard_normal((8, pp))
    V = np.einsum("cndk,dk->cn", Bc, np.einsum("dsk,sk->dk", H, M))
    L = np.einsum("ctn,cn->tn", H, V) / 8
    assert np.allclose(L, np.einsum("tnsk,sk->tn", B, M), atol=1e-12 * scale)

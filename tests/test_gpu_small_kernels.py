"""The one-CTA dense kernels of the eigensolver, called as its host code calls them (svqb_small,
rayleigh_ritz_small of the library): nearly dependent blocks, and matrices that hold a NaN.
"""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MAX_BLOCK, MAX_SMALL = 24, 72
SVQB = "_ZN3iwf10svqb_smallERKNS_5BatchEPK7double2idPS3_PiS7_P11CUstream_st"
RR = "_ZN3iwf19rayleigh_ritz_smallERKNS_5BatchEPK7double2iiPKiiPdPS3_S9_PiSA_P11CUstream_st"


class Batch(C.Structure):
    _fields_ = [("nprob", C.c_int), ("pstride", C.c_longlong), ("active", C.c_void_p),
                ("engine", C.c_int), ("exps", C.c_void_p), ("err", C.c_void_p)]


def _lib():
    from paper_2404_04507_gb300 import build
    assert torch.cuda.is_available()
    return C.CDLL(build.build())


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def orthonormaliser(G, drop=1e-14):
    """T (b x b) and the mask of svqb_small for the Gram matrix G."""
    b = len(G)
    g = torch.zeros(MAX_SMALL * MAX_SMALL, dtype=torch.complex128, device="cuda")
    g[:b * b] = torch.from_numpy(np.ascontiguousarray(G).reshape(-1)).cuda()
    t = torch.full((MAX_BLOCK * MAX_BLOCK,), float("nan"), dtype=torch.complex128, device="cuda")
    mask = torch.full((MAX_BLOCK,), -1, dtype=torch.int32, device="cuda")
    batch = Batch(1, 0, None, 0, None, None)
    torch.cuda.synchronize()
    st = getattr(_lib(), SVQB)(C.byref(batch), _ptr(g), b, C.c_double(drop), _ptr(t), _ptr(mask), None, None)
    assert st == 0
    torch.cuda.synchronize()
    return t[:b * b].cpu().numpy().reshape(b, b), mask[:b].cpu().numpy()


def rayleigh_ritz(A, b, x_rows, mask=None):
    m = len(A)
    a = torch.zeros(MAX_SMALL * MAX_SMALL, dtype=torch.complex128, device="cuda")
    a[:m * m] = torch.from_numpy(np.ascontiguousarray(A).reshape(-1)).cuda()
    on = torch.zeros(MAX_SMALL, dtype=torch.int32, device="cuda")
    on[:m] = 1 if mask is None else torch.from_numpy(mask.astype(np.int32)).cuda()
    th = torch.zeros(MAX_BLOCK, dtype=torch.float64, device="cuda")
    cx, cp = (torch.zeros(MAX_SMALL * MAX_BLOCK, dtype=torch.complex128, device="cuda") for _ in range(2))
    mp, st = (torch.full((MAX_BLOCK,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    batch = Batch(1, 0, None, 0, None, None)
    torch.cuda.synchronize()
    r = getattr(_lib(), RR)(C.byref(batch), _ptr(a), m, b, _ptr(on), x_rows, _ptr(th), _ptr(cx), _ptr(cp),
                            _ptr(mp), _ptr(st), None)
    assert r == 0
    torch.cuda.synchronize()
    return (th[:b].cpu().numpy(), cx[:m * b].cpu().numpy().reshape(m, b), cp[:m * b].cpu().numpy().reshape(m, b),
            mp[:b].cpu().numpy(), int(st[0]))


def _randn(rng, *s):
    return rng.standard_normal(s) + 1j * rng.standard_normal(s)


def _dependent(kind, n, b, rng):
    if kind == "powers":                                # columns x^k: singular values fall to 1e-18
        x = np.linspace(0.0, 1.0, n)
        return np.stack([x ** k for k in range(b)], 1).astype(complex)
    if kind == "krylov":
        d = np.logspace(0, 3, n)
        cols = [_randn(rng, n)]
        for _ in range(b - 1):
            cols.append(d * cols[-1] / np.linalg.norm(d * cols[-1]))
        return np.stack(cols, 1)
    if kind == "rank5":
        return _randn(rng, n, 5) @ _randn(rng, 5, b)
    if kind == "rank5_noise":
        return _randn(rng, n, 5) @ _randn(rng, 5, b) + 1e-7 * _randn(rng, n, b)
    if kind == "pairs":
        Y = _randn(rng, n, b)
        Y[:, 1::2] = Y[:, ::2][:, :Y[:, 1::2].shape[1]] + 3e-8 * Y[:, 1::2]
        return Y
    u, v = np.linalg.qr(_randn(rng, n, b))[0], np.linalg.qr(_randn(rng, b, b))[0]
    return u @ np.diag(np.logspace(0, -10, b)) @ v      # graded


@pytest.mark.parametrize("b", [24, 11, 2])
@pytest.mark.parametrize("kind", ["powers", "krylov", "rank5", "rank5_noise", "pairs", "graded"])
def test_nearly_dependent_blocks(kind, b):
    # two passes, as in the solver, on a block without components in an orthonormal X. The second
    # leaves orthonormal columns. What the first amplifies: a direction is kept down to an
    # eigenvalue of 1e-14, so that the rounding 2^-53 of unit columns may appear times 1e7 as a
    # component in X: 1.1e-9 at most, and directions below stay out (a margin of 100 either side for
    # a test that knows pivots, not eigenvalues).
    rng = np.random.default_rng(b)
    n, drop = 2000, 1e-14
    X = np.linalg.qr(_randn(rng, n, 48))[0]
    Y = _dependent(kind, n, b, rng)
    Y /= np.linalg.norm(Y, axis=0)
    for _ in range(2):
        Y = Y - X @ (X.conj().T @ Y)
    D = 1.0 / np.linalg.norm(Y, axis=0)
    lam = np.linalg.eigvalsh((Y * D).conj().T @ (Y * D))
    for _ in range(2):
        T, mask = orthonormaliser(Y.conj().T @ Y, drop)
        assert np.all(T[:, mask == 0] == 0)
        Y = Y @ T
    assert np.sum(lam > 100 * drop * lam[-1]) <= mask.sum() <= np.sum(lam > 0.01 * drop * lam[-1])
    Q = Y[:, mask == 1]
    assert np.max(np.abs(Q.conj().T @ Q - np.eye(Q.shape[1]))) <= 1e-14
    assert np.max(np.abs(X.conj().T @ Q)) <= 2.0 ** -53 * 1e7


@pytest.mark.parametrize("bits", [0xFFF8000000000000, 0x7FF8000000000000])
@pytest.mark.parametrize("row,col", [(5, 0), (7, 6), (40, 21), (71, 70)])
def test_a_nan_off_the_diagonal_reaches_every_eigenvalue(row, col, bits):
    # a quiet NaN with the sign that the GPU's own arithmetic gives it, and with the other one
    rng = np.random.default_rng(2)
    A = _randn(rng, 72, 72)
    A = A + A.conj().T
    nan = np.array([bits], dtype=np.uint64).view(np.float64)[0]
    A[row, col], A[col, row] = complex(nan, nan), complex(nan, -nan)
    theta, Cx, _, _, _ = rayleigh_ritz(A, 24, 24)
    assert np.all(np.isnan(theta)) and np.all(np.isnan(Cx))


def _orthonormal(Y):
    """An orthonormal basis of Y's columns in extended precision."""
    Q = []
    for v in Y.T:
        for _ in range(3):
            for q in Q:
                v = v - q * np.vdot(q, v)
        Q.append(v / np.sqrt(np.vdot(v, v).real))
    return np.stack(Q, 1)


@pytest.mark.parametrize("coupling", [1.0, 1e-3, 1e-8])
@pytest.mark.parametrize("m,b", [(72, 24), (36, 12), (9, 3)])
def test_p_coefficients_span_what_they_should(m, b, coupling):
    # S Cp spans the W and P parts of Cx's columns, orthogonal to S Cx. A column of it comes from a sum
    # of b + 2 products of unit columns, (b + 2) 2^-53 at worst before the orthonormalisation, whose
    # condition (below 20 here) multiplies rms errors a fifth of that: 64 2^-53 bounds the part
    # outside the exact span
    rng = np.random.default_rng(m)
    R = _randn(rng, m, m) * coupling
    A = np.diag(np.sort(rng.uniform(1.0, 100.0, m))) + R + R.conj().T
    theta, Cx, Cp, mask_p, status = rayleigh_ritz(A, b, b)
    assert status == 0 and np.all(mask_p == 1)
    assert np.max(np.abs(theta - np.linalg.eigvalsh(A)[:b])) <= 1e-14 * np.linalg.norm(A, 2)
    for U, V, eye in ((Cx, Cx, np.eye(b)), (Cp, Cp, np.eye(b)), (Cx, Cp, 0.0)):
        assert np.max(np.abs(U.conj().T @ V - eye)) <= 1e-14
    X = _orthonormal(Cx.astype(np.clongdouble))
    Y = Cx.astype(np.clongdouble)
    Y[:b] = 0
    Y = Y - X @ (X.conj().T @ Y)
    Q = _orthonormal(Y / np.sqrt(np.sum(np.abs(Y) ** 2, axis=0)))
    out = Cp - Q @ (Q.conj().T @ Cp)
    assert np.max(np.sqrt(np.sum(np.abs(out) ** 2, axis=0))) <= 64 * 2.0 ** -53

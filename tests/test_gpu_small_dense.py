"""The eigensolver's one-CTA dense problems (Rayleigh-Ritz, orthonormalisation) through
iwf_eigensolve, against the dense oracle, at the sizes where their kernels change: block 1 (bases of
1, 2 and 3 vectors), odd blocks, bases around 16, 32 and 48 columns, the largest (24 -> 72);
windows with barely more points than the basis; eigenvalues of exact multiplicity (clusters in
the inverse iteration); dependent and zero columns in the start block.

Tolerance: the solver's residual target 1e-10 bounds an eigenvalue's error by itself; eigenvectors
are orthonormal to 1e-12 (FP64 rounding of sums of at most 768 terms is below 1e-13).
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_2404_04507_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def iwf():
    import paper_2404_04507_gb300 as iwf
    assert torch.cuda.is_available()
    return iwf


def _solve(iwf, pb, nev, **kw):
    plan = iwf.Plan(pb.P, pb.K, pb.L, method=pb.method)
    plan.set_potential(pb.modes, pb.coef)
    ev, X, res, info = plan.eigensolve(nev, tol=1e-10, maxit=3000, **kw)
    assert info["converged"] == 1 and np.all(res <= 1e-10)
    win = O.build_window(pb.P, pb.K, pb.L, method=pb.method)
    ref = O.eigen.dense_eigs(win, O.grid_coefficients(pb.modes, pb.coef, win.lens), nev)[0]
    assert np.all(np.abs(ev - ref) <= 1e-10 * np.maximum(1.0, np.abs(ref))), np.max(np.abs(ev - ref))
    X = X.cpu().numpy()
    assert np.max(np.abs(X.conj() @ X.T - np.eye(nev))) <= 1e-12
    return info


@pytest.mark.parametrize("block", [1, 2, 5, 6, 8, 11, 16, 17, 21, 24])
def test_block_sizes(iwf, block):
    _solve(iwf, W.config_1d(), max(1, block - 3), block=block)


@pytest.mark.parametrize("K,L,block", [(2, 2, 5), (3, 4, 16), (6, 6, 24)])
def test_windows_barely_larger_than_the_basis(iwf, K, L, block):
    _solve(iwf, W.config_1d(K=K, L=L), block // 2, block=block)


@pytest.mark.parametrize("block", [6, 12, 24])
def test_exact_multiplicities(iwf, block):
    # separable: every eigenvalue of mixed indices comes twice (PM box, two equal 1D problems),
    # and without a potential the spectrum is the kinetic diagonal with its +-k pairs
    m, c = W.cosine_modes(4, 1.3)
    P = np.concatenate([np.eye(2), math.sqrt(2.0) * np.eye(2)], axis=1)
    _solve(iwf, W.Problem("kron", P, (2, 2), (3, 3), m, c, method="pm"), block // 2, block=block)
    free = W.Problem("free", P, (3, 3), (2, 2), np.zeros((1, 4), int), np.array([0.25 + 0j]), method="pm")
    _solve(iwf, free, block // 2, block=block)


@pytest.mark.parametrize("kind", ["repeated", "zero", "nearly"])
def test_dependent_start_columns(iwf, kind):
    pb = W.config_1d()
    X = W.random_block(pb.dof, 10, seed=3).T.copy()
    if kind == "repeated":
        X[4], X[7] = X[1], 2.5j * X[0]
    elif kind == "zero":
        X[2] = 0.0
    else:
        X[5] = X[3] + 1e-9 * X[5]
    _solve(iwf, pb, 6, block=10, X0=torch.from_numpy(X).cuda())

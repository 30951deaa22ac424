"""The direct convolution inside iwf_apply, against the CPU oracle.

iwf_apply runs potentials with few folded modes as a direct convolution. These cases sit where
its kernel's index arithmetic can go wrong: one to five k_I axes (32-bit offsets for up to
three), slices smaller than a CTA's threads (several slices share one) and larger than 256 with a
remainder, 1 to 6 vectors (groups of 1, 2 and 4 with a repeated tail), shifts by more than one
slice, modes on several axes at once, a constant term, the limits of the mode count on both
sides, and batches whose problems have different modes. The transforms, which the default path
no longer reaches for these potentials, are held to the same oracle through set_path.

Tolerances are those of the other apply tests: 1e-12 (complex double) and 2e-5 (complex float)
of max |H psi|; a direct sum of at most 48 products rounds less than the transforms.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_2404_04507_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {torch.complex128: 1e-12, torch.complex64: 2e-5}


@pytest.fixture(scope="module")
def iwf():
    import paper_2404_04507_gb300 as iwf
    assert torch.cuda.is_available()
    return iwf


def _axis_modes(n, count, seed, real, const=0.0, lens=None):
    """count modes in +-m pairs, the k-th pair on axis k mod n with shift 1 + k // n."""
    rng = np.random.default_rng(seed)
    m, c = ([[0] * n], [complex(const)]) if const else ([], [])
    for k in range(count // 2):
        v = [0] * n
        v[k % n] = 1 + k // n
        z = complex(rng.standard_normal(), 0.0 if real else rng.standard_normal())
        m += [v, [-t for t in v]]
        c += [z, z.conjugate()]
    return np.array(m), np.array(c)


def _problem(d, n, K, L, modes, **kw):
    return W.Problem("p", W.random_P(d, n, seed=11), K, L, *modes, **kw)


GEOS = {
    "d1_small_slices": _problem(1, 3, (2,), (5, 3), _axis_modes(3, 6, 1, False, const=0.7)),
    "d1_long_slice": _problem(1, 2, (150,), (3,), _axis_modes(2, 8, 2, True)),
    "d2_ragged": _problem(2, 4, (5, 3), (4, 6), _axis_modes(4, 16, 3, False)),
    "d2_remainder": _problem(2, 3, (9, 11), (7,), _axis_modes(3, 6, 4, True, const=-2.0)),
    "d3": _problem(3, 5, (3, 2, 4), (2, 3), _axis_modes(5, 10, 5, False), method="pm"),
    "d4": _problem(4, 5, (2, 3, 2, 2), (3,), _axis_modes(5, 10, 6, False)),
    "d5_round": _problem(5, 6, (2, 1, 2, 1, 2), (2,), _axis_modes(6, 6, 7, True), shift_round=True),
    "several_axes": _problem(2, 4, (4, 5), (3, 4), W.random_modes(4, 8, 2, seed=8)),
    "no_modes": _problem(1, 2, (4,), (5,), (np.array([[0, 0]]), np.array([1.5 + 0j]))),
}


def _plan(iwf, pb):
    plan = iwf.Plan(pb.P, pb.K, pb.L, method=pb.method, shift_round=pb.shift_round)
    plan.set_potential(pb.modes, pb.coef)
    return plan


def _check(plan, pb, dtype, nvec, launches=None, iwf=None):
    win = O.build_window(pb.P, pb.K, pb.L, shift_round=pb.shift_round, method=pb.method)
    Vg = O.grid_coefficients(pb.modes, pb.coef, win.lens)
    X = W.random_block(win.N, nvec, seed=nvec)
    x = torch.from_numpy(np.ascontiguousarray(X.T)).to(dtype).cuda()
    before = iwf.kernel_launches() if iwf else 0
    got = plan.apply(x, out=torch.full_like(x, float("nan")))
    if launches is not None:
        assert iwf.kernel_launches() - before == launches
    want = O.apply_stencil(win, Vg, x.cpu().numpy().T.astype(np.complex128))
    err = np.max(np.abs(got.cpu().numpy().T.astype(np.complex128) - want))
    assert err <= TOL[dtype] * np.max(np.abs(want)), err


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("name", list(GEOS))
def test_direct_apply_matches_oracle(iwf, name, dtype):
    pb = GEOS[name]
    plan = _plan(iwf, pb)
    for nvec in (1, 2, 3, 6):
        _check(plan, pb, dtype, nvec, launches=1, iwf=iwf)


@pytest.mark.parametrize("dtype,real,limit", [(torch.complex128, True, 48), (torch.complex128, False, 24),
                                              (torch.complex64, False, 20)])
def test_mode_limit_of_the_direct_apply(iwf, dtype, real, limit):
    for count, launches in ((limit, 1), (limit + 2, 3)):
        pb = _problem(2, 4, (8, 8), (8, 8), _axis_modes(4, count, 9, real, const=0.3))
        _check(_plan(iwf, pb), pb, dtype, 2, launches=launches, iwf=iwf)


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("name", ["tiled16", "pencil16", "tiled_ragged", "long", "split", "ex43"])
def test_transforms_stay_reachable(iwf, name, dtype):
    pb = {"tiled16": W.config_moire(K=8, L=8, phases=[0.1, 2.0, 3.0, 5.5]),
          "pencil16": W.config_moire(K=8, L=8, phases=[0.1, 2.0, 3.0, 5.5]),
          "tiled_ragged": W.config_moire(K=5, L=3, method="pm"),
          "long": W.example_41(2.5, 21, 60),
          "split": _problem(1, 4, (2,), (12, 12, 12), W.cosine_modes(4, 1.5)),
          "ex43": W.example_43(math.pi, K=2, L=4)}[name]
    plan = _plan(iwf, pb)
    for prec in ("f64", "c64"):
        plan.set_path(prec, "pencil" if name == "pencil16" else "tiled")
    _check(plan, pb, dtype, 3, 
           launches=7 if name == "split" and dtype == torch.complex128 else 3, iwf=iwf)


def test_noalloc_and_host_take_the_same_kernel(iwf):
    import ctypes as C
    from paper_2404_04507_gb300 import capi
    pb = GEOS["d2_ragged"]
    plan = _plan(iwf, pb)
    x = torch.from_numpy(np.ascontiguousarray(W.random_block(plan.N, 5, seed=4).T)).cuda()
    want, got = plan.apply(x), torch.empty_like(x)
    capi.check(capi.iwf_apply_noalloc(plan.handle, capi.IWF_PREC_F64, C.c_void_p(x.data_ptr()),
                                      C.c_void_p(got.data_ptr()), 5,
                                      C.c_void_p(torch.cuda.current_stream().cuda_stream)), "noalloc")
    assert torch.equal(got, want)
    assert torch.equal(plan.apply_host(x.cpu()), want.cpu())


def test_autotune_keeps_the_direct_apply(iwf):
    pb = W.config_moire(eps=0.5, K=8, L=8)
    plan = _plan(iwf, pb)
    plan.autotune("f64", nvec=8)
    _check(plan, pb, torch.complex128, 3, launches=1, iwf=iwf)


@pytest.mark.parametrize("precision", ["f64", "c64"])
@pytest.mark.parametrize("long_list", [False, True])
def test_batch_of_different_modes_matches_dense(iwf, precision, long_list):
    # four problems with their own mode lists (one without any but the constant); a fifth with a
    # long list sends the whole batch to the transforms
    P, K, L = np.array([[1.0, math.sqrt(5.0)]]), (5,), (12,)
    pots = [W.cosine_modes(2, 1.0), W.cosine_modes(2, 0.6, phases=[0.4, 2.2], const=0.5),
            _axis_modes(2, 8, 21, False), (np.array([[0, 0]]), np.array([2.0 + 0j]))]
    if long_list:
        rng = np.random.default_rng(5)
        m = [[0, 1 + k] for k in range(11)] + [[1 + k, 0] for k in range(4)]
        c = rng.standard_normal(len(m)) * 0.3
        pots.append((np.array(m + [[-a, -b] for a, b in m] + [[5, 0], [0, 12]]),
                     np.concatenate([c, c, [0.2, 0.1]]).astype(complex)))
    plan = iwf.Plan(P, K, L)
    ev, _, res, _, info = plan.batch_eigensolve(pots, 3, block=6, precision=precision)
    assert info["converged"] == 1
    win = O.build_window(P, K, L)
    for q, (m, c) in enumerate(pots):
        ref = O.eigen.dense_eigs(win, O.grid_coefficients(m, c, win.lens), 3)[0]
        assert np.all(np.abs(ev[q] - ref) <= 1e-10 * np.maximum(1.0, np.abs(ref))), q

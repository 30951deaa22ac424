"""The transform passes of iwf_apply (tiled, pencil, shared-memory FFT, per-axis k_II) against the
CPU oracle, on the path that is set: potentials with few modes leave them on IWF_PATH_AUTO, so
each test here sets the path, or brings a potential of more modes than the direct convolution
takes, and counts the kernels that ran.

Geometries, schedules and tolerances are those of test_gpu_apply: 1e-12 (complex double) and 2e-5
(complex float) of max |H psi|.
"""

import numpy as np
import pytest

import oracle as O
from paper_2404_04507_gb300 import workloads as W

from test_gpu_apply import LONG, PENCIL, PROBS, SPLIT, _gpu_apply, _oracle, _plan, iwf  # noqa: F401
from test_zz_no_alloc import _noalloc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "c64": 2e-5}
DTYPE = {"f64": torch.complex128, "c64": torch.complex64}


def _block(plan, nvec, prec, seed):
    X = W.random_block(plan.N, nvec, seed=seed)
    return X.astype(np.complex64).astype(np.complex128) if prec == "c64" else X


def _check(iwf, plan, pb, prec, nvec, launches, seed=21, columns=None):  # noqa: F811
    win, Vg = _oracle(pb, pb.shift_round)
    X = _block(plan, nvec, prec, seed)
    before = iwf.kernel_launches()
    got = _gpu_apply(plan, X, DTYPE[prec])
    ran = iwf.kernel_launches() - before
    assert ran >= 3 if launches is None else ran == launches, ran
    for c in range(nvec) if columns is None else columns:
        want = O.apply_stencil(win, Vg, X[:, c])
        assert np.max(np.abs(got[:, c] - want)) <= TOL[prec] * np.max(np.abs(want)), c


@pytest.mark.parametrize("name", list(PROBS))
@pytest.mark.parametrize("prec", ["f64", "c64"])
def test_tiled(iwf, name, prec):  # noqa: F811
    pb = PROBS[name]
    plan = _plan(iwf, pb, pb.shift_round)
    plan.set_path(prec, "tiled")
    _check(iwf, plan, pb, prec, 3, 3)


@pytest.mark.parametrize("sched", [(128, 24, 24), (128, 96, 48), (256, 48, 96), (256, 160, 48)])
@pytest.mark.parametrize("prec", ["f64", "c64"])
@pytest.mark.parametrize("name", ["moire_ragged", "qse1d", "moire16"])
def test_every_schedule(iwf, sched, prec, name):  # noqa: F811
    pb = PENCIL[name] if name == "moire16" else PROBS[name]
    plan = _plan(iwf, pb)
    plan.set_path(prec, "tiled")
    plan.set_schedule(prec, *sched)
    _check(iwf, plan, pb, prec, 5, 3)


@pytest.mark.parametrize("name", list(PENCIL))
@pytest.mark.parametrize("prec", ["f64", "c64"])
@pytest.mark.parametrize("path", ["pencil", "tiled"])
def test_pencil_geometries(iwf, name, prec, path):  # noqa: F811
    pb = PENCIL[name]
    plan = _plan(iwf, pb)
    plan.set_path(prec, path)
    _check(iwf, plan, pb, prec, 3, 3)


@pytest.mark.parametrize("prec", ["f64", "c64"])
def test_full_size_paths_agree(iwf, prec):  # noqa: F811
    # 16 vectors of the 32^4 grid through both kernel sets and the direct convolution; a chunk of 32
    # or 16 MB holds two vectors
    pb = W.config_moire(eps=5.0, phases=[0.4, 1.9, 3.3, 5.0])
    plan = _plan(iwf, pb)
    plan.set_schedule(prec, 128, 96, 16 if prec == "c64" else 32)
    plan.set_path(prec, "pencil")
    _check(iwf, plan, pb, prec, 16, 24, columns=(0, 15))
    x = torch.from_numpy(np.ascontiguousarray(_block(plan, 16, prec, 5).T)).to(DTYPE[prec]).cuda()
    outs = [plan.apply(x), plan.apply_stencil(x)]
    plan.set_path(prec, "tiled")
    outs.append(plan.apply(x))
    scale = float(outs[0].abs().max())
    for y in outs[1:]:
        assert float((outs[0] - y).abs().max()) <= 2 * TOL[prec] * scale


@pytest.mark.parametrize("name", list(LONG) + list(SPLIT))
@pytest.mark.parametrize("prec", ["f64", "c64"])
def test_long_and_split_groups(iwf, name, prec):  # noqa: F811
    pb = LONG[name] if name in LONG else SPLIT[name]
    plan = _plan(iwf, pb, pb.shift_round)
    plan.set_path(prec, "tiled")
    _check(iwf, plan, pb, prec, 2, 3 if name in LONG else None)


@pytest.mark.parametrize("prec", ["f64", "c64"])
def test_longest_axis(iwf, prec):  # noqa: F811
    pb = W.config_1d(K=5, L=4096)
    plan = _plan(iwf, pb)
    plan.set_path(prec, "tiled")
    _check(iwf, plan, pb, prec, 4, 3)


# Potentials of 60 modes on several axes at once: a full potential grid, which the automatic path
# leaves to the transforms in either precision.
MANY = {
    "tiled_ragged": W.Problem("m0", W.random_P(2, 4, seed=7), (5, 4), (3, 6), *W.random_modes(4, 30, 2, seed=8)),
    "pencil16": W.Problem("m1", W.random_P(2, 4, seed=7), (8, 8), (8, 8), *W.random_modes(4, 30, 3, seed=9)),
    "pencil16_32": W.Problem("m2", W.random_P(2, 4, seed=7), (8, 8), (16, 16), *W.random_modes(4, 30, 3, seed=9)),
    "pencil32_16": W.Problem("m3", W.random_P(2, 4, seed=7), (16, 16), (8, 8), *W.random_modes(4, 30, 3, seed=9)),
    "long": W.Problem("m4", W.random_P(1, 2, seed=3), (6,), (50,), *W.random_modes(2, 30, 5, seed=4)),
    "split": W.Problem("m5", W.random_P(1, 4, seed=3), (2,), (12, 12, 12), *W.random_modes(4, 30, 2, seed=7)),
}


@pytest.mark.parametrize("name", list(MANY))
@pytest.mark.parametrize("prec", ["f64", "c64"])
def test_potentials_of_many_modes(iwf, name, prec):  # noqa: F811
    pb = MANY[name]
    plan = _plan(iwf, pb)
    _check(iwf, plan, pb, prec, 3, None if name == "split" else 3)


# Windows and blocks for which a tile of the k_I passes takes several slices, with a remainder: few
# points a slice (10, 18, 6 x 4, 4 x 2 x 2), many slices over all vectors.
TILES = {
    "1d": (W.Problem("t0", W.random_P(1, 2, seed=5), (5,), (16,), *W.cosine_modes(2, 1.0)), 96),
    "1d_odd": (W.Problem("t1", W.random_P(1, 3, seed=5), (9,), (5, 7), *W.cosine_modes(3, 1.0)), 24),
    "2d": (W.Problem("t2", W.random_P(2, 4, seed=5), (3, 2), (5, 3), *W.cosine_modes(4, 1.0)), 40),
    "2d_moire": (W.config_moire(eps=2.0, K=9, L=11), 6),
    "3d": (W.Problem("t3", W.random_P(3, 5, seed=5), (2, 1, 1), (7, 5), *W.cosine_modes(5, 1.0)), 31),
}


@pytest.mark.parametrize("name", list(TILES))
@pytest.mark.parametrize("prec", ["f64", "c64"])
def test_tiles_of_several_slices(iwf, name, prec):  # noqa: F811
    pb, nvec = TILES[name]
    plan = _plan(iwf, pb)
    plan.set_path(prec, "tiled")
    _check(iwf, plan, pb, prec, nvec, 3, columns=range(0, nvec, 5))


@pytest.mark.parametrize("path", ["pencil", "tiled"])
@pytest.mark.parametrize("prec,launches", [("f64", 9), ("c64", 6)])
def test_noalloc_in_chunks(iwf, path, prec, launches):  # noqa: F811
    # one vector of the 32^4 grid takes 16 or 8 of the static array's 32 MiB: five run in chunks of
    # two or four; the second call finds the first one's data in the array
    pb = W.config_moire(eps=5.0)
    plan = _plan(iwf, pb)
    plan.set_path(prec, path)
    for seed in (21, 22):
        x = torch.from_numpy(np.ascontiguousarray(_block(plan, 5, prec, seed).T)).to(DTYPE[prec]).cuda()
        want = plan.apply_stencil(x)
        before = iwf.kernel_launches()
        got = _noalloc(plan, x, torch.full_like(x, float("nan")))
        assert iwf.kernel_launches() - before == launches
        assert float((got - want).abs().max()) <= 2 * TOL[prec] * float(want.abs().max())


@pytest.mark.parametrize("precision", ["f64", "c64"])
def test_batch_on_the_paths(iwf, precision):  # noqa: F811
    # two problems on one 16^4 window: per-problem potential tables and skipped converged problems
    # inside the kernels of each path, certified by the oracle
    probs = [W.config_moire(eps=e, K=8, L=8, phases=ph)
             for e, ph in ((0.7, [0.2, 1.4, 2.2, 0.9]), (5.0, [3.0, 0.3, 4.1, 1.7]))]
    plan = iwf.Plan(probs[0].P, probs[0].K, probs[0].L)
    ev = {}
    for path in ("pencil", "tiled"):
        plan.set_path("f64", path)
        plan.set_path("c64", path)
        ev[path], X, _, _, info = plan.batch_eigensolve([(p.modes, p.coef) for p in probs], 4, block=8,
                                                        precision=precision, want_vectors=True)
        assert info["converged"] == 1
        for q, pb in enumerate(probs):
            win, Vg = _oracle(pb)
            assert np.max(O.eigen.residual_norms(win, Vg, X[q].cpu().numpy().T, ev[path][q])) <= 2e-10
    assert np.allclose(ev["pencil"], ev["tiled"], rtol=1e-10, atol=1e-10)


def test_host_blocks(iwf):  # noqa: F811
    pb = PENCIL["moire16_phases"]
    plan = _plan(iwf, pb)
    for path in ("pencil", "tiled"):
        for prec in ("f64", "c64"):
            plan.set_path(prec, path)
            x = torch.from_numpy(np.ascontiguousarray(_block(plan, 7, prec, 8).T)).to(DTYPE[prec])
            assert torch.equal(plan.apply_host(x), plan.apply(x.cuda()).cpu())


@pytest.mark.parametrize("prec", ["f64", "c64"])
@pytest.mark.parametrize("K,L,nvec", [(8, 8, 1), (8, 8, 16), (8, 16, 2), (16, 8, 1)])
def test_autotune_keeps_the_transforms_it_reports(iwf, prec, K, L, nvec):  # noqa: F811
    # tuned with a potential that the direct convolution applies; a later one of many modes runs on
    # the kernels of the best schedule, bit for bit those of the path that the plan reports
    pb = W.config_moire(eps=0.5, K=K, L=L)
    plan = _plan(iwf, pb)
    ms, best = plan.autotune(prec, nvec=nvec)
    sched = plan.schedule(prec)
    assert ms > 0 and (sched["path"] == "pencil") == (best[:2] == (0, 0))
    plan.set_potential(*W.random_modes(4, 30, 3, seed=9))
    x = torch.from_numpy(np.ascontiguousarray(_block(plan, nvec, prec, 3).T)).to(DTYPE[prec]).cuda()
    got = plan.apply(x)
    plan.set_path(prec, sched["path"])
    assert torch.equal(got, plan.apply(x))
    plan.set_path(prec, "auto")
    assert plan.schedule(prec)["path"] == "pencil"


def test_a_tuned_tiled_path_refuses_double_float_dfts(iwf):  # noqa: F811
    from paper_2404_04507_gb300 import capi
    pb = PENCIL["moire16"]
    plan = _plan(iwf, pb)
    plan.set_path("f64", "tiled")
    plan.autotune("f64", nvec=1)
    with pytest.raises(capi.IwfError) as e:
        plan.set_arith("df")
    assert e.value.status == -10

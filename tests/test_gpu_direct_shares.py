"""The direct convolution on windows of few slices, where CTAs share a slice (iwf_apply, and the
batched solver's apply through it).

Correctness at the edges of the shares: slices of one run of threads and a bit, of as many runs as
there are shares and of more, a ragged last run, one to five k_I axes, 1 to 6 vectors; against the
CPU oracle, with the tolerances of the other apply tests (1e-12 and 2e-5 of max |H psi|).

Speed, coarsely: with 16 slices and a CTA each the direct convolution took 2.4 times as long as the
transforms that the same plan can be told to take; it may not be slower than they are by a half.
"""
import numpy as np
import pytest

import oracle as O
from paper_2404_04507_gb300 import workloads as W

from test_gpu_direct import TOL, _axis_modes, _check, _plan, _problem, iwf  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FEW = {
    "d1": _problem(1, 2, (160,), (2,), _axis_modes(2, 6, 1, False, const=0.7)),       # 320 x 4
    "d1_many_runs": _problem(1, 2, (640,), (1,), _axis_modes(2, 8, 2, True)),         # 1280 x 2
    "d2": _problem(2, 3, (9, 16), (3,), _axis_modes(3, 6, 3, True, const=-1.0)),      # 18 x 32 x 6
    "d2_long": _problem(2, 3, (20, 21), (1,), _axis_modes(3, 6, 4, False)),           # 40 x 42 x 2
    "d3": _problem(3, 4, (5, 6, 7), (1,), _axis_modes(4, 8, 5, False)),               # 1680 x 2
    "d4": _problem(4, 5, (4, 4, 4, 4), (2,), _axis_modes(5, 20, 6, False)),           # 4096 x 4
    "d5": _problem(5, 6, (2, 3, 2, 3, 2), (1,), _axis_modes(6, 12, 7, True)),         # 2304 x 2
}


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("name", list(FEW))
def test_shared_slices_match_oracle(iwf, name, dtype):  # noqa: F811
    pb = FEW[name]
    plan = _plan(iwf, pb)
    for nvec in (1, 2, 6):
        _check(plan, pb, dtype, nvec, launches=1, iwf=iwf)


def test_batch_on_few_slices_matches_dense(iwf):  # noqa: F811
    P, K, L = np.array([[1.0, 5.0 ** 0.5]]), (150,), (1,)
    pots = [W.cosine_modes(2, 1.0), W.cosine_modes(2, 0.6, phases=[0.4, 2.2], const=0.5)]
    plan = iwf.Plan(P, K, L)
    ev, _, _, _, info = plan.batch_eigensolve(pots, 3, block=6)
    assert info["converged"] == 1
    win = O.build_window(P, K, L)
    for q, (m, c) in enumerate(pots):
        ref = O.eigen.dense_eigs(win, O.grid_coefficients(m, c, win.lens), 3)[0]
        assert np.all(np.abs(ev[q] - ref) <= 1e-10 * np.maximum(1.0, np.abs(ref))), q


@pytest.mark.parametrize("nvec", [1, 4])
def test_few_slices_are_no_slower_than_the_transforms(iwf, nvec):  # noqa: F811
    pb = _problem(4, 5, (4, 4, 4, 4), (8,), _axis_modes(5, 48, 9, True))              # 8^4 x 16
    plan = _plan(iwf, pb)
    x = torch.from_numpy(np.ascontiguousarray(W.random_block(plan.N, nvec, seed=1).T)).cuda()
    y = torch.empty_like(x)

    def best():
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        plan.apply(x, y)
        times = []
        for _ in range(5):
            e0.record()
            for _ in range(20):
                plan.apply(x, y)
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        return min(times)

    direct = best()
    plan.set_path("f64", "tiled")
    assert direct <= 1.5 * best()

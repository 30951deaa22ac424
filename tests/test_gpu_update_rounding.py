"""Rounding of the tensor-core block update where the leading bits of a sum cancel, against exact
integer arithmetic.

Every row has magnitudes in [1/2, 1), every coefficient too, so that the scales are 1 and the
values' digits exact; Im S = Re S and Im C = Re C up to 2^-12, so that Re Y = sum Re S Re C -
Im S Im C is small and its FP64 rounding negligible. What is left: the digit pairs above level 10
(dropped: rms 1365 sqrt(12 m) 2^-63 units of 2^-12 for digits of rms 37), the one rounding of the sum
of levels 7..10 to 24 bits (its rms is 1365 sqrt(12 m) = 2^12.2 sqrt(m) of its unit 2^-35, so the
rounding's is 2^-12.8 sqrt(m) of it) and the assembly's last place, 2^-49: together 2^-47.8 sqrt(m)
of 2^-12. The bound is 1.3 bits above that; an assembly that rounds at 2^-42 lies at 2^-43.8.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _near(rng, shape):
    a = rng.uniform(0.51, 0.98, size=shape) * rng.choice([-1.0, 1.0], size=shape)
    return a, a + rng.uniform(-1.0, 1.0, size=shape) * 2.0 ** -12


def _exact(a):
    return np.vectorize(lambda v: int(v * 2.0 ** 53), otypes=[object])(a)


@pytest.mark.parametrize("subtract", [False, True])
@pytest.mark.parametrize("m,q", [(1, 1), (3, 2), (8, 2), (24, 3)])
def test_cancelling_sums(m, q, subtract):
    import paper_2404_04507_gb300 as iwf
    rng = np.random.default_rng(m)
    nrows = 1500
    (sr, si), (cr, ci) = _near(rng, (m, nrows)), _near(rng, (m, q))
    S, Cm = torch.from_numpy(sr + 1j * si).cuda(), torch.from_numpy(cr + 1j * ci).cuda()
    if subtract:
        Y = torch.zeros((q, nrows), dtype=torch.complex128, device="cuda")
        iwf.block_update(S, Cm, Y=Y, subtract=True)
        Y = -Y
    else:
        Y = iwf.block_update(S, Cm)
    got = Y.cpu().numpy().real
    want = _exact(cr).T.dot(_exact(sr)) - _exact(ci).T.dot(_exact(si))      # in units of 2^-106
    err = (np.vectorize(lambda v: int(v * 2.0 ** 106), otypes=[object])(got) - want).astype(float) * 2.0 ** -106
    assert np.sqrt(np.mean(err ** 2)) <= 2.0 ** -58.5 * np.sqrt(m)

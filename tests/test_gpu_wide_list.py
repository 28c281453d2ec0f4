"""The one-candidate-per-lane list build of small passes against the per-thread build
(variant 0): the same words in the same order. Sizes at the edges of its spans (8, 16
and 32 slots), runs of many cells (low density), cells fuller than one round of
staged candidates, one-cell boxes, both list kinds."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu

CASES = [  # n, density, rc, half
    (33, 0.3, 1.9, False), (500, 0.85, 2.5, False), (1000, 0.8442, 2.5, False), (1000, 0.8442, 2.5, True),
    (4863, 0.8, 2.5, False), (4865, 0.8, 3.0, True), (9729, 0.7, 2.5, False), (2000, 0.02, 2.5, False),
    (3000, 1.6, 3.9, False), (41600, 0.75, 2.5, False), (41601, 0.75, 2.5, False),
]


@pytest.mark.parametrize("n,rho,rc,half", CASES)
def test_same_list_words(n, rho, rc, half):
    from paper_1210_3450_gb300 import MD_FP32_FORCE, LJSystem
    from paper_1210_3450_gb300.ljmd import MD_LIST_HALF
    x, box = li.perturbed_fcc(n, rho, 0.1, n)
    got = []
    with LJSystem(box, n, rc, 0.3, MD_FP32_FORCE) as s:
        if half:
            s.set_pair_list(MD_LIST_HALF)
        for variant in (5, 0):
            s.set_tuning(list_variant=variant)
            s.set_state(x, np.zeros_like(x))
            got.append(s.get_list())
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_position_not_finite_in_one_cell(precision, value):
    """A one-cell box in which a position is not finite: the particle has no partners, as in
    the other builds, and the other forces are those without it."""
    from paper_1210_3450_gb300 import LJSystem
    n = 60
    x, box = li.perturbed_fcc(n, 0.3, 0.05, 5)
    x = np.mod(x - x[3] + 0.4, box)  # a partner in reach of the origin
    x[7, 1] = value
    got = []
    for keep in (np.arange(n), np.delete(np.arange(n), 7)):
        with LJSystem(box, len(keep), 1.9, 0.3, precision) as s:
            s.set_state(x[keep], np.zeros((len(keep), 3)))
            start, partners = s.get_list()
            got.append(s.forces())
        if len(keep) == n:
            assert start[8] == start[7] and not (partners == 7).any()
    assert box < 3 * 2.2
    rms = np.sqrt((got[1] ** 2).sum(1).mean())
    assert np.abs(np.delete(got[0], 7, 0) - got[1]).max() <= (1e-12 if precision == 0 else 1e-5) * rms

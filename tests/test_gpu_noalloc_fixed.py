"""The fixed-point form of md_forces_noalloc at the edges of its ranges (threads per
particle, cutoff, cell side, pairs per particle) against the oracle at the FP64
tolerance; each case twice, bit for bit equal. A position that is not finite has no
pairs and leaves the other particles' forces finite."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu

CASES = [  # n, density, rc
    (500, 0.8, 2.5), (2432, 0.8442, 2.5), (2433, 0.6, 3.0), (4000, 0.85, 3.99), (4000, 0.85, 4.0),
    (1100, 0.5, 3.98),           # cells wider than 3.99: the FP64 form
    (3150, 1.9, 3.9),            # more pairs than the 96-bit sums take
    (19456, 0.7, 2.5), (19457, 0.7, 2.5), (65535, 0.6, 3.0),
]


def _forces(ljmd, x, box, rc):
    import torch
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    fd = torch.full_like(xd, float("nan"))
    ljmd.forces_noalloc(xd, box, rc, fd)
    torch.cuda.synchronize()
    return fd.cpu().numpy()


@pytest.mark.parametrize("n,rho,rc", CASES)
def test_matches_oracle(ljmd, oracle, n, rho, rc):
    x, box = li.perturbed_fcc(n, rho, 0.08, n)
    ref = oracle.forces(x, box, rc)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    a, b = _forces(ljmd, x, box, rc), _forces(ljmd, x, box, rc)
    assert np.abs(a - ref).max() <= 1e-12 * rms
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_position_not_finite(ljmd, oracle, value):
    x, box = li.perturbed_fcc(2000, 0.8, 0.08, 9)
    ref = oracle.forces(np.delete(x, 7, 0), box, 2.5)
    x[7, 1] = value
    f = _forces(ljmd, x, box, 2.5)
    assert np.isfinite(np.delete(f, 7, 0)).all()
    assert np.abs(np.delete(f, 7, 0) - ref).max() <= 1e-12 * np.sqrt((ref ** 2).sum(1).mean())


@pytest.mark.parametrize("rc", [1e-2, 1e-4, 1e-6, 1e-7, 1e-9])
def test_short_cutoffs(ljmd, rc):
    """Pairs at 0.3 to 0.999 of cutoffs near and below the resolution of the candidate test:
    each force within 1e-12 of its terms in numpy's FP64 (a few tens of roundings)."""
    m = 6
    g = np.random.Generator(np.random.PCG64(41))
    k = np.arange(m ** 3)
    c = np.stack([k % m, k // m % m, k // m ** 2], 1) / m + 0.05 + g.uniform(0, 0.05, (m ** 3, 3))
    u = g.standard_normal((m ** 3, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x = np.concatenate([c, c + u * (rc * np.linspace(0.3, 0.999, m ** 3))[:, None]])
    d = x[m ** 3:] - x[:m ** 3]
    y = 1.0 / (d * d).sum(1)
    yc = rc ** -2.0
    inside = y > yc
    assert inside.sum() > 0.9 * m ** 3
    f = ((24 * y ** 4 - 48 * y ** 7 + 8 * (6 * yc ** 7 - 3 * yc ** 4)) * inside)[:, None] * d
    size = (24 * y ** 4 + 48 * y ** 7 + 8 * (6 * yc ** 7 + 3 * yc ** 4)) / np.sqrt(y)
    got = _forces(ljmd, x, 1.0, rc)
    for a, b in ((got[:m ** 3], f), (got[m ** 3:], -f)):
        assert (np.abs(a - b).max(1) <= 1e-12 * size).all()

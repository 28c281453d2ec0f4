"""Forces of pairs at every distance up to the cutoff, each against exact rational
arithmetic: the FP64 form is as accurate for a weak pair, relative to its own terms, as
for a close one, in every loop that computes it.

Bound (u = 2^-53, y = 1 / r^2, yc at the cutoff), the worst case of the FP64 operations of
Eq. 1's factor: r^2 within 2 u and the reciprocal within 1.5 u give y^4 and y^7 within
4 x 3.5 + 2 = 16 u and 7 x 3.5 + 4 = 28.5 u, c2 has 6 roundings, and the factor, its product
with the separation and the sum two more:
|F| errs by at most u |d| (18 x 24 y^4 + 30.5 x 48 y^7 + 8 x 8 (6 yc^7 + 3 yc^4)) per pair."""
from fractions import Fraction as Q

import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _dimers(rc, box, m):
    """m^3 pairs at distances from 0.9 to rc in random directions, in a box of m cells."""
    g = np.random.Generator(np.random.PCG64(17))
    k = np.arange(m ** 3)
    c = np.stack([k % m, k // m % m, k // m ** 2], 1) * (box / m) + 4.2 + g.uniform(0, 0.5, (m ** 3, 3))
    u = g.standard_normal((m ** 3, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    return np.mod(np.concatenate([c, c + u * np.linspace(0.9, rc, m ** 3)[:, None]]), box)


def _exact(x, box, rc):
    """Forces as exact rationals and their bounds, minimum image."""
    n = len(x)
    d = x[None, :, :] - x[:, None, :]
    k = np.round(d / box)
    r2 = ((d - box * k) ** 2).sum(2)
    rq = Q(rc) ** 2
    c2 = 6 / rq ** 7 - 3 / rq ** 4
    yc = rc ** -2.0
    f, bound = [[Q(0)] * 3 for _ in range(n)], np.zeros(n)
    xq = [[Q(v) for v in p] for p in x.tolist()]
    for i, j in np.argwhere((r2 < rc * rc * (1 + 1e-9)) & ~np.eye(n, dtype=bool)).tolist():
        s = [b - a - int(q) * Q(box) for a, b, q in zip(xq[i], xq[j], k[i, j])]
        rr = sum(v * v for v in s)
        if not rr < rq:
            continue
        y = 1 / rr
        g = 24 * y ** 4 - 48 * y ** 7 + 8 * c2
        f[i] = [a + g * v for a, v in zip(f[i], s)]
        z = float(y)
        bound[i] += U * float(rr) ** 0.5 * (18 * 24 * z ** 4 + 30.5 * 48 * z ** 7 + 64 * (6 * yc ** 7 + 3 * yc ** 4))
    return f, bound


def _check(f, exact):
    ref, bound = exact
    for a, r, b in zip(f.tolist(), ref, bound):
        err = sum((Q(v) - w) ** 2 for v, w in zip(a, r))
        assert float(err) ** 0.5 <= b


@pytest.mark.parametrize("rc,box,m", [(2.5, 47.0, 5), (3.9, 47.0, 5), (3.99, 47.5, 5)])
def test_each_pair_within_its_own_terms(ljmd, rc, box, m):
    import torch
    x = _dimers(rc, box, m)
    v = np.zeros_like(x)
    exact = _exact(x, box, rc)
    with ljmd.LJSystem(box, len(x), rc, 0.3) as s:
        for queue in (1, 0):
            s.set_tuning(fp64_queue=queue)
            s.set_state(x, v)
            _check(s.forces(), exact)
        s.set_state(x, v)
        s.step(1, 0.0)  # the persistent loop's closing forces, at the same positions
        _check(s.forces(), exact)
    xd = torch.from_numpy(x).cuda()
    fd = torch.empty_like(xd)
    ljmd.forces_noalloc(xd, box, rc, fd)
    torch.cuda.synchronize()
    _check(fd.cpu().numpy(), exact)


def test_dilute_gas(ljmd):
    """Most particles with one or two far partners, at the longest cutoff of the range."""
    x, box = li.perturbed_fcc(256, 0.02, 1.2, 19)
    exact = _exact(x, box, 3.9)
    with ljmd.LJSystem(box, len(x), 3.9, 0.3) as s:
        s.set_state(x, np.zeros_like(x))
        _check(s.forces(), exact)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("half", [False, True], ids=["full", "half"])
def test_energy_and_virial_of_weak_pairs(ljmd, half, precision):
    """125 pairs near the cutoff. With the errors above, r^-12 within 6 x 3.5 + 3 = 24 u and
    r^-6 within 12.5 u; the sums, their products with the coefficients (8 roundings in c2
    and c0) and the final sums 3 more."""
    from paper_1210_3450_gb300.ljmd import MD_LIST_HALF
    rc, box, m = 3.99, 50.0, 5
    x = _dimers(rc, box, m)
    x[125:] = x[:125] + (x[125:] - x[:125]) * (np.linspace(3.5, 3.989, 125) / np.linspace(0.9, rc, 125))[:, None]
    rq = Q(rc) ** 2
    c2, c0 = 6 / rq ** 7 - 3 / rq ** 4, 4 / rq ** 3 - 7 / rq ** 6
    d = x[None, :, :] - x[:, None, :]
    k = np.round(d / box)
    near = np.argwhere(np.triu(((d - box * k) ** 2).sum(2) < rc * rc * (1 + 1e-9), 1))
    pe, w, bound = Q(0), Q(0), np.zeros(2)
    for i, j in near.tolist():
        rr = sum((Q(b) - Q(a) - int(q) * Q(box)) ** 2 for a, b, q in zip(x[i].tolist(), x[j].tolist(), k[i, j]))
        if rr < rq:
            s = 1 / rr ** 3
            pe += 4 * (s * s - s) + 4 * (c2 * rr + c0)
            w += 48 * s * s - 24 * s - 8 * c2 * rr
            s, k2, k0 = float(s), abs(float(c2 * rr)), abs(float(c0))
            bound += U * np.array([4 * (27 * s * s + 15.5 * s + 11 * k2 + 11 * k0), 48 * 27 * s * s + 24 * 15.5 * s + 88 * k2])
    assert len(near) >= 125
    with ljmd.LJSystem(box, len(x), rc, 0.3, precision) as s:
        if half:
            s.set_pair_list(MD_LIST_HALF)
        s.set_state(x, np.zeros_like(x))
        o = s.observables()
    assert abs(float(Q(o["pe"]) - pe)) <= bound[0]
    assert abs(float(Q(o["virial"]) - w)) <= bound[1]


def test_virial_of_many_pairs_has_no_bias(ljmd):
    """The virial of 64,000 close pairs against integers of 200 bits: independent rounding
    errors of the pairs, each of the worst case above, add up to less than 4 times the
    square root of their number (1.6 % of the sum of the worst cases)."""
    m, box, rc = 40, 240.0, 2.5
    g = np.random.Generator(np.random.PCG64(23))
    k = np.arange(m ** 3)
    c = np.stack([k % m, k // m % m, k // m ** 2], 1) * 6.0 + 1.5 + g.uniform(0, 0.5, (m ** 3, 3))
    u = g.standard_normal((m ** 3, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x = np.concatenate([c, c + u * g.uniform(1.0, 1.2, m ** 3)[:, None]])
    one = 1 << 60  # positions of 2^-8 and more are whole numbers of 2^-60
    q = np.array([[int(v * 2.0 ** 45) << 15 if v >= 128 else int(v * one) for v in p] for p in x.tolist()], dtype=object)
    d = q[m ** 3:] - q[:m ** 3]
    rr = (d * d).sum(1)                                      # 2^-120
    y = np.array([(1 << 320) // v for v in rr.tolist()], dtype=object)  # 2^-200
    s = np.array([v * v * v >> 400 for v in y.tolist()], dtype=object)  # 2^-200
    s6, s12 = sum(s.tolist()), sum(v * v >> 200 for v in s.tolist())
    rq = Q(rc) ** 2
    w = Q(48 * s12 - 24 * s6, 1 << 200) - 8 * (6 / rq ** 7 - 3 / rq ** 4) * Q(sum(rr.tolist()), 1 << 120)
    worst = U * (48 * 27 * float(Q(s12, 1 << 200)) + 24 * 15.5 * float(Q(s6, 1 << 200)))
    with ljmd.LJSystem(box, len(x), rc, 0.3) as h:
        h.set_state(x, np.zeros_like(x))
        got = h.observables()["virial"]
    assert abs(float(Q(got) - w)) <= 4.0 / m ** 1.5 * worst

"""Fixed-point pair arithmetic of the FP64 form at the edges of its range: the change
to the FP64 pipe at close pairs, at long lists and at large cutoffs, positions at both
ends of a large box, pairs at the cutoff. The bound is the FP64 form's 1e-12 of the
rms force; both force loops give the same bits."""
import numpy as np
import pytest

import lj_inputs as li
import oracle

pytestmark = pytest.mark.gpu


def _dimers(r, box, seed):
    """Pairs at the given distances in random directions, the pairs 7 apart."""
    g = np.random.Generator(np.random.PCG64(seed))
    m = int(box // 7.0)
    k = np.arange(len(r))
    assert m ** 3 >= len(r)
    c = np.stack([k % m, k // m % m, k // m ** 2], 1) * 7.0 + 0.5 + g.uniform(0, 0.5, (len(r), 3))
    u = g.standard_normal((len(r), 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    return np.mod(np.concatenate([c, c + u * r[:, None]]), box)


def _case(name):
    if name == "close":  # around r^2 = 0.84, where the fixed-point range ends
        r = np.concatenate([np.sqrt(0.84) * (1 + np.linspace(-1e-6, 1e-6, 41)), np.linspace(0.7, 1.1, 59)])
        return _dimers(r, 40.0, 1), 40.0, 2.5
    if name == "cutoff":
        r = np.concatenate([2.5 * (1 + np.linspace(-1e-9, 1e-9, 41)), np.linspace(2.3, 2.7, 59)])
        return _dimers(r, 40.0, 2), 40.0, 2.5
    if name == "far corner":  # positions near 0 and near a large L, pairs across every face
        r = np.linspace(0.9, 2.6, 60)
        x = _dimers(r, 30.0, 3)
        x[::3] += 1200.5 - 15.0
        x[1::3] -= 15.0
        return np.mod(x, 1200.5), 1200.5, 2.5
    if name == "long lists":  # more partners than the 96-bit sums take, some below the limit
        x, box = li.perturbed_fcc(3001, 1.5, 0.02, 4)
        keep = (x[:, 0] < 0.55 * box) | (np.arange(len(x)) % 3 == 0)
        return np.ascontiguousarray(x[keep]), box, 3.9
    if name == "rc 3.99":
        return *li.perturbed_fcc(2000, 0.85, 0.1, 5), 3.99
    if name == "rc 4.0":
        return *li.perturbed_fcc(2000, 0.85, 0.1, 6), 4.0
    return *li.perturbed_fcc(33, 0.3, 0.05, 7), 1.9  # one cell: every pair a candidate


@pytest.mark.parametrize("name", ["close", "cutoff", "far corner", "long lists", "rc 3.99", "rc 4.0", "small"])
def test_forces_at_the_edges(name):
    from paper_1210_3450_gb300 import MD_FP64, LJSystem
    x, box, rc = _case(name)
    ref = oracle.forces_brute(x, box, rc)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    got = []
    with LJSystem(box, len(x), rc, 0.3, MD_FP64) as s:
        for queue in (1, 0):
            s.set_tuning(fp64_queue=queue)
            s.set_state(x, np.zeros_like(x))
            got.append(s.forces())
        if name == "long lists":
            cnt = np.diff(s.get_list()[0])
            assert cnt.min() <= 448 < cnt.max()
    np.testing.assert_array_equal(got[0], got[1])
    assert np.abs(got[0] - ref).max() <= 1e-12 * rms


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("half", [False, True], ids=["full", "half"])
@pytest.mark.parametrize("name", ["close", "cutoff", "far corner", "long lists", "rc 4.0", "small"])
def test_energy_and_virial_at_the_edges(name, half, precision):
    """Potential energy and virial (each pair once, fixed-point sums) within 1e-12 of the
    oracle's, relative to the sum of the pairs' magnitudes."""
    from paper_1210_3450_gb300 import LJSystem
    from paper_1210_3450_gb300.ljmd import MD_LIST_HALF
    x, box, rc = _case(name)
    v = li.maxwell_boltzmann(len(x), 1.0, 3)
    d = x[:, None, :] - x[None, :, :]
    d -= box * np.round(d / box)
    r2 = (d ** 2).sum(2)[np.triu_indices(len(x), 1)]
    r2 = r2[r2 < rc * rc]
    scale = (4 * r2 ** -6 + 4 * r2 ** -3).sum(), (48 * r2 ** -6 + 24 * r2 ** -3).sum()
    ref = oracle.observables(x, v, box, rc)
    with LJSystem(box, len(x), rc, 0.3, precision) as s:
        if half:
            s.set_pair_list(MD_LIST_HALF)
        s.set_state(x, v)
        got = s.observables()
    assert abs(got["pe"] - ref["pe"]) <= 1e-12 * scale[0]
    assert abs(got["virial"] - ref["virial"]) <= 1e-12 * scale[1]
    assert abs(got["ke"] - ref["ke"]) <= 1e-12 * ref["ke"]


def test_leaving_and_entering_the_fixed_point_form():
    """Positions in pair units are held only by the FP64 form's full lists: changing the
    precision or the list kind and back gives the same forces and steps bit for bit."""
    from paper_1210_3450_gb300 import MD_FP64, LJSystem
    from paper_1210_3450_gb300.ljmd import MD_LIST_FULL, MD_LIST_HALF
    x, box = li.perturbed_fcc(864, 0.8442, 0.1, 5)
    v = li.maxwell_boltzmann(864, 0.7, 6)

    def run(s):
        s.set_state(x, v)
        f = s.forces()
        s.step(20, 0.005)
        return (f,) + tuple(s.get_state())

    with LJSystem(box, 864, 2.5, 0.3, MD_FP64) as s:
        ref = run(s)
        s.set_precision(1)
        run(s)
        s.set_precision(MD_FP64)
        again = run(s)
        s.set_pair_list(MD_LIST_HALF)
        run(s)
        s.set_pair_list(MD_LIST_FULL)
        for got in (again, run(s)):
            for p, q in zip(ref, got):
                np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("rho,amp", [(1.5, 0.02), (6.6, 0.01)])
def test_lists_beyond_the_sums(rho, amp):
    """Lists around 448 and 1,880 partners, where the range of the fixed-point pairs is cut
    back, in the same warps as shorter ones: every force within 1e-12 of the rms force of its
    own kind of list, both force loops equal."""
    from paper_1210_3450_gb300 import MD_FP64, LJSystem
    x, box = li.perturbed_fcc(6000, rho, amp, 8)
    keep = (x[:, 0] < 0.6 * box) | (np.arange(len(x)) % 3 == 0)
    x = np.ascontiguousarray(x[keep])
    ref = oracle.forces_brute(x, box, 3.9)
    size = np.sqrt((ref ** 2).sum(1))
    got = []
    with LJSystem(box, len(x), 3.9, 0.3, MD_FP64) as s:
        for queue in (1, 0):
            s.set_tuning(fp64_queue=queue)
            s.set_state(x, np.zeros_like(x))
            got.append(s.forces())
        cnt = np.diff(s.get_list()[0])
    limit = 448 if rho < 2 else 1880
    assert cnt.min() <= limit < cnt.max()
    np.testing.assert_array_equal(got[0], got[1])
    for part in (cnt <= limit, cnt > limit):
        rms = np.sqrt((size[part] ** 2).mean())
        assert np.abs(got[0] - ref)[part].max() <= 1e-12 * rms

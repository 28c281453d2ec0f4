"""Arenas without, with only and with some systems in the range of the fixed-point pairs
(rc <= 3.99): every system as it runs alone, bit for bit, when one of the others joins or
leaves, with and without pair queues, and forces within the FP64 form's 1e-12."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("queue", [0, 1])
def test_mixed_arena(ljmd, oracle, queue):
    spec = [(1500, 0.7, 4.5), (1200, 0.8, 2.5), (1100, 0.6, 4.0)]
    syss = []
    for k, (n, rho, rc) in enumerate(spec):
        x, box = li.perturbed_fcc(n, rho, 0.1, 90 + k)
        syss.append((n, box, rc, x, li.maxwell_boltzmann(n, 1.0, 95 + k)))
    alone = []
    for n, box, rc, x, v in syss:
        with ljmd.LJSystem(box, n, rc, 0.3) as s:
            s.set_tuning(fp64_queue=queue)
            s.set_state(x, v)
            f = s.forces()
            ref = oracle.forces(x, box, rc)
            assert np.abs(f - ref).max() <= 1e-12 * np.sqrt((ref ** 2).sum(1).mean())
            got = []
            for steps in (21, 20, 13):
                s.step(steps, 0.004)
                o = s.observables()
                got.append([*s.get_state(), s.forces(), np.array([o["pe"], o["virial"]])])
            alone.append(got)
    foot = [ljmd.footprint(n, box, rc, 0.3) for n, box, rc, _, _ in syss]
    with ljmd.LJBatch(arena=dict(slots=8192, cells=1 << 15, list_words=4 * sum(f["list_words"] for f in foot),
                                 max_systems=8)) as b:
        b.set_tuning(fp64_queue=queue)

        def add(k):
            n, box, rc, x, v = syss[k]
            i = b.add(n, box, rc, 0.3)
            b.set_state(i, x, v)
            return i

        def same(i, k, turn):
            o = b.observables([i])[i]
            for p, q in zip([*b.get_state(i), b.forces(i), o[:2]], alone[k][turn]):
                np.testing.assert_array_equal(p, q)

        i0 = add(0)  # none in the range
        b.step(21, 0.004)
        same(i0, 0, 0)
        i1 = add(1)  # some
        b.step(20, 0.004)
        same(i0, 0, 1)
        b.step(1, 0.004)
        same(i1, 1, 0)
        b.remove(i0)  # only
        b.step(20, 0.004)
        same(i1, 1, 1)
        i2 = add(2)
        b.step(13, 0.004)
        same(i1, 1, 2)
        b.remove(i1)  # none
        b.step(8, 0.004)
        same(i2, 2, 0)
        b.step(20, 0.004)
        same(i2, 2, 1)


@pytest.mark.parametrize("mode", [2, 3, 4, 5])
def test_reciprocal_modes_queue(ljmd, mode):
    x, box = li.perturbed_fcc(1500, 0.8, 0.1, 99)
    got = []
    with ljmd.LJSystem(box, 1500, 2.5, 0.3, mode) as s:
        for queue in (1, 0):
            s.set_tuning(fp64_queue=queue)
            s.set_state(x, np.zeros_like(x))
            got.append(s.forces())
    np.testing.assert_array_equal(got[0], got[1])

"""Wide skins in dilute FP64 systems: listed pairs come apart by rc + 2 skin before the
list is rebuilt, past the 8 length units that separations in pair units can hold. The
persistent loop, the graph loop and the host loop, with and without pair queues, agree
bit for bit, with the oracle's trajectory within 1e-9, and the closing forces with an
all-pairs sum."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu

N, BOX = 500, 40.0


def _gas(seed):
    """Uniform positions, no two closer than 0.95."""
    g = np.random.Generator(np.random.PCG64(seed))
    x = np.empty((0, 3))
    while len(x) < N:
        p = g.uniform(0, BOX, 3)
        d = x - p
        d -= BOX * np.round(d / BOX)
        if not len(x) or (d * d).sum(1).min() > 0.95 ** 2:
            x = np.vstack([x, p])
    return x


@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
@pytest.mark.parametrize("rule", [0, 1], ids=["displacement", "velocity"])
@pytest.mark.parametrize("rc,skin", [(2.5, 2.6), (2.5, 2.75), (2.5, 4.0), (3.9, 4.0), (2.5, 6.0), (3.9, 6.0), (2.5, 12.0),
                                     (3.9, 12.0)])
def test_all_loops_agree(ljmd, oracle, rc, skin, rule, nvt):
    x, v = _gas(31), li.maxwell_boltzmann(N, 2.0, 32)
    q = 3.0 * N * 0.5
    out = []
    for graph in (0, 1):
        for queue in (0, 1):
            with ljmd.LJSystem(BOX, N, rc, skin) as s:
                s.set_tuning(graph=graph, fp64_queue=queue)
                s.set_validity_rule(rule)
                s.set_state(x, v)
                ze = s.step_nvt(150, 0.005, 2.0, q) if nvt else s.step(150, 0.005)
                out.append([*s.get_state(), s.forces(), np.array(ze if nvt else [0.0])])
    for o in out[1:]:
        for a, b in zip(out[0], o):
            np.testing.assert_array_equal(a, b)
    xs, vs, f = out[0][:3]
    ref = oracle.run_nvt(x, v, BOX, rc, skin, 150, 0.005, 2.0, q) if nvt else oracle.run(x, v, BOX, rc, skin, 150, 0.005)
    d = xs - ref["x"]
    d -= BOX * np.round(d / BOX)
    assert np.abs(d).max() < 1e-9
    assert np.abs(f - oracle.forces_brute(xs, BOX, rc)).max() < 1e-9

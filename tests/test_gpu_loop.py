"""The persistent step loop of small arenas against the host-driven loop: positions,
velocities, forces and rebuild counts bit for bit, at the edges of its ranges of
threads per particle, with pairs below the fixed-point range (few and many per
particle), under the velocity bound, in a batch with a paused system, over odd and
single steps."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu


def _run(ljmd, n, rho, rc, amp, temp, precision, graph, calls, dt, rule=0):
    x, box = li.perturbed_fcc(n, rho, amp, n)
    v = li.maxwell_boltzmann(n, temp, n + 1)
    with ljmd.LJSystem(box, n, rc, 0.3, precision) as s:
        s.set_tuning(graph=graph)
        s.set_validity_rule(rule)
        s.set_state(x, v)
        for k in calls:
            s.step(k, dt)
        return (*s.get_state(), s.forces(), s.stats())


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("n,rho,rc,amp,temp,calls,dt,rule", [
    (33, 0.3, 1.9, 0.05, 1.0, (40,), 0.005, 0),
    (2432, 0.8442, 2.5, 0.1, 0.722, (25, 1, 4), 0.005, 0),
    (2433, 0.8442, 2.5, 0.1, 0.722, (25, 1), 0.005, 1),
    (4864, 0.7, 3.0, 0.1, 1.2, (21,), 0.005, 0),
    (4865, 0.7, 3.0, 0.1, 1.2, (20, 3), 0.005, 0),
    (9729, 0.6, 2.5, 0.1, 0.9, (20,), 0.005, 0),
    (29185, 0.8, 2.5, 0.1, 0.9, (12,), 0.005, 0),
    (38912, 0.8, 2.5, 0.1, 0.9, (12,), 0.005, 0),
    (1000, 1.05, 2.5, 0.12, 2.0, (30,), 0.001, 0),   # close pairs in most lists
    (1500, 1.6, 2.5, 0.05, 1.0, (12,), 0.0005, 0),   # every list holds many
])
def test_equals_host_loop(ljmd, n, rho, rc, amp, temp, calls, dt, rule, precision):
    a = _run(ljmd, n, rho, rc, amp, temp, precision, 0, calls, dt, rule)
    b = _run(ljmd, n, rho, rc, amp, temp, precision, 1, calls, dt, rule)
    for p, q in zip(a[:3], b[:3]):
        np.testing.assert_array_equal(p, q)
    assert a[3] == b[3]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_batch_with_a_paused_system(ljmd, precision):
    specs, states = [], []
    for k, (n, rho) in enumerate([(700, 0.8), (1500, 0.7), (513, 0.6), (300, 0.85)]):
        x, box = li.perturbed_fcc(n, rho, 0.1, 40 + k)
        specs.append((n, box, 2.5, 0.3))
        states.append((x, li.maxwell_boltzmann(n, 1.0, 50 + k)))
    out = []
    for graph in (0, 1):
        with ljmd.LJBatch(systems=specs, precision=precision) as b:
            b.set_tuning(graph=graph)
            for k, (x, v) in enumerate(states):
                b.set_state(k, x, v)
            b.step(15, 0.005)
            b.set_active(1, False)
            b.step(21, [0.005, 0.0, 0.004, 0.003])
            b.set_active(1, True)
            b.step(10, 0.005)
            out.append([(*b.get_state(k), b.forces(k), b.stats(k)) for k in range(4)])
    for p, q in zip(*out):
        for a, c in zip(p[:3], q[:3]):
            np.testing.assert_array_equal(a, c)
        assert p[3] == q[3]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("n,rho,rc", [(500, 0.85, 2.5), (2433, 0.7, 3.0), (9729, 0.6, 2.5)])
def test_nvt_equals_host_loop(ljmd, n, rho, rc, precision):
    x, box = li.perturbed_fcc(n, rho, 0.1, n)
    v = li.maxwell_boltzmann(n, 1.3, n + 1)
    out = []
    for graph in (0, 1):
        with ljmd.LJSystem(box, n, rc, 0.3, precision) as s:
            s.set_tuning(graph=graph)
            s.set_state(x, v)
            z, e = s.step_nvt(24, 0.005, 0.9, 3.0 * n * 0.05)
            z, e = s.step_nvt(1, 0.005, 0.9, 3.0 * n * 0.05, z, e)
            s.step(3, 0.005)
            out.append((*s.get_state(), s.forces(), np.array([z, e]), s.stats()))
    for p, q in zip(out[0][:4], out[1][:4]):
        np.testing.assert_array_equal(p, q)
    assert out[0][4] == out[1][4]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
def test_first_lists_overflow(ljmd, precision, nvt):
    """A dense block in a wide box: the first list build of the launch outgrows the
    capacity expected from the density, is grown by the host and taken up again."""
    n = 1372
    x, box = li.perturbed_fcc(n, 0.9, 0.05, 5)
    x, box = x + 0.1, 2.0 * box
    v = li.maxwell_boltzmann(n, 0.7, 6)
    out = []
    for graph in (0, 1):
        with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
            s.set_tuning(graph=graph)
            s.set_state(x, v)
            ze = s.step_nvt(12, 0.004, 0.7, 3.0 * n * 0.05) if nvt else s.step(12, 0.004)
            out.append((*s.get_state(), s.forces(), ze, s.stats()))
    for p, q in zip(out[0][:3], out[1][:3]):
        np.testing.assert_array_equal(p, q)
    assert out[0][3:] == out[1][3:]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_several_threads(ljmd, precision):
    """Systems stepped by threads of their own at the same time, each on its stream: every
    one as it runs alone, bit for bit."""
    from concurrent.futures import ThreadPoolExecutor
    args = [(n, rho, 2.5, 0.1, 0.9, precision, 1, (30, 7, 30), 0.005)
            for n, rho in ((1000, 0.8442), (9729, 0.6), (29185, 0.8), (29185, 0.75))]
    alone = [_run(ljmd, *a) for a in args]
    with ThreadPoolExecutor(len(args)) as pool:
        together = list(pool.map(lambda a: _run(ljmd, *a), args))
    for a, b in zip(alone, together):
        for p, q in zip(a[:3], b[:3]):
            np.testing.assert_array_equal(p, q)
        assert a[3] == b[3]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
def test_more_steps_than_a_launch(ljmd, precision, nvt):
    """A call of more steps than the loop takes in one launch, an odd number of launches."""
    n, steps = 108, 4003
    x, box = li.perturbed_fcc(n, 0.3, 0.1, 3)
    v = li.maxwell_boltzmann(n, 1.0, 4)
    out = []
    for graph in (0, 1):
        with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
            s.set_tuning(graph=graph)
            s.set_state(x, v)
            ze = s.step_nvt(steps, 0.002, 1.0, 3.0 * n * 0.05) if nvt else s.step(steps, 0.002)
            out.append((*s.get_state(), s.forces(), np.array(ze if nvt else [0.0]), np.array(list(s.stats().values()))))
    for p, q in zip(*out):
        np.testing.assert_array_equal(p, q)


def test_several_threads_share_the_device(ljmd):
    """Handles stepped at the same time take smaller launches or graph launches: the same
    results, NVE and Nose-Hoover, over several calls."""
    from concurrent.futures import ThreadPoolExecutor
    cases = [(1000 + 700 * (k % 5), k % 2, k % 3 == 0) for k in range(10)]

    def run(case):
        n, precision, nvt = case
        x, box = li.perturbed_fcc(n, 0.8, 0.1, n)
        v = li.maxwell_boltzmann(n, 0.9, n + 1)
        with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
            s.set_state(x, v)
            ze = [0.0, 0.0]
            for steps in (40, 1, 33, 80):
                if nvt:
                    ze = s.step_nvt(steps, 0.004, 0.9, 3.0 * n * 0.05, *ze)
                else:
                    s.step(steps, 0.004)
            return (*s.get_state(), s.forces(), np.array(ze))

    alone = [run(c) for c in cases]
    with ThreadPoolExecutor(len(cases)) as pool:
        together = list(pool.map(run, cases))
    for a, b in zip(alone, together):
        for p, q in zip(a, b):
            np.testing.assert_array_equal(p, q)

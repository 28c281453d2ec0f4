"""Lists that outgrow their capacity under the persistent step loop: grown within an
arena's spare words, grown twice in a system of exact size, past the longest list of the
fixed-point sums, and in the middle of a call. Positions, velocities, forces, thermostat
and rebuild counts equal the host-driven loop's bit for bit."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu

N = 1372


def _block(rho, box, amp=0.03):
    """A dense block in the middle of a wide box."""
    x, side = li.perturbed_fcc(N, rho, amp, 11)
    assert side < box - 4.6
    return x + 0.5 * (box - side)


def _capacity(ljmd, box, rc):
    return ljmd.footprint(N, box, rc, 0.3)["list_words"] // (-(-N // 32) * 32)


def _same(a, b):
    assert len(a) == len(b)
    for p, q in zip(a, b):
        np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("box,rc,rho,longest", [(24.0, 2.5, 0.9, (70, 104)), (21.0, 3.9, 1.55, (449, 600))])
def test_grown_within_spare_words(ljmd, precision, box, rc, rho, longest):
    x, v = _block(rho, box), li.maxwell_boltzmann(N, 0.5, 12)
    f = ljmd.footprint(N, box, rc, 0.3)
    out = []
    for graph in (0, 1):
        with ljmd.LJBatch(arena=dict(slots=f["slots"], cells=f["cells"], list_words=40 * f["list_words"], max_systems=4),
                          precision=precision) as b:
            b.set_tuning(graph=graph)
            k = b.add(N, box, rc, 0.3)
            g = li.fcc_positions(N, box)
            b.set_state(k, g, v)
            b.step(3, 0.0005)  # the plan for the first capacity
            b.set_state(k, x, v)
            for steps in (6, 1, 5):
                b.step(steps, 0.0005)
            out.append([*b.get_state(k), b.forces(k), np.array(list(b.stats(k).values()))])
    _same(*out)
    with ljmd.LJSystem(box, N, rc, 0.3, precision) as s:
        s.set_state(x, v)
        most = np.diff(s.get_list()[0]).max()
    assert _capacity(ljmd, box, rc) < longest[0] <= most <= longest[1]


@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_grown_twice(ljmd, precision, nvt):
    box = (N / 0.258) ** (1.0 / 3.0)
    first, second = _block(0.75, box), _block(1.22, box)
    v = li.maxwell_boltzmann(N, 0.5, 12)
    most, out = [], []
    for graph in (0, 1):
        with ljmd.LJSystem(box, N, 2.5, 0.3, precision) as s:
            s.set_tuning(graph=graph)
            ze = []
            for x in (first, second):
                s.set_state(x, v)
                if graph == 0:
                    most.append(np.diff(s.get_list()[0]).max())
                    s.set_state(x, v)
                ze += s.step_nvt(8, 0.002, 0.5, 3.0 * N * 0.05) if nvt else [s.step(8, 0.002)]
                s.step(4, 0.002)
            out.append([*s.get_state(), s.forces(), np.array(ze if nvt else [0.0])])
    _same(*out)
    # both lists outgrow the capacity before them, the second within the words that the
    # first growth left
    cap = _capacity(ljmd, box, 2.5)
    grown = [(int(m * 1.25) + 16 + 7) // 8 * 8 for m in most]
    assert most[0] > cap and grown[0] < most[1] and grown[1] <= cap + grown[0]


@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_grown_in_the_middle_of_a_call(ljmd, precision, nvt):
    box = 22.0
    x = _block(0.4, box, 0.02)
    v = -1.5 * (x - 0.5 * box) + li.maxwell_boltzmann(N, 0.01, 13)
    cap = _capacity(ljmd, box, 2.5)
    out = []
    for graph in (0, 1):
        with ljmd.LJSystem(box, N, 2.5, 0.3, precision) as s:
            s.set_tuning(graph=graph)
            s.set_state(x, v)
            assert np.diff(s.get_list()[0]).max() <= cap
            s.set_state(x, v)
            ze = s.step_nvt(60, 0.004, 1.0, 3.0 * N) if nvt else s.step(60, 0.004)
            out.append([*s.get_state(), s.forces(), np.array(ze if nvt else [0.0]), np.array(list(s.stats().values()))])
            assert np.diff(s.get_list()[0]).max() > cap
    _same(*out)

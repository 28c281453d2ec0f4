"""A grid barrier of the persistent step loop that gives up (its limit set to a few polls):
the call returns MD_ERR_TIMEOUT, the system has no state, and after a new one the handle
runs as a new one bit for bit."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu


def _state_lost(ljmd, s):
    for call in (s.get_state, s.forces, lambda: s.step(1, 0.005), s.checkpoint):
        with pytest.raises(ljmd.MDError) as e:
            call()
        assert e.value.code == ljmd.MD_ERR_STATE


@pytest.mark.parametrize("polls", [0, 1, 4])
@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_state_is_lost_and_can_be_set_again(ljmd, precision, nvt, polls):
    n = 4000
    x, box = li.perturbed_fcc(n, 0.8442, 0.1, 21)
    v = li.maxwell_boltzmann(n, 0.9, 22)

    def run(s, steps):
        if nvt:
            return s.step_nvt(steps, 0.005, 0.9, 3.0 * n * 0.05)
        return s.step(steps, 0.005)

    with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
        s.set_state(x, v)
        run(s, 25)
        ref = (*s.get_state(), s.forces())
    with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
        for steps in (0, 3):  # at the first lists, and with lists in use
            s.debug_loop_polls(1 << 21)
            s.set_state(x, v)
            run(s, steps)
            s.debug_loop_polls(polls)
            with pytest.raises(ljmd.MDError) as e:
                run(s, 500)
            assert e.value.code == ljmd.MD_ERR_TIMEOUT
            _state_lost(ljmd, s)
        s.debug_loop_polls(1 << 21)
        s.set_state(x, v)
        run(s, 25)
        for p, q in zip(ref, (*s.get_state(), s.forces())):
            np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("nvt", [False, True], ids=["nve", "nvt"])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_refused_launch(ljmd, precision, nvt):
    """A refused launch: the call takes its steps as without the loop, and so does the next."""
    n = 2000
    x, box = li.perturbed_fcc(n, 0.8442, 0.1, 23)
    v = li.maxwell_boltzmann(n, 0.9, 24)
    out = []
    for polls in (1 << 21, -1):
        with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
            s.debug_loop_polls(polls)
            s.set_state(x, v)
            ze = []
            for steps in (11, 1, 4):
                ze += s.step_nvt(steps, 0.005, 0.9, 3.0 * n * 0.05) if nvt else [s.step(steps, 0.005)]
            out.append((*s.get_state(), s.forces(), np.array(ze if nvt else [0.0]), np.array(list(s.stats().values()))))
    for p, q in zip(*out):
        np.testing.assert_array_equal(p, q)


def test_limit_is_checked(ljmd):
    with ljmd.LJSystem(20.0, 100, 2.5, 0.3) as s:
        for bad in (-2, 1 << 31):
            with pytest.raises(ljmd.MDError) as e:
                s.debug_loop_polls(bad)
            assert e.value.code == ljmd.MD_ERR_ARG

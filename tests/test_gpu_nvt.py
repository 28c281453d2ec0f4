"""Nose-Hoover NVT (md_step_nvt) against the oracle's NVT integrator: positions
within 1e-9, velocities within 1e-8, thermostat variables within 1e-9 after 100
steps (only the order of the kinetic-energy sums differs), in a batch each system
equal to its run alone."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu


def test_nvt_matches_oracle(ljmd, oracle):
    x, box = li.perturbed_fcc(864, 0.70, 0.05, 801)
    v = li.maxwell_boltzmann(864, 1.3, 802)
    q = 0.5 * 3 * 863 * 0.9 * 0.25
    with ljmd.LJSystem(box, 864, 3.0, 0.3) as s:
        s.set_state(x, v)
        z, e = s.step_nvt(100, 0.005, 0.9, q, 0.0, 0.0)
        xg, vg = s.get_state()
    r = oracle.run_nvt(x, v, box, 3.0, 0.3, 100, 0.005, 0.9, q)
    d = xg - r["x"]
    d -= box * np.round(d / box)
    assert np.abs(d).max() < 1e-9
    assert np.abs(vg - r["v"]).max() < 1e-8
    assert abs(z - r["zeta"]) < 1e-9 and abs(e - r["eta"]) < 1e-9


def test_nvt_batch_equals_alone(ljmd):
    syss = li.batch_systems(count=4, seed=803)
    dt = [c.dt for c in syss]
    T = [0.9] * 4
    Q = [0.5 * 3 * (c.n - 1) * 0.9 * 0.25 for c in syss]
    import ctypes as C
    with ljmd.LJBatch(systems=[(c.n, c.box, c.rc, c.skin) for c in syss]) as b:
        for k, c in enumerate(syss):
            b.set_state(k, c.x, c.v)
        z = np.zeros(4)
        e = np.zeros(4)
        arr = lambda a: np.ascontiguousarray(a, dtype=np.float64)
        dts, Ts, Qs = arr(dt), arr(T), arr(Q)
        lib = ljmd.load_library()
        pd = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
        rc = lib.md_batch_step_nvt(b._h, 40, pd(dts), pd(Ts), pd(Qs), pd(z), pd(e))
        assert rc == 0, lib.md_last_error()
        for k, c in enumerate(syss):
            xb, vb = b.get_state(k)
            with ljmd.LJSystem(c.box, c.n, c.rc, c.skin) as s:
                s.set_state(c.x, c.v)
                zk, ek = s.step_nvt(40, c.dt, 0.9, Q[k])
                xs, vs = s.get_state()
            np.testing.assert_array_equal(xb, xs)
            np.testing.assert_array_equal(vb, vs)
            assert z[k] == zk and e[k] == ek


def test_thermostat_after_an_error(ljmd):
    """A step that ends with MD_ERR_NONFINITE gives back the thermostat that the velocities
    have moved with: the opening half step, with and without the loop."""
    import ctypes as C
    n, dt, T, Q, z0, e0 = 500, 0.005, 0.9, 70.0, 0.25, -1.0
    x, box = li.perturbed_fcc(n, 0.8, 0.05, 805)
    x[7, 1] = np.nan
    v = li.maxwell_boltzmann(n, 1.3, 806)
    ke = 0.5 * (v * v).sum()
    gT = 3.0 * (n - 1) * T
    zeta = z0 + 0.25 * dt * (2.0 * ke - gT) / Q
    eta = e0 + 0.5 * dt * zeta
    zeta += 0.25 * dt * (2.0 * ke * np.exp(-dt * zeta) - gT) / Q
    for graph in (0, 1):
        with ljmd.LJSystem(box, n, 2.5, 0.3) as s:
            s.set_tuning(graph=graph)
            s.set_state(x, v)
            z, e = C.c_double(z0), C.c_double(e0)
            rc = ljmd.load_library().md_step_nvt(s._h, 50, dt, T, Q, C.byref(z), C.byref(e))
            assert rc == ljmd.MD_ERR_NONFINITE
            assert b"non-finite" in ljmd.load_library().md_last_error()
            assert abs(z.value - zeta) < 1e-12 and abs(e.value - eta) < 1e-12


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("speed", [1e-12, 1e-9, 1e-6, 1e-3, 1.0, 1e4, 1e9])
def test_kinetic_energy_at_any_scale(ljmd, speed, precision, graph):
    """Particles out of each other's reach: the thermostat variables after one step are
    those of the kinetic energy alone, whatever its scale. Their FP64 chain of a few
    operations and the sum of 375 squares leave a relative 1e-13."""
    n, box = 125, 60.0
    k = np.arange(n)
    x = np.stack([k % 5, k // 5 % 5, k // 25], 1) * 12.0 + 1.0
    v = speed * li.maxwell_boltzmann(n, 1.0, 807)
    dt, Q = min(0.005, 1e-3 / speed), n * speed ** 2 * 0.01
    ke, zeta, eta = 0.5 * (v * v).sum(), 0.0, 0.0
    for _ in range(2):
        zeta += 0.25 * dt * 2.0 * ke / Q
        eta += 0.5 * dt * zeta
        ke *= np.exp(-0.5 * dt * zeta) ** 2
        zeta += 0.25 * dt * 2.0 * ke / Q
    with ljmd.LJSystem(box, n, 2.5, 0.3, precision) as s:
        s.set_tuning(graph=graph)
        s.set_state(x, v)
        z, e = s.step_nvt(1, dt, 0.0, Q)
        vs = s.get_state()[1]
    assert abs(z - zeta) <= 1e-13 * zeta and abs(e - eta) <= 1e-13 * eta
    assert abs(0.5 * (vs * vs).sum() - ke) <= 1e-13 * ke

"""The FP64 form's positions in pair units share the memory of the half list's force sums
and of the rebuild's velocities: the form takes no memory beyond an arena's capacities,
a paused system keeps its positions there, and half lists start from zero sums."""
import numpy as np
import pytest

import lj_inputs as li

pytestmark = pytest.mark.gpu


def _used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_memory_of_a_server(ljmd, precision):
    """A server's arena in use stays within its budget (and 32 MB for the handle itself),
    whatever the form."""
    from paper_1210_3450_gb300 import serve

    def use(budget):
        before = _used()
        s = serve.MDServer(budget, precision=precision, max_systems=64)
        for k in range(3):
            s.submit(serve.Request(id=k, arrival=0.0, n=2000 + k, rho=0.8, temperature=1.0, steps=30, seed=k))
        s.admit(0.0)
        while s.running:
            s.step_chunk()
        used = _used() - before
        s.close()
        return used

    use(1 << 28)  # kernels and graphs loaded
    assert use(3 << 30) <= (3 << 30) + (32 << 20)


@pytest.mark.parametrize("graph", [0, 1])
def test_paused_between_rebuilds(ljmd, graph):
    """A system paused after an odd number of steps while the others rebuild, in an arena
    of graph launches: each system as it runs alone, bit for bit."""
    sizes = [(40000, 0.8), (1500, 0.7), (700, 0.85)]
    syss = []
    for k, (n, rho) in enumerate(sizes):
        x, box = li.perturbed_fcc(n, rho, 0.1, 60 + k)
        syss.append((n, box, x, li.maxwell_boltzmann(n, 1.0, 70 + k)))
    with ljmd.LJBatch(systems=[(n, box, 2.5, 0.3) for n, box, _, _ in syss]) as b:
        b.set_tuning(graph=graph)
        for k, (_, _, x, v) in enumerate(syss):
            b.set_state(k, x, v)
        b.step(9, 0.005)
        b.set_active(1, False)
        b.step(20, 0.005)
        b.set_active(1, True)
        b.set_active(2, False)
        b.step(1, 0.005)
        b.set_active(2, True)
        b.step(10, 0.005)
        got = [(*b.get_state(k), b.forces(k)) for k in range(3)]
        obs = b.observables()
    for k, (n, box, x, v) in enumerate(syss):
        with ljmd.LJSystem(box, n, 2.5, 0.3) as s:
            s.set_tuning(graph=graph)
            s.set_state(x, v)
            s.step((40, 20, 39)[k], 0.005)
            alone = (*s.get_state(), s.forces())
            o = s.observables()
        for p, q in zip(got[k], alone):
            np.testing.assert_array_equal(p, q)
        assert obs[k, 0] == o["pe"] and obs[k, 1] == o["virial"]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
def test_half_lists_after_full_ones(ljmd, oracle, precision):
    from paper_1210_3450_gb300.ljmd import MD_LIST_HALF
    x, box = li.perturbed_fcc(2001, 0.8442, 0.1, 81)
    v = li.maxwell_boltzmann(2001, 0.9, 82)
    ref = oracle.forces(x, box, 2.5)
    rms = np.sqrt((ref ** 2).sum(1).mean())
    with ljmd.LJSystem(box, 2001, 2.5, 0.3) as s:
        s.set_state(x, v)
        s.step(3, 0.005)
        s.set_precision(precision)
        s.set_pair_list(MD_LIST_HALF)
        s.set_state(x, v)
        assert np.abs(s.forces() - ref).max() <= (1e-12 if precision == 0 else 1e-5) * rms

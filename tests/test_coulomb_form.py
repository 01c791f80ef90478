"""The Coulomb pass takes small cells in groups, a warp each, and large ones a
block each.  Which form runs follows the particles that the cells hold, not the
capacity a handle was made with; both give the same bits."""
import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _sim(n_op, n_cells=256, **kw):
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(**dict(dict(n_op=n_op, n_cells=n_cells, fp64=False, n2=10, weight_override=1e6), **kw))
    return o2pic.Simulation([d], inputs.xs_tables())


def _pass_us(sim):
    best = 1e9
    for _ in range(5):
        sim.set_timing(True)
        sim.step(20)
        k = sim.kernel_timing("coulomb", reset=True)
        sim.set_timing(False)
        best = min(best, 1e3 * k["ms"] / k["launches"])
    return best


@pytest.mark.parametrize("per_cell", [100, 3000])
def test_the_pass_takes_the_same_time_whatever_the_capacity(per_cell):
    n_op = per_cell * 512
    times = []
    for capacity in (1.5, 40.0 if per_cell < 1000 else 6.0):
        sim = _sim(n_op, n_cells=512, capacity_factor=capacity)
        sim.step(20)
        times.append(_pass_us(sim))
        sim.close()
    assert max(times) <= 1.3 * min(times), times


def test_both_forms_give_the_same_bits():
    rng = np.random.default_rng(7)
    n, L = 580 * 256, 0.025  # between the lines of the two directions
    state = [(rng.uniform(0.0, L, n), *(v * rng.standard_normal((3, n)))) for v in (1e6, 600.0, 400.0)]
    states = []
    for n_op in (256 * 100, 256 * 2000):  # comes from few particles per cell, from many
        sim = _sim(n_op, capacity_factor=1.0, capacity_extra=2 * n)
        sim.step(20)
        for s in range(3):
            sim.set_state(0, s, *state[s])
        sim.set_step(20)
        sim.step(20)
        states.append([sim.get_state(0, s) for s in range(3)])
        assert sim.diagnostics(0)["coulomb_particles"] > 0
        sim.close()
    for s in range(3):
        for key in ("x", "vx", "vy", "vz", "alive"):
            assert np.array_equal(states[0][s][key], states[1][s][key]), (s, key)

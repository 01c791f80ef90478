"""A birth beyond the capacity is dropped with its charge: after a reported
overflow the density sums and the fields are those of the particles that
pic_get_state returns, step by step and inside a captured stretch.

Both node weights of a particle add up to exactly one, so the density summed
over the nodes counts the particles: exact in the FP32 path (integers), to
rounding in the FP64 path (a dropped birth is a whole particle)."""
import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

QE = 1.602176634e-19
STEPS = 60
SIZES = {
    "one block": [dict(n_op=20000)],
    "cluster": [dict(n_op=20000, n_cells=1500), dict(n_op=20001, capacity_factor=2.0), dict(n_op=5000, n_cells=9)],
    "several append blocks": [dict(n_op=150000, n_cells=300)],
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _sim(sizes, fp64, numeric_budget=None, **kw):
    from paper_0705_0495_gb300 import o2pic
    base = dict(fp64=fp64, U_rf=300.0, T0_eV=(8.0, inputs.T_ION_EV, inputs.T_ION_EV), capacity_factor=1.0,
                capacity_extra=0, **kw)
    ds = [inputs.cfg1(**dict(base, seed=3 + k, **q)) for k, q in enumerate(sizes)]
    return o2pic.Simulation(ds, inputs.xs_tables(), numeric_budget=numeric_budget), ds


def _step(sim, n):
    """True when the call reported an overflow"""
    from paper_0705_0495_gb300 import o2pic
    try:
        sim.step(n)
    except o2pic.PicError as e:
        assert "CAPACITY" in str(e)
        return True
    return False


def _volumes(d):
    v = np.full(d.n_cells + 1, d.L / d.n_cells)
    v[[0, -1]] *= 0.5
    return v


def _live(sim, k):
    return np.array([int(sim.get_state(k, s)["alive"].sum()) for s in range(3)])


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("scheme", [0, 1])
def test_fields_after_an_overflow_hold_the_particles_only(sizes, fp64, scheme):
    sim, ds = _sim(SIZES[sizes], fp64, numeric_budget=1.0, gas_scheme=scheme)
    over = False
    for _ in range(STEPS):
        over |= _step(sim, 1)
        for k, d in enumerate(ds):
            n = _live(sim, k)
            net = float((sim.fields(k)[0] * _volumes(d)).sum() / (QE * d.weight))
            assert abs(net - (n[2] - n[0] - n[1])) < 1e-6, (k, net, n)
    assert over
    sim.close()


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("sub", [1, 2])
def test_a_stretch_with_overflows_samples_the_particles_only(sizes, fp64, sub):
    a, ds = _sim(SIZES[sizes], fp64, diag_every=sub, ion_subcycle=sub)
    b, _ = _sim(SIZES[sizes], fp64, diag_every=sub, ion_subcycle=sub)
    assert _step(a, STEPS)  # graphs of one period
    assert a.diagnostics(0)["graph_launch_calls"] == STEPS // 10
    want = np.zeros((len(ds), 3))
    for n in range(STEPS):
        if n % sub == 0:
            for k in range(len(ds)):
                want[k] += _live(b, k)
        _step(b, 1)
    assert b.diagnostics(0)["graph_launch_calls"] == 0
    for k, d in enumerate(ds):
        for sim in (a, b):
            g = sim.diagnostics(k)
            assert g["n_samples"] == STEPS // sub
            got = (g["dens_sum"] * _volumes(d)).sum(axis=1) / d.weight
            assert np.all(np.abs(got - want[k]) < 1e-6 * STEPS), (k, got, want[k])
        if fp64:
            continue
        for s in range(3):
            sa, sb = a.get_state(k, s), b.get_state(k, s)
            for key in ("x", "vx", "vy", "vz", "alive"):
                assert np.array_equal(sa[key], sb[key]), (k, s, key)
    a.close()
    b.close()

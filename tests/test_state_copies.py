"""State copies through the spare particle buffer: what goes in comes out,
over chunk borders (one species holding nearly all slots), with dead slots,
positions next to the walls, skipped arrays, and with a refused state leaving
the old one in place; and the charge that a replaced state deposits."""
import ctypes as C

import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
QE = 1.602176634e-19


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _state(d, n, rng):
    N, dx = d.n_cells, d.L / d.n_cells
    x = rng.uniform(0.0, d.L, n)
    x[:6] = [0.0, np.nextafter(d.L, 0.0), dx, np.nextafter(dx, 0.0), (N - 1) * dx, np.nextafter(2 * dx, 0.0)]
    v = [rng.normal(0.0, 1e4, n) for _ in range(3)]
    alive = rng.random(n) < 0.9
    alive[:6] = True
    return x, v, alive


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n_op,factor", [(4001, 1.0), (50, 1500.0)])
def test_state_goes_in_and_comes_out(fp64, n_op, factor):
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_op=n_op, n_cells=37, fp64=fp64, capacity_factor=factor, capacity_extra=0)
    sim = o2pic.Simulation([inputs.cfg1(n_op=100, fp64=fp64), d], inputs.xs_tables())
    rng = np.random.default_rng(3)
    dx, vs = d.L / d.n_cells, d.L / d.n_cells / d.dt
    kept = []
    for s in range(3):
        n = d.capacity[s] - (s == 1)
        x, v, alive = _state(d, n, rng)
        sim.set_state(1, s, x, *v, alive)
        g = sim.get_state(1, s)
        assert np.array_equal(g["alive"], alive)
        real = np.float64 if fp64 else np.float32
        xx = x / dx
        c = np.minimum(np.floor(xx), d.n_cells - 1)
        off = (xx - c).astype(real)
        up = off >= 1
        if not fp64:
            c = np.where(up & (c + 1 < d.n_cells), c + 1, c)
            off = np.where(up, np.where(xx < d.n_cells - 1, real(0), np.nextafter(real(1), real(0))), off)
        want = np.where(alive, (c + off.astype(np.float64)) * dx, 0.0)
        assert np.array_equal(g["x"], want)
        for key, a in zip(("vx", "vy", "vz"), v):
            assert np.array_equal(g[key], (a * (d.dt / dx)).astype(real).astype(np.float64) * vs), key
        kept.append((want[alive], alive.sum()))
    # the charge of the new state: total charge of the nodes
    rho, _, _ = sim.fields(1)
    vol = np.full(d.n_cells + 1, dx)
    vol[[0, -1]] = 0.5 * dx
    total = QE * d.weight * (kept[2][1] - kept[0][1] - kept[1][1])
    assert abs(np.sum(rho * vol) - total) <= 1e-9 * QE * d.weight * sum(k[1] for k in kept)
    sim.close()


@pytest.mark.parametrize("bad", [-1e-9, 0.025, np.nan, np.inf])
def test_a_refused_state_changes_nothing(bad):
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_op=5000, fp64=False)
    sim = o2pic.Simulation([d], inputs.xs_tables())
    old, f_old = sim.get_state(0, 2), sim.fields(0)
    x = np.full(4000, 0.01)
    x[3777] = bad
    v = np.zeros(4000)
    with pytest.raises(o2pic.PicError) as e:
        sim.set_state(0, 2, x, v, v, v)
    assert e.value.code == 1
    new = sim.get_state(0, 2)
    assert all(np.array_equal(old[k], new[k]) for k in old)
    assert all(np.array_equal(a, b) for a, b in zip(f_old, sim.fields(0)))
    alive = np.ones(4000, dtype=bool)
    alive[3777] = False  # dead: its position does not matter
    sim.set_state(0, 2, x, v, v, v, alive)
    assert sim.count(0, 2) == 4000
    sim.close()


def test_skipped_state_arrays():
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_op=3000, fp64=False)
    sim = o2pic.Simulation([d], inputs.xs_tables())
    full = sim.get_state(0, 0)
    n = sim.count(0, 0)
    vy = np.zeros(n + 7)
    m = C.c_longlong()
    rc = sim.lib.pic_get_state(sim.h, 0, 0, None, None, vy.ctypes.data_as(C.POINTER(C.c_double)), None, None, n + 7,
                               C.byref(m))
    assert rc == 0 and m.value == n
    assert np.array_equal(vy[:n], full["vy"]) and not vy[n:].any()
    sim.close()

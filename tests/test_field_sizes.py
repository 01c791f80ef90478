"""The field solve at the edges of its work split: one block per discharge up
to 1024 cells, a cluster of blocks beyond; discharges of very different size
in one launch; and the push's tile table of many discharges.

Reference: rho, phi and E from the particles' positions in extended
precision.  The FP32 path rounds each particle's weight to 2^-24, an error of
at most 2^-25 of a particle per node: that gives the bounds below (plus 1e-10
of the largest value for the FP64 arithmetic, as in the other field tests)."""
import math

import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

QE, EPS0 = 1.602176634e-19, 8.8541878128e-12


def _reference(d, states, step):
    N, dx = d.n_cells, d.L / d.n_cells
    q = np.zeros(N + 1, dtype=np.longdouble)
    per_node = np.zeros(N + 1)
    for sign, st in zip((-1, -1, 1), states):
        x = st["x"][st["alive"]].astype(np.longdouble) / dx
        c = np.minimum(np.floor(x).astype(np.int64), N - 1)
        o = x - c
        np.add.at(q, c, sign * (1 - o))
        np.add.at(q, c + 1, sign * o)
        np.add.at(per_node, c, 1.0)
        np.add.at(per_node, c + 1, 1.0)
    vol = np.full(N + 1, dx)
    vol[[0, N]] = 0.5 * dx
    rho = QE * d.weight * q / vol
    phi0 = d.U_rf * math.sin(2 * math.pi * d.f_rf * step * d.dt + d.rf_phase)
    s = rho[1:N] * dx * dx / EPS0
    s2 = np.cumsum(np.cumsum(s))
    slope = (s2[-1] - phi0) / N
    phi = np.zeros(N + 1, dtype=np.longdouble)
    phi[0] = phi0
    phi[1:N] = phi0 + np.arange(1, N) * slope
    phi[2:N] -= s2[:-1]
    E = np.empty(N + 1, dtype=np.longdouble)
    E[1:N] = -(phi[2:] - phi[:-2]) / (2 * dx)
    E[0] = -(phi[1] - phi[0]) / dx - rho[0] * dx / (2 * EPS0)
    E[N] = -(phi[N] - phi[N - 1]) / dx + rho[N] * dx / (2 * EPS0)
    return rho, phi, E, per_node, vol


@pytest.mark.gpu
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("cells", [(2,), (1023,), (1024, 3), (1025, 2, 300), (4096, 9)])
def test_fields_match_the_particles(cells, fp64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    ds = [inputs.cfg1(n_cells=N, n_op=6000 + 2 * k, seed=4 + k, fp64=fp64, rf_phase=0.3) for k, N in enumerate(cells)]
    sim = o2pic.Simulation(ds, inputs.xs_tables())
    sim.step(3)
    for k, d in enumerate(ds):
        rho, phi, E = sim.fields(k)
        states = [sim.get_state(k, s) for s in range(3)]
        r, p, e, per_node, vol = _reference(d, states, 3)
        w = 0.0 if fp64 else 2.0 ** -25
        K = QE * d.weight / EPS0
        total = per_node.sum()
        assert np.all(np.abs(rho - r) <= QE * d.weight / vol * w * per_node + 1e-10 * np.max(np.abs(r)))
        assert np.max(np.abs(E - e)) <= K * w * total + 1e-10 * np.max(np.abs(e))
        assert np.max(np.abs(phi - p)) <= K * w * total * d.L + 1e-10 * np.max(np.abs(p))
    sim.close()


@pytest.mark.gpu
def test_many_discharges_match_runs_of_a_few():
    """300 discharges (more than the tile table's threads), some empty: the
    slots and event counts of single-discharge handles cannot be compared (the
    random streams carry the discharge number), so the counts are checked
    against the states: every slot is visited once per step"""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    ds = [inputs.cfg1(n_op=(k * 37) % 2100, n_cells=8 + k % 40, seed=k, fp64=False, n1=0, sort_interval=0,
                      diag_every=0, numax_bins=4, capacity_extra=256) for k in range(300)]
    sim = o2pic.Simulation(ds, [])  # no collisions: nothing is born
    sim.step(5)
    for k, d in enumerate(ds):
        g = sim.diagnostics(k)
        n = sum(d.n_init)
        assert list(g["slots"]) == list(d.n_init)
        assert g["slots_visited"] == 5 * n
        alive = sum(int(sim.get_state(k, s)["alive"].sum()) for s in range(3))
        assert alive + int(g["absorbed"].sum()) == n
    sim.close()

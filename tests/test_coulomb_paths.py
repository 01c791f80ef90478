"""The Coulomb passes over their work splits, FP64 against the oracle slot by
slot: a warp or a block per cell inside a group of cells (up to and beyond the
682 particles a warp stages), and in the inter-species pass few chains on
prepared random numbers (several tiles of 1024 collisions, staged and in
place, chains of one) next to many chains.  Tolerance 1e-9 of the gap and of
the thermal speed, as in the other FP64 step-by-step tests."""
import math

import numpy as np
import pytest

import oracle
from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
QE, AMU, ME = 1.602176634e-19, 1.66053906660e-27, 9.1093837015e-31
MASS = (ME, 16 * AMU + ME, 32 * AMU - ME)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _compare(d, sim, orc, k=0):
    for s in range(3):
        g, o = sim.get_state(k, s), orc.get(s)
        assert np.array_equal(g["alive"], o["alive"]), s
        m = o["alive"]
        if not m.any():
            continue
        vt = math.sqrt(max(d.T0_eV[s], 0.0259) * QE / MASS[s])
        assert np.max(np.abs(g["x"][m] - o["x"][m])) < 1e-9 * d.L, s
        for c in ("vx", "vy", "vz"):
            assert np.max(np.abs(g[c][m] - o[c][m])) < 1e-9 * vt, (s, c)


@pytest.mark.parametrize("n_cells,n_op", [(7, 9000), (5, 6821), (33, 700), (2, 2731)])
def test_fp64_groups_of_cells(n_cells, n_op):
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_cells=n_cells, n_op=n_op, n2=1, coulomb_log=1e4, n1=0)
    tabs = inputs.xs_tables()
    sim, orc = o2pic.Simulation([d], tabs), oracle.Oracle(d, tabs)
    for _ in range(3):
        sim.step(2)
        orc.step(2)
        _compare(d, sim, orc)


@pytest.mark.parametrize("n_cells,n_op,keep", [(3, 9001, 0.02), (2, 40001, 0.004), (4, 5000, 0.0008), (3, 3000, 0.5)])
def test_fp64_few_chains(n_cells, n_op, keep):
    """most electrons removed: the ions of a cell queue up for the few left"""
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_cells=n_cells, n_op=n_op, n2=1, coulomb_log=1e4, coulomb_inter=True, n1=0)
    tabs = inputs.xs_tables()
    sim, orc = o2pic.Simulation([d], tabs), oracle.Oracle(d, tabs)
    st = orc.get(0)
    alive = np.random.default_rng(2).random(len(st["x"])) < keep
    alive[:2] = True
    sim.set_state(0, 0, st["x"], st["vx"], st["vy"], st["vz"], alive)
    orc.set(0, st["x"], st["vx"], st["vy"], st["vz"], alive)
    for _ in range(3):
        sim.step(1)
        orc.step(1)
        _compare(d, sim, orc)

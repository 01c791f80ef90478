"""The cell sort's rows: how many slots a warp takes follows the particle
number and the rows the workspace has.  CPU: the rows always suffice.  GPU:
batched discharges of very uneven size (one-slot and empty ones among them)
against their oracles, slot by slot, over steps with a sort each."""
import numpy as np
import pytest

import oracle
from paper_0705_0495_gb300 import inputs

ROWS, WARPS, MOST, LEAST, CHUNK = 1216, 4, 8192, 256, 1024


def _min_slots(N):
    w = LEAST
    while w < MOST and WARPS * w < N:
        w *= 2
    return w


def _warp_slots(n, gmax, N):
    w = _min_slots(N)
    while w < MOST and gmax * WARPS * w < n:
        w *= 2
    return w


def test_rows_cover_every_count_up_to_the_capacity():
    rng = np.random.default_rng(8)
    for _ in range(400):
        D = int(rng.integers(1, 40))
        caps = np.exp(rng.uniform(0, np.log(6e7 / D), size=3 * D)).astype(np.int64) + 1
        caps = (caps + CHUNK - 1) // CHUNK * CHUNK
        for cap in caps[:6]:
            N = int(rng.integers(2, 4097))
            fine = WARPS * _min_slots(N)
            gmax = max(-(-cap // (WARPS * MOST)), min(-(-cap // fine), ROWS * cap // caps.sum()))
            assert gmax >= 1
            for n in (0, 1, cap // 3, cap - 1, cap):
                w = _warp_slots(n, gmax, N)
                assert w & (w - 1) == 0 and w <= MOST
                assert -(-n // (WARPS * w)) <= gmax, (cap, N, n, w, gmax)


@pytest.mark.gpu
def test_fp64_sorted_slots_of_uneven_discharges_match_their_oracles():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    sizes = ((300_001, 16), (2, 300), (0, 64), (1023, 1500), (4097, 7))
    ds = [inputs.cfg1(n_op=n, n_cells=N, seed=5 + k, sort_interval=1) for k, (n, N) in enumerate(sizes)]
    tabs = inputs.xs_tables()
    sim = o2pic.Simulation(ds, tabs)
    sim.step(4)
    for k, d in enumerate(ds):
        orc = oracle.Oracle(d, tabs, discharge=k)
        orc.step(4)
        for s in range(3):
            g, o = sim.get_state(k, s), orc.get(s)
            assert np.array_equal(g["alive"], o["alive"]), (k, s)
            m = o["alive"]
            if m.any():
                assert np.max(np.abs(g["x"][m] - o["x"][m])) < 1e-9 * d.L
                for c in ("vx", "vy", "vz"):
                    assert np.max(np.abs(g[c][m] - o[c][m])) < 1e-9 * max(np.max(np.abs(o[c][m])), 1.0)
    sim.close()

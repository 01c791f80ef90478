"""Births and the next step's field in one launch (inside captured stretches)
against one launch each (single steps): the FP32 state, event counts,
histograms and density sums bit for bit, for handles whose discharges differ
much in size: clusters and single blocks for the field, an empty discharge,
one whose births span several append blocks."""
import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HOT = dict(T0_eV=(8.0, inputs.T_ION_EV, inputs.T_ION_EV), U_rf=300.0, fp64=False)


@pytest.mark.parametrize("diag_every", [1, 10])
@pytest.mark.parametrize("sub", [1, 2])
@pytest.mark.parametrize("sizes", [
    [(1500, 9000), (37, 0), (300, 150_000), (4096, 3001), (2, 500)],
    [(128, 0), (64, 4000), (1024, 150_001), (5, 70)],
])
def test_merged_launches_give_the_same_bits(sizes, sub, diag_every):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    diag_every = max(diag_every, sub)
    ds = [inputs.cfg1(n_cells=N, n_op=n, seed=5 + k, diag_every=diag_every, ion_subcycle=sub, **HOT)
          for k, (N, n) in enumerate(sizes)]
    a = o2pic.Simulation(ds, inputs.xs_tables())
    b = o2pic.Simulation(ds, inputs.xs_tables())
    a.step(30)
    assert a.diagnostics(0)["graph_launch_calls"] == 3
    for _ in range(30):
        b.step(1)
    assert b.diagnostics(0)["graph_launch_calls"] == 0
    ionisations = 0
    for k in range(len(ds)):
        ga, gb = a.diagnostics(k), b.diagnostics(k)
        for key in ("events", "absorbed", "eedf", "iedf", "fm", "dens_sum", "phi_sum", "slots", "slots_visited"):
            assert np.array_equal(ga[key], gb[key]), (k, key)
        for s in range(3):
            sa, sb = a.get_state(k, s), b.get_state(k, s)
            for key in ("x", "vx", "vy", "vz", "alive"):
                assert np.array_equal(sa[key], sb[key]), (k, s, key)
        for fa, fb in zip(a.fields(k), b.fields(k)):
            assert np.array_equal(fa, fb), k
        ionisations += int(ga["events"][18])
    assert ionisations > 100
    a.close()
    b.close()

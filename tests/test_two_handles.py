"""Handles of different grid size live side by side: the limits that a handle
asks of the kernels (dynamic shared memory) hold for every other one, also
while two threads replace states."""
import threading

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


def _sim(n_cells, fp64, stream=None, **kw):
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_op=4000, n_cells=n_cells, fp64=fp64, **kw)
    return o2pic.Simulation([d], inputs.xs_tables(), stream=stream)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("kw", [dict(), dict(n2=10, coulomb_inter=True), dict(gas_scheme=1)])
def test_a_later_smaller_handle_leaves_a_larger_one_working(fp64, kw):
    large = _sim(4096, fp64, **kw)
    small = _sim(16, fp64, eedf_bins=0, iedf_bins=0, fm_bins=0, **kw)
    small.step(21)
    large.step(21)  # captured and single steps, with and without diagnostics
    st = large.get_state(0, 2)
    large.set_state(0, 2, st["x"], st["vx"], st["vy"], st["vz"], st["alive"])
    large.step(1)
    small.step(1)
    large.close()
    small.close()


@pytest.mark.parametrize("fp64", [False, True])
def test_two_threads_replace_states_of_different_grids(fp64):
    sims = [_sim(n, fp64, stream=torch.cuda.Stream()) for n in (4096, 16)]
    states = [s.get_state(0, 2) for s in sims]
    fields = [s.fields(0)[0] for s in sims]
    bad = []

    def work(k):
        st = states[k]
        try:
            for _ in range(300):
                sims[k].set_state(0, 2, st["x"], st["vx"], st["vy"], st["vz"], st["alive"])
        except Exception as e:
            bad.append((k, str(e)))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
    for k, s in enumerate(sims):
        assert np.max(np.abs(s.fields(0)[0] - fields[k])) <= 1e-10 * np.max(np.abs(fields[k]))
        s.close()

"""What the host reads between steps comes through one gather: a window's
reset clears what it returned and nothing of another discharge, skipped arrays
stay untouched, and two threads may read one handle."""
import ctypes as C
import threading

import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SUMS = ("dens_sum", "phi_sum", "eedf", "iedf", "fm")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _sim(fp64):
    from paper_0705_0495_gb300 import o2pic
    ds = [inputs.cfg1(n_op=6000, n_cells=5, fp64=fp64, eedf_bins=7, iedf_bins=3, fm_bins=5, fm_xbins=3),
          inputs.cfg1(n_op=3001, n_cells=400, fp64=fp64, eedf_bins=0, iedf_bins=0, fm_bins=0),
          inputs.cfg1(n_op=9000, n_cells=1500, fp64=fp64, U_rf=300.0)]
    sim = o2pic.Simulation(ds, inputs.xs_tables())
    sim.step(40)
    return sim


@pytest.mark.parametrize("fp64", [False, True])
def test_reset_clears_one_window_only(fp64):
    sim = _sim(fp64)
    before = [sim.diagnostics(k) for k in range(3)]
    got = sim.diagnostics(1, reset=True)
    for k in SUMS:
        assert np.array_equal(got[k], before[1][k]), k
    for k in (0, 2):
        again = sim.diagnostics(k)
        for key in SUMS:
            assert np.array_equal(again[key], before[k][key]), (k, key)
    empty = sim.diagnostics(1)
    assert empty["n_samples"] == 0 and all(not empty[k].any() for k in SUMS)
    assert np.array_equal(empty["events"], got["events"]) and empty["steps"] == 40
    assert sim.diagnostics(0, reset=True)["n_samples"] == 4 and sim.diagnostics(0)["n_samples"] == 0
    sim.close()


def test_skipped_arrays_are_left_alone():
    sim = _sim(False)
    phi = np.full(1501, 7.0)
    n = C.c_longlong(-1)
    rc = sim.lib.pic_diagnostics(sim.h, 2, None, phi.ctypes.data_as(C.POINTER(C.c_double)), None, None, None, None,
                                 C.byref(n), 0)
    assert rc == 0 and n.value == 4
    assert np.array_equal(phi, sim.diagnostics(2)["phi_sum"])
    sim.close()


def test_two_threads_read_one_handle():
    sim = _sim(False)
    want = [sim.diagnostics(k) for k in range(3)]
    fields = [sim.fields(k) for k in range(3)]
    bad = []

    def reader(first):
        for r in range(20):
            k = (first + r) % 3
            g, f = sim.diagnostics(k), sim.fields(k)
            if not all(np.array_equal(g[key], want[k][key]) for key in SUMS) or \
                    not all(np.array_equal(a, b) for a, b in zip(f, fields[k])):
                bad.append(k)

    ts = [threading.Thread(target=reader, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
    sim.close()

"""pic_set_launch takes one and two blocks per SM of the FP64 push, with the
same results; the counts that pic_get_launch and pic_launch_shapes give are
those that are accepted."""
import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_the_fp64_push_takes_two_blocks_per_sm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    d = inputs.cfg1(n_op=400_000, n_cells=500, fp64=True)
    sims = [o2pic.Simulation([d], inputs.xs_tables()) for _ in range(2)]
    sims[1].set_launch(2)
    assert sims[1].launch() == (2, 2)
    assert sims[1].launch_shapes()[0][2] == 2
    sims[1].set_launch_shape(0, 2)
    for bad in (0, 3):
        with pytest.raises(o2pic.PicError):
            sims[1].set_launch(bad)
    for s in sims:
        s.step(20)
    for s in range(3):
        a, b = (x.get_state(0, s) for x in sims)
        assert np.array_equal(a["alive"], b["alive"])
        for key in ("x", "vx", "vy", "vz"):
            assert np.max(np.abs(a[key] - b[key])) <= 1e-9 * np.max(np.abs(a[key])), (s, key)
    for s in sims:
        s.close()

"""pic_field_solve_static in FP64 on sparse states, where a node holds a few small
weights: rho of every node to FP64 rounding of its own value.

An offset from 2^-11 on enters exactly, the sums are integers; what is rounded
is the node's charge as a double, the factor e weight / dx (twice) and their
product: four roundings, at most 4.5 units of 2^-53 with the reference's own.
Smaller offsets are rounded at 2^-64 of a particle."""
import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
QE = 1.602176634e-19


@pytest.mark.parametrize("n_cells,n,low", [(4096, 1500, -11), (4095, 9, -11), (64, 20, -11), (2, 1, -11), (4096, 3000, -40)])
def test_rho_of_sparse_nodes(n_cells, n, low):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0705_0495_gb300 import o2pic
    rng = np.random.default_rng(n_cells + n)
    d = inputs.cfg1(n_cells=n_cells, fp64=True)
    dx = d.L / n_cells
    cells = [rng.integers(0, n_cells, n + s).astype(np.int32) for s in range(3)]
    offs = [2.0 ** rng.uniform(low, 0.0, n + s) for s in range(3)]
    vol = np.full(n_cells + 1, dx)
    vol[[0, -1]] *= 0.5
    q = np.zeros(n_cells + 1, dtype=np.longdouble)
    count = np.zeros(n_cells + 1)
    for sign, c, o in zip((-1, -1, 1), cells, offs):
        o = o.astype(np.longdouble)
        np.add.at(q, c, sign * (1 - o))
        np.add.at(q, c + 1, sign * o)
        np.add.at(count, c, 1.0)
        np.add.at(count, c + 1, 1.0)
    want = np.longdouble(QE) * np.longdouble(d.weight) * q / vol
    out = [torch.zeros(n_cells + 1, dtype=torch.float64, device="cuda") for _ in range(3)]
    dev = [torch.from_numpy(a).cuda() for a in cells + offs]
    o2pic.field_solve_static(o2pic.make_config(d), 0, [t.data_ptr() for t in dev[:3]], [t.data_ptr() for t in dev[3:]],
                             [n, n + 1, n + 2], *(t.data_ptr() for t in out), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    got = out[0].cpu().numpy()
    bound = 4.5 * 2.0 ** -53 * np.abs(want) + QE * d.weight / vol * count * 2.0 ** -64
    assert np.all(np.abs(got - want) <= bound), float(np.max(np.abs(got - want) / bound))

"""pic_field_solve_static over its work splits: one launch for few particles,
deposit and solve apart for many; one block or a cluster for the solve;
aligned and unaligned arrays; empty species, slots off the grid, offsets
outside [0, 1] and NaN.

FP32: the charge is an exact integer of 2^-24 of a particle, so rho must agree
with the integer reference to FP64 rounding (1e-14); FP64: the weights are
rounded to 2^-53 of a particle and a node's sum to 2^-53 of its size, a few
times (1e-15 of the node's particle count).  phi and E: FP64 rounding of a few
operations on sums of that size (1e-12 of the largest value, as the double sums
of the reference alone would give)."""
import math

import numpy as np
import pytest

from paper_0705_0495_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
QE, EPS0 = 1.602176634e-19, 8.8541878128e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _particles(N, counts, fp64, ordered, rng):
    cells, offs = [], []
    for n in counts:
        x = rng.uniform(-0.5, N + 0.5, n)
        if ordered:
            x = np.sort(x)
        c = np.floor(x).astype(np.int32)   # some off the grid, at both ends
        o = (x - c).astype(np.float64 if fp64 else np.float32)
        odd = rng.integers(0, 200, n)
        o[odd == 0] = -0.25
        o[odd == 1] = 1.5
        o[odd == 2] = np.nan
        o[odd == 3] = 1.0
        cells.append(c)
        offs.append(o)
    return cells, offs


def _reference(d, cells, offs, step):
    """node charge as exact integers (FP32: units of 2^-24) or extended sums"""
    N, dx = d.n_cells, d.L / d.n_cells
    q = np.zeros(N + 1, dtype=np.longdouble)
    count = np.zeros(N + 1)
    for sign, c, o in zip((-1, -1, 1), cells, offs):
        live = (c >= 0) & (c < N)
        c, o = c[live], np.clip(np.nan_to_num(o[live], nan=0.0), 0.0, 1.0)
        if o.dtype == np.float32:
            w1 = np.rint(o.astype(np.float64) * 2.0 ** 24) / 2.0 ** 24
        else:
            w1 = o.astype(np.longdouble)
        np.add.at(q, c, sign * (1 - w1.astype(np.longdouble)))
        np.add.at(q, c + 1, sign * w1.astype(np.longdouble))
        np.add.at(count, c, 1.0)
        np.add.at(count, c + 1, 1.0)
    vol = np.full(N + 1, dx)
    vol[[0, N]] = 0.5 * dx
    rho = QE * d.weight * q / vol
    phi0 = d.U_rf * math.sin(2 * math.pi * d.f_rf * step * d.dt + d.rf_phase)
    s2 = np.cumsum(np.cumsum(rho[1:N] * dx * dx / EPS0))
    slope = (s2[-1] - phi0) / N
    phi = np.zeros(N + 1, dtype=np.longdouble)
    phi[0] = phi0
    phi[1:N] = phi0 + np.arange(1, N) * slope
    phi[2:N] -= s2[:-1]
    E = np.empty(N + 1, dtype=np.longdouble)
    E[1:N] = -(phi[2:] - phi[:-2]) / (2 * dx)
    E[0] = -(phi[1] - phi[0]) / dx - rho[0] * dx / (2 * EPS0)
    E[N] = -(phi[N] - phi[N - 1]) / dx + rho[N] * dx / (2 * EPS0)
    return rho, phi, E, QE * d.weight / vol * count


SMALL = (1 << 17) - 3 * 128 * 8  # slots of the largest call that is one launch
CASES = [(2, (5, 0, 3)), (7, (0, 0, 0)), (128, (10_001, 9_999, 20_000)), (4096, (1, 2049, 40_000)),
         (300, (SMALL - 70_000, 30_000, 40_000)), (300, (SMALL - 70_000, 30_000, 40_001)),
         (1024, (200_003, 0, 77)), (1025, (100_000, 130_001, 250_007)), (4096, (600_001, 600_002, 1_200_003)),
         (16, (2_000_000, 0, 1_000_000))]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("N,counts", CASES)
def test_static_solve_matches_the_reference(N, counts, fp64, shift):
    from paper_0705_0495_gb300 import o2pic
    rng = np.random.default_rng(N + sum(counts))
    d = inputs.Discharge(n_cells=N, n_op=max(2, counts[2]), fp64=fp64, rf_phase=0.4)
    cells, offs = _particles(N, counts, fp64, ordered=N % 2 == 0, rng=rng)
    dev = []
    for a in cells + offs:  # arrays that start `shift` elements into an allocation
        t = torch.zeros(len(a) + shift, dtype=torch.from_numpy(a).dtype, device="cuda")
        t[shift:] = torch.from_numpy(a).cuda()
        dev.append(t)
    size = [4, 4, 4] + [8 if fp64 else 4] * 3
    ptr = [t.data_ptr() + shift * b for t, b in zip(dev, size)]
    out = [torch.full((N + 1,), math.nan, dtype=torch.float64, device="cuda") for _ in range(3)]
    for _ in range(2):  # the second call must not see the first one's sums
        o2pic.field_solve_static(o2pic.make_config(d), 11, ptr[:3], ptr[3:], counts, *[t.data_ptr() for t in out],
                                 torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    rho, phi, E = (t.cpu().numpy() for t in out)
    r, p, e, per = _reference(d, cells, offs, 11)
    assert np.all(np.abs(rho - r) <= (1e-15 if fp64 else 0.0) * per + 1e-14 * np.abs(r))
    assert np.max(np.abs(phi - p)) <= 1e-12 * np.max(np.abs(p))
    assert np.max(np.abs(E - e)) <= 1e-12 * np.max(np.abs(e)) * max(1.0, N / 64)

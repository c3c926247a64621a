"""Totals of float64 instances around the edges of the two-stage reduction, at
the tile shapes that float64 batches run (GPU)."""
import numpy as np
import pytest

from paper_2508_16997_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbve():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2508_16997_gb300 import lbve as m
    return m


@pytest.mark.parametrize("records", [511, 512, 513, 767, 768, 769])
@pytest.mark.parametrize("nx,tile_tx,rows", [
    (16, 0, 8),     # 128-thread CTAs by default (256 to 385 tiles of 256 nodes): 16 x 8 tiles
    (40, 40, 3),    # 128-thread CTAs, 40 x 3 tiles asked for
    (128, 128, 2),  # 256-thread CTAs, 128 x 2 tiles asked for
])
def test_float64_totals_match_fields(lbve, nx, tile_tx, rows, records):
    """One column of tiles, one record each.  The sums are compared with the
    fields' own: n additions of values of order one round by at most n 2^-53 of the
    sum of magnitudes on either side."""
    inst = wl.Instance(nx, records * rows, True, 0.5, 2.0, 1.0, 1e4, 0.05, 32.0, Fx=1e-5, Fy=-3e-6)
    init = wl.random_fields(inst.nx, inst.ny, seed=1, du=1e-3)
    s = lbve.Simulation([inst], precision=0, init_fields=[init], tile_tx=tile_tx)
    s.step(1)
    before = s.fields(0)
    s.step(2)
    f, t = s.fields(0), s.totals(0)
    rho, u = f[0], f[1:3]
    for got, v in ((t[0], f[0]), (t[1], rho * u[0]), (t[2], rho * u[1]), (t[3], f[3]), (t[4], f[4]),
                   (t[5], f[5])):
        assert abs(got - v.sum()) <= 4 * v.size * 2.0 ** -53 * np.abs(v).sum()
    res = np.abs(u - before[1:3]).max() / wl.velocity_scale(inst.Ma)
    assert abs(s.residual(0) - res) <= 2.0 ** -50 * res
    assert not s.status().any()

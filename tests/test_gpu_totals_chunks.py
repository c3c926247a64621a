"""Totals of instances around the edges of the two-stage reduction (GPU): up to
two chunks of 256 partial records go through one stage, more through two."""
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


@pytest.mark.parametrize("precision,rows", [(1, 3), (0, 8)])
@pytest.mark.parametrize("records", [1, 511, 512, 513, 767, 768, 769, 1537])
def test_totals_match_fields(lbve, precision, rows, records):
    """One column of 32 x rows tiles per record (float64: 256-thread tiles from 152
    records on), next to a second instance whose records must stay its own.  The
    sums are compared with the fields' own in float64: n additions of values of
    order one round by at most n 2^-53 of the sum of magnitudes."""
    ny = records * rows
    big = wl.Instance(32, ny, True, 0.5, 2.0, 1.0, 1e4, 0.05, 32.0, Fx=1e-5, Fy=-3e-6)
    small = wl.frm(20, Wi=2.0, Re=1.0, Ma=0.05)
    inits = [wl.random_fields(i.nx, i.ny, seed=k, du=1e-3) for k, i in enumerate((big, small))]
    s = lbve.Simulation([big, small], precision=precision, init_fields=inits)
    s.step(1)
    before = [s.fields(i) for i in range(2)]
    s.step(2)
    for i, inst in enumerate((big, small)):
        f, t = s.fields(i), s.totals(i)
        rho, u = f[0], f[1:3]
        if precision:  # the momentum's factor is the float32 density
            rho = rho.astype(np.float32).astype(np.float64)
        for got, v in ((t[0], f[0]), (t[1], rho * u[0]), (t[2], rho * u[1]), (t[3], f[3]), (t[4], f[4]),
                       (t[5], f[5])):
            # float32 instances sum exact products of float32 values
            assert abs(got - v.sum()) <= 4 * v.size * 2.0 ** -53 * np.abs(v).sum()
        Uc = wl.velocity_scale(inst.Ma)
        res = np.abs(u - before[i][1:3]).max() / Uc
        # a float32 instance subtracts float32 values: half an ulp of the difference
        assert abs(s.residual(i) - res) <= (2.0 ** -23 if precision else 2.0 ** -50) * res
    assert not s.status().any()

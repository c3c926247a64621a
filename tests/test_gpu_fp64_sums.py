"""Float64 steps over states whose populations span many binades: the block
fixed-point sums of the float64 kernels against the oracle (GPU)."""
import numpy as np
import pytest

from oracle_helpers import oracle_sim
from paper_2508_16997_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbve():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2508_16997_gb300 import lbve as m
    return m


def _instance(kind, nx):
    if kind == "mill":
        return wl.Instance(nx, 11, True, 0.5, 2.0, 1.0, 1e4, 0.05, 16.0, Fx=1e-5, Fy=-3e-6)
    return wl.channel(10, nx=nx, Wi=3.0)


@pytest.mark.parametrize("nx", [1, 5, 32, 33, 70])
@pytest.mark.parametrize("kind", ["mill", "channel"])
@pytest.mark.parametrize("du,dA,stretch", [(1e-2, 0.1, 1.0), (1e-12, 1e-12, 1.0), (0.0, 0.0, 1e-9)])
def test_wide_ranges_against_oracle(lbve, kind, nx, du, dA, stretch):
    """Three steps from random fields (velocities from 0 to 1e-2, conformations
    down to 1e-9).  The oracle carries full populations, so both sides are
    within a few hundred roundings (3 steps, 36 populations) of 2^-53 of the
    largest value of a field's lattice: 1e-13 of it."""
    inst = _instance(kind, nx)
    init = wl.random_fields(inst.nx, inst.ny, seed=3, du=du, drho=0.1 * du, dA=dA)
    init[3:] *= stretch
    s = lbve.Simulation([inst], precision=lbve.LBVE_FP64, init_fields=[init])
    o = oracle_sim(inst, init)
    s.step(3)
    o.step(3)
    got, ref = s.fields(0), o.fields()
    hydro = max(1.0, np.abs(ref[:3]).max())
    cde = max(1.0, np.abs(ref[3:]).max())
    # the stress feeds the velocity with mu_p / lambda A
    assert np.abs(got[:3] - ref[:3]).max() <= 1e-13 * max(hydro, cde)
    assert np.abs(got[3:] - ref[3:]).max() <= 1e-13 * cde


def test_rest_state_stays_exact(lbve):
    """Without force the rest state has zero deviations: they stay exactly zero."""
    inst = wl.Instance(20, 9, True, 0.5, 2.0, 1.0, 1e4, 0.05, 16.0)
    s = lbve.Simulation([inst], precision=lbve.LBVE_FP64)
    s.step(50)
    rest = np.array([1.0, 0, 0, 1, 0, 1])[:, None, None]
    np.testing.assert_array_equal(s.fields(0), np.broadcast_to(rest, (6, 9, 20)))


def test_overflow_is_reported(lbve):
    """Values whose sums leave the float64 range set the non-finite flag."""
    inst = wl.frm(16, Wi=2.0, Re=1.0, Ma=0.05)
    init = np.ones((6, 16, 16))
    init[1:3] = 0.0
    init[3:] = 1e308
    s = lbve.Simulation([inst], precision=lbve.LBVE_FP64, init_fields=[init])
    s.step(2)
    assert s.status()[0] & 1


@pytest.mark.parametrize("nx,ny,periodic", [(200, 200, True), (203, 197, False), (130, 400, True)])
def test_mid_size_cta_bit_identical(lbve, nx, ny, periodic):
    """152 to 759 tiles of 256 threads: the default 128-thread CTAs against the
    256-thread ones that a 128-wide tile asks for, bit for bit."""
    inst = wl.Instance(nx, ny, periodic, 0.5, 2.0, 1.0, 1e4, 0.05, 100.0, Fx=1e-5, Fy=-3e-6)
    init = wl.random_fields(nx, ny, seed=4, du=1e-3)
    runs = []
    for tx in (0, 128):
        s = lbve.Simulation([inst], precision=lbve.LBVE_FP64, init_fields=[init], tile_tx=tx)
        s.step(20)
        runs.append(s.fields(0))
    np.testing.assert_array_equal(runs[0], runs[1])

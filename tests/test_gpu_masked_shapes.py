"""The two launch shapes of masked tiles (few: for latency, many: for
throughput) and the 128-thread float64 CTAs with a mask (GPU)."""
import numpy as np
import pytest

from gpu_helpers import parity_errors
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


def fene(nx, ny, periodic=True):
    """Every tile of a FENE-P instance runs in the masked variant."""
    inst = wl.Instance(nx, ny, periodic, 0.5, 2.0, 1.0, 1e4, 0.05, 64.0, Fx=1e-5, Fy=-3e-6)
    inst.model, inst.L2 = 1, 60.0
    return inst


def gaps(nx, ny, periodic):
    """Two-node gaps along x and y (both difference rules next to solid
    nodes), solid nodes in a corner tile and in the ragged last one."""
    inst = wl.Instance(nx, ny, periodic, 0.5, 2.0, 1.0, 1e4, 0.05, 64.0, Fx=1e-5, Fy=-3e-6)
    s = np.zeros((ny, nx), np.uint8)
    s[6:13, 8] = s[6:13, 11] = 1
    s[9, 14:19] = s[12, 14:19] = 1
    s[ny - 9:ny - 4, nx - 9:nx - 5] = 1
    inst.solid = s
    return inst


def fields_of(lbve, batch, precision, inits, steps=12):
    s = lbve.Simulation(batch, precision=precision, init_fields=inits)
    s.step(steps)
    return s.fields(0), s.totals(0)


@pytest.mark.parametrize("precision,filler", [
    (1, 200),   # 32 x 3 tiles: 469 of the filler's
    (0, 136),   # 64-thread CTAs, 8 x 8 tiles: 289 and the first instance's 35 to 45
    (0, 200),   # 128-thread CTAs, 16 x 8 tiles: 325
    (0, 420)])  # 256-thread CTAs, 32 x 8 tiles: 742
@pytest.mark.parametrize("make", [lambda: fene(40, 67), lambda: gaps(45, 61, True),
                                  lambda: gaps(53, 50, False)], ids=["fene", "gaps", "gaps_walls"])
def test_shapes_agree_bit_for_bit(lbve, precision, filler, make):
    """An instance beside many masked tiles (throughput shape) and beside as many
    plain ones (latency shape; the CTA size follows the batch's size, so it
    is the same): the same fields and the same totals."""
    a = make()
    plain = wl.Instance(filler, filler, True, 0.5, 2.0, 1.0, 1e4, 0.05, 64.0)
    many = fene(filler, filler)
    inits = [wl.random_fields(i.nx, i.ny, seed=7, du=1e-3) for i in (a, plain)]
    few_f, few_t = fields_of(lbve, [a, plain], precision, inits)
    many_f, many_t = fields_of(lbve, [a, many], precision, inits)
    np.testing.assert_array_equal(few_f, many_f)
    np.testing.assert_array_equal(few_t, many_t)


@pytest.mark.parametrize("nx,ny,periodic", [(200, 200, True), (211, 203, False)])
def test_masked_mid_size_cta(lbve, nx, ny, periodic):
    """175 and 182 tiles of 256 threads: the masked 128-thread CTAs against the
    256-thread ones that a 128-wide tile asks for, bit for bit, and against the
    oracle."""
    inst = gaps(nx, ny, periodic)
    init = wl.random_fields(nx, ny, seed=4, du=1e-3)
    runs = []
    for tx in (0, 128):
        s = lbve.Simulation([inst], precision=lbve.LBVE_FP64, init_fields=[init], tile_tx=tx)
        s.step(20)
        runs.append(s.fields(0))
    np.testing.assert_array_equal(runs[0], runs[1])
    o = oracle_sim(inst, init)
    o.set_mask(inst.solid, None)
    o.step(20)
    err = parity_errors(runs[0], o.fields())
    assert err["u"] <= 1e-12 and err["C"] <= 1e-12 and err["C-I"] <= 1e-10, err


def test_open_cylinder_mid_size(lbve):
    """The open cylinder at R = 18 (170 tiles of 256 threads: 128-thread CTAs
    with mask, wall fractions and open columns) against the oracle."""
    inst = wl.cylinder_channel(18, Wi=0.5, Ma=0.05, open_x=True)
    s = lbve.Simulation([inst], precision=lbve.LBVE_FP64)
    o = oracle_sim(inst)
    o.set_mask(inst.solid, inst.wall_q)
    s.step(40)
    o.step(40)
    err = parity_errors(s.fields(0), o.fields())
    assert err["u"] <= 1e-12 and err["C"] <= 1e-12 and err["C-I"] <= 1e-10, err

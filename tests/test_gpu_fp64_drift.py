"""Mass of a float64 run over 1e5 steps: the roundings of the lattice sums have
no sign beyond those of the constants and of ties (GPU)."""
import math

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


@pytest.mark.parametrize("beta,drho", [(1.0, 1e-5), (0.5, 1e-5), (0.5, -1e-5)])
def test_mean_density_does_not_drift(lbve, beta, drho):
    """A slow periodic mill whose density is off 1 by drho, one-signed and a
    hundredth of rho u.  Allowed over the steps: per step 2^-53 of drho (the
    constant 1/9 is off by 2^-54, ties by half a last place at most); six standard
    errors of the two means read (fields round at 2^-53: rms 2^-53 / sqrt(3) a
    node); and six of the random walk of nine population roundings per node and
    step (populations up to rho u / 3, below 2^-8: last place 2^-61)."""
    N, steps = 32, 100000
    inst = wl.frm(N, beta=beta, Wi=0.5, Re=1.0, Ma=0.01)
    init = np.zeros((6, N, N))
    init[0], init[3], init[5] = 1.0 + drho, 1.0, 1.0
    s = lbve.Simulation([inst], precision=lbve.LBVE_FP64, init_fields=[init])
    means = []
    for n in (2000, steps):  # the start-up's transient first
        s.step(n)
        means.append(math.fsum((s.fields(0)[0] - 1.0).ravel()) / N ** 2)
    reading = 6 * math.sqrt(2) * 2.0 ** -53 / math.sqrt(3) / N
    walk = 6 * math.sqrt(9 * steps / 12) * 2.0 ** -61 / N
    assert abs(means[1] - means[0]) <= steps * 2.0 ** -53 * abs(drho) + reading + walk

"""The adjoint's workspace: what one more stored state takes, and the same
gradient from every checkpoint interval that a workspace allows (GPU)."""
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


def open_channel():
    inst = wl.channel(13, nx=12, Wi=1.0, Sc=1e3)
    inst.open_x = True
    inst.inlet = wl.poiseuille_inlet(13, 1.2 * wl.velocity_scale(inst.Ma), 20.0)
    return inst


CASES = {"mill": lambda: wl.frm(8, Wi=1.0, Re=1.0, Ma=0.05),
         "channel": lambda: wl.channel(9, nx=5, Wi=1.0, Sc=1e3),
         "disc": lambda: wl.circle_box(14, 12, R=2.3, cx=6.2, cy=5.6, Fx=1e-4, Wi=1.0),
         "open": open_channel}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", ["mill", "channel", "open"])
def test_a_stored_state_takes_a_state(lbve, case, precision):
    """Interval 1 stores every state: 41 planes (256-byte aligned) per step and no
    tables that grow with the steps, so workspaces sized by the states keep their
    interval."""
    inst = CASES[case]()
    sim = lbve.Simulation([inst], precision=precision)
    stride = -(-inst.n_nodes // 64) * 64
    state = 41 * stride * (4 if precision else 8)
    n = [lbve.lbve_adjoint_workspace_bytes_interval(sim.h, 0, T, 1) for T in (1000, 1001, 5000)]
    assert abs(n[1] - n[0] - state) < 256
    assert abs(n[2] - n[0] - 4000 * state) < 256


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", sorted(CASES))
def test_every_interval_gives_the_same_gradient(lbve, case, precision):
    """70 steps with all states stored, with every second, third and fifth, and at
    the square-root interval (9): the forward sweep's descriptors go up in pieces
    of 64 with a shorter last one.  Bit for bit the same gradients."""
    import torch
    inst, T = CASES[case](), 70
    sim = lbve.Simulation([inst], precision=precision)
    init = wl.random_fields(inst.nx, inst.ny, seed=3, du=1e-3)
    seed = torch.from_numpy(np.random.default_rng(2).standard_normal((6, inst.ny, inst.nx))).cuda()
    if inst.solid is not None:
        seed *= torch.from_numpy(1.0 - inst.solid.astype(float)).cuda()
    grads = []
    for interval in (1, 2, 3, 5, 9):
        n = lbve.lbve_adjoint_workspace_bytes_interval(sim.h, 0, T, interval)
        ws = torch.full((n,), 0xff, dtype=torch.uint8, device="cuda")  # NaN where nothing is written
        out = torch.empty((2, inst.ny, inst.nx), dtype=torch.float64, device="cuda")
        lbve.lbve_adjoint_step(sim.h, 0, init, seed.data_ptr(), T, ws.data_ptr(), n, out.data_ptr(),
                               inst.n_nodes)
        grads.append(out.cpu().numpy())
    assert np.isfinite(grads[0]).all() and np.abs(grads[0]).max() > 0
    for g in grads[1:]:
        np.testing.assert_array_equal(g, grads[0])

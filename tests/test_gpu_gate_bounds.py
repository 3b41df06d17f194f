"""The near-contact list that a step writes, at the threshold where the gate's edge is widest in phi
(q_th = 0.25): the pass over the listed tiles must find the films of the pass over every tile, in the step
in which their cells begin to pass the gate. Nothing acts on the flow (equal densities, no surface tension,
no repulsion, D = 0), so a uniform velocity carries phi and the cells' phi after a step can be set."""
import numpy as np
import pytest

from paper_2603_17481_gb300 import binding as B
from paper_2603_17481_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2603_17481_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    return True


def _inside(edge):
    """The fixed-point value next to edge that passes the gate with its 8 neighbours on either side (below
    1/2 the rounding of 1 - phi lets through three values of four)."""
    v = int(edge * 2 ** 30) + np.arange(-500, 500)
    pc = v.astype(np.float32) * np.float32(2.0 ** -30)
    run = np.convolve(pc * (np.float32(1) - pc) >= np.float32(0.25), np.ones(17), "same") == 17
    return float(v[run][np.argmin(np.abs(v[run] - edge * 2 ** 30))]) / 2 ** 30


def _stepped(sim, row, cells):
    """phi along x after one step from rows equal to row, in a flow of 0.04 along x."""
    phi = np.tile(row, cells // row.size)
    u = np.zeros((3, cells))
    u[0] = 0.04
    sim.init_fields(phi, u)
    sim.step(1)
    ph, _, _ = sim.read_fields()
    return ph


@pytest.mark.parametrize("edge", [0.49993, 0.49997, 0.50003, 0.50007])
@pytest.mark.parametrize("dim,dims", [(3, (44, 12, 9)), (3, (64, 16, 8)), (2, (70, 40, 1))])
def test_film_whose_cells_enter_the_gate_at_its_edge(dim, dims, edge):
    """Two parallel interfaces three cells apart. Only the cells in columns 15 and 18 pass the gate after the
    step, with phi = edge, and none before it."""
    cfg = W.base_config(dim, *dims, 19 if dim == 3 else 9, rho_g=1.0, sigma=0.0, A_rep=0.0, D=0.0, q_th=0.25)
    cells, edge = dims[0] * dims[1] * dims[2], _inside(edge)
    row = np.full(dims[0], 0.02)
    row[14:20] = [0.8, edge, 0.1, 0.1, edge, 0.8]
    sim = B.Lbm(cfg)
    for _ in range(40):  # the start whose step ends at edge: phi moves by a few percent: a contraction
        row = W.to_q30_grid(row)
        ph = _stepped(sim, row, cells)
        row[[15, 18]] += edge - ph[[15, 18]]
    row = W.to_q30_grid(row)
    assert np.all(np.abs(row[[15, 18]] - 0.5) > 2e-3)  # not gated before the step
    sim.close()

    sim = B.Lbm(cfg)  # no force of an earlier pass is held
    ph = _stepped(sim, row, cells)
    gated = np.float32(ph) * (np.float32(1) - np.float32(ph)) >= np.float32(0.25)
    assert gated.sum() == 2 * dims[1] * dims[2] and np.max(np.abs(ph[gated] - edge)) < 1e-6
    listed = sim.nci_diagnostics()["V_film"]
    part, _ = sim.read_nci()
    assert listed == (part[:, 0] != B.NO_PARTNER).sum() == 2 * dims[1] * dims[2]
    sim.close()

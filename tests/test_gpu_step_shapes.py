"""The step's kernels at the edges of their tiles and dispatch rules, against the FP64 oracle: paired
hydrodynamic tiles (32 x 2 x 4 cells) that are cut in x, y and z, a grid with more tiles in y than one
launch may have blocks, phase marches with two and with four rows per thread on both sides of their
rule, and 2D grids most of whose phase tiles are empty. Tolerances are those of the parity tests:
1e-6 on populations and velocities and 1e-7 on phi after one step from the same input; 1e-5 on phi and
1e-6 on velocities of a trajectory."""
import numpy as np
import pytest

import oracle as O
from paper_2603_17481_gb300 import binding as B
from paper_2603_17481_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2603_17481_gb300 import build
    build.build()
    O.build()
    torch.cuda.set_device(0)
    return True


@pytest.mark.parametrize("Q,shape", [(19, (2, 1, 1)), (19, (34, 3, 5)), (27, (30, 2, 4)), (27, (66, 5, 3)), (19, (62, 131, 2)),
                                     (19, (2, 131080, 1)), (19, (84, 52, 31)), (19, (198, 202, 133))])
def test_one_step_on_cut_tiles(Q, shape):
    """One step from a random non-equilibrium state; sum(phi) is unchanged in fixed point."""
    cfg = W.base_config(3, *shape, Q, rho_g=0.1, nci_on=0)
    phi, u = W.smooth_random_fields(cfg, seed=sum(shape), pairs=False)
    phi = W.to_q30_grid(phi)
    P = O.make_params(cfg)
    N = W.ncells(cfg)
    _, w = O.lattice(3, Q)
    f = O.init(P, phi, u, pstar=W.noise(N, 5, 5e-3)) + 2e-3 * w[:, None] * W.noise((Q, N), 6)
    sim = B.Lbm(cfg)
    sim.set_state(f, phi)
    sim.step(1)
    fg, phg = sim.get_state()
    fo, pho, _ = O.step(P, f, phi, 1)
    assert np.max(np.abs(fg - fo)) < 1e-6
    assert np.max(np.abs(phg - pho)) < 1e-7
    assert np.round(phg * 2 ** 30).sum() == np.round(phi * 2 ** 30).sum()
    sim.close()


@pytest.mark.parametrize("shape,centers", [((301, 203, 1), [(70.3, 60.1, 0.0), (98.9, 63.7, 0.0)]),
                                           ((256, 96, 1), [(3.2, 2.4, 0.0), (247.5, 80.3, 0.0)]),
                                           ((129, 65, 1), [])])
def test_2d_with_empty_tiles(shape, centers):
    """Two droplets (inside the grid, and across its corner) in a grid that is otherwise exactly zero,
    through 60 steps with the repulsion on, and a grid that is zero everywhere."""
    cfg = W.base_config(2, *shape, 9)
    phi, u = W.droplet_fields(cfg, centers, [12.0, 12.0], [(0.02, 0.005, 0.0), (-0.02, 0.0, 0.0)])
    phi = W.to_q30_grid(phi)
    assert np.mean(phi == 0.0) > 0.5
    P = O.make_params(cfg)
    fo, pho, _ = O.step(P, O.init(P, phi, u), phi, 60)
    _, uo = O.moments(P, fo, pho)
    sim = B.Lbm(cfg)
    sim.init_fields(phi, u)
    sim.step(60)
    phg, ug, _ = sim.read_fields()
    assert np.max(np.abs(phg - pho)) <= 1e-5
    assert np.max(np.abs(ug - uo)) <= 1e-6
    assert np.round(phg * 2 ** 30).sum() == np.round(phi * 2 ** 30).sum()
    part, _ = sim.read_nci()
    film = part[:, 0] != B.NO_PARTNER
    assert sim.nci_diagnostics()["V_film"] == film.sum()  # the pass over the listed tiles misses none
    sim.close()

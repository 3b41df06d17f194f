"""The step's kernels where the tests of cut tiles, of the split step and of the march's rule leave a gap: paired
tiles cut in x, y and z with 2-byte populations, the split step where the last near-contact tile holds one
to three rows in y, and a grid far beyond the line at which the march takes four rows per thread."""
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


@pytest.mark.parametrize("store", ["f16", "bf16"])
@pytest.mark.parametrize("Q,shape", [(19, (2, 1, 1)), (19, (34, 3, 5)), (27, (30, 2, 4)), (27, (66, 5, 3)), (19, (62, 131, 2))])
def test_one_step_with_2_byte_populations(store, Q, shape):
    """One step from a random non-equilibrium state as the store holds it. Populations within one unit of
    the storage precision of f / w plus the 1e-6 of the FP32 tests; velocities within 1e-6, phi 1e-7."""
    cfg = W.base_config(3, *shape, Q, rho_g=0.1, nci_on=0)
    phi, u = W.smooth_random_fields(cfg, seed=sum(shape), pairs=False)
    phi = W.to_q30_grid(phi)
    P = O.make_params(cfg)
    N = W.ncells(cfg)
    _, w = O.lattice(3, Q)
    f = O.init(P, phi, u, pstar=W.noise(N, 5, 5e-3)) + 2e-3 * w[:, None] * W.noise((Q, N), 6)
    sim = B.Lbm(cfg, store=store)
    sim.set_state(f, phi)
    f, _ = sim.get_state()
    _, ug, _ = sim.read_fields()
    _, uo = O.moments(P, f, phi)
    assert np.max(np.abs(ug - uo)) < 1e-6
    sim.step(1)
    fg, phg = sim.get_state()
    sim.close()
    fo, pho, _ = O.step(P, f, phi, 1)
    ulp = 2.0 ** -10 if store == "f16" else 2.0 ** -7
    assert np.all(np.abs(fg - fo) <= 1e-6 + ulp * np.abs(fo) + 2.0 ** -24 * w[:, None])
    assert np.max(np.abs(phg - pho)) < 1e-7
    assert np.round(phg * 2 ** 30).sum() == np.round(phi * 2 ** 30).sum()


@pytest.mark.parametrize("store,Q", [("f32", 19), ("bf16", 19), ("f16", 27)])
@pytest.mark.parametrize("dims", [(66, 41, 30), (34, 42, 29), (64, 43, 31)])
def test_split_step_with_a_film_in_a_cut_tile(dims, store, Q):
    """Two droplets closing in on the last rows of y (and their periodic images in the first), on 40 steps
    of the split step and of the one-stream step: the same bits."""
    cfg = W.base_config(3, *dims, Q, rho_g=0.1)
    c = [dims[0] / 2.0, dims[1] - 1.6, dims[2] / 2.0]
    phi, u = W.droplet_fields(cfg, [(c[0] - 9.2, c[1], c[2]), (c[0] + 9.4, c[1] + 0.3, c[2] - 0.4)], [7.0, 7.0],
                              [(0.02, 0.0, 0.0), (-0.02, 0.0, 0.0)])
    phi = W.to_q30_grid(phi)
    out = []
    for blocks in (0, 38):
        sim = B.Lbm(cfg, store=store)
        sim.set_overlap(blocks)
        sim.init_fields(phi, u)
        sim.step(40)
        out.append(sim.get_state() + sim.read_nci())
        sim.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    film = out[0][2][:, 0].reshape(dims[2], dims[1], dims[0]) != B.NO_PARTNER
    assert film[:, dims[1] // 8 * 8:].any()  # in the cut tiles


def test_four_rows_per_thread_far_beyond_the_line():
    """One step on 230 x 210 x 150, 1.34 times the line's 44 planes per warp on 152 SMs."""
    cfg = W.base_config(3, 230, 210, 150, 19, rho_g=0.1, nci_on=0)
    assert (230 + 27) // 28 * ((210 + 3) // 4) * 150 > 1.3 * 44 * 4 * 2 * 152
    phi, u = W.smooth_random_fields(cfg, seed=7, pairs=False)
    phi = W.to_q30_grid(phi)
    P = O.make_params(cfg)
    f = O.init(P, phi, u)
    sim = B.Lbm(cfg)
    sim.set_state(f, phi)
    sim.step(1)
    fg, phg = sim.get_state()
    sim.close()
    fo, pho, _ = O.step(P, f, phi, 1)
    assert np.max(np.abs(fg - fo)) < 1e-6
    assert np.max(np.abs(phg - pho)) < 1e-7
    assert np.round(phg * 2 ** 30).sum() == np.round(phi * 2 ** 30).sum()

"""A grid of one plane of more than 2^30 cells, whose row offsets within the plane exceed 32 bits in bytes: the
phase march takes its 64-bit instance there. As in the test of the largest grids, a field that repeats a
small period must stay the small grid's state repeated, cell by cell."""
import numpy as np
import pytest

from paper_2603_17481_gb300 import binding as B
from paper_2603_17481_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _host_free():
    with open("/proc/meminfo") as f:
        return next(int(s.split()[1]) * 1024 for s in f if s.startswith("MemAvailable"))


def test_plane_beyond_32_bit_offsets_matches_the_repeated_small_grid():
    import torch
    from paper_2603_17481_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    # odd sides: both grids run the one-cell hydrodynamic kernel. 2^30 cells are 32731 rows and 1369 cells of the
    # large grid, which is no multiple of the period, so an offset that wrapped would read another phase of it.
    small, reps = (45, 40, 1), (729, 820)
    big = (small[0] * reps[0], small[1] * reps[1], 1)
    N = big[0] * big[1]
    assert 2 ** 30 < N < 2 ** 31
    if torch.cuda.mem_get_info()[0] < 200e9 or _host_free() < 60e9:
        pytest.skip("needs 182 GB of device and 45 GB of host memory")
    steps = 3
    cs, cb = W.base_config(3, *small, 19, rho_g=0.1), W.base_config(3, *big, 19, rho_g=0.1)
    phi, _ = W.smooth_random_fields(cs, seed=13)
    phi = W.to_q30_grid(phi)
    s = B.Lbm(cs, store="f16")
    s.init_fields(phi, np.zeros((3, phi.size)))
    film_s = s.nci_diagnostics()["V_film"]
    s.step(steps)
    ph_s, _, _ = s.read_fields(want=("phi",))
    s.close()
    assert film_s > 0 and np.max(np.abs(ph_s - phi)) > 1e-3  # near contact is active, phi moves

    field = np.tile(phi.reshape(small[1], small[0]), (reps[1], reps[0])).reshape(-1)
    b = B.Lbm(cb, store="f16")
    b.init_fields(field, np.zeros((3, N)))
    assert b.nci_diagnostics()["V_film"] == film_s * reps[0] * reps[1]
    b.step(steps)
    b.read_fields(phi=field, want=())
    b.close()
    # The same arithmetic on both; a population whose FP32 value rounded to the other side in FP16 would move a
    # velocity by up to 5e-6, and phi by as much a step.
    want = np.tile(ph_s.reshape(small[1], small[0]), (1, reps[0]))
    for y in range(0, big[1], small[1]):
        rows = field[y * big[0]:(y + small[1]) * big[0]].reshape(small[1], big[0])
        assert np.max(np.abs(rows - want)) <= 2e-5, y

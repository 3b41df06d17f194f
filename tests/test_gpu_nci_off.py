"""Contexts with the near-contact interaction off: they hold none of its mask records, and the read-back of
the near-contact pass, which runs on them too, finds what a context with it on finds."""
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


def test_no_masks_without_the_interaction():
    """256^3 cells: the masks take a byte per cell, the brick ranges and lists of a context that has the
    interaction on a quarter of that."""
    import torch
    N = 256 ** 3

    def held(nci_on):
        free = torch.cuda.mem_get_info()[0]
        sim = B.Lbm(W.base_config(3, 256, 256, 256, 19, nci_on=nci_on))
        used = free - torch.cuda.mem_get_info()[0]
        sim.close()
        return used
    for on in (1, 0):  # modules and the driver's own pools
        held(on)
    assert held(1) - held(0) > N


@pytest.mark.parametrize("dim,dims", [(3, (40, 24, 20)), (3, (33, 17, 5)), (2, (70, 45, 1))])
def test_read_back_without_the_interaction(dim, dims):
    Q = 19 if dim == 3 else 9
    out = []
    for on in (1, 0):
        cfg = W.base_config(dim, *dims, Q, rho_g=0.1, w=1, cos_opp=0.1, nci_on=on)
        phi, u = W.smooth_random_fields(cfg, seed=3)
        sim = B.Lbm(cfg)
        sim.init_fields(W.to_q30_grid(phi), u)
        out.append([sim.read_nci() for _ in range(2)][1])
        sim.close()
    (p1, f1), (p0, f0) = out
    assert (p1[:, 0] != B.NO_PARTNER).sum() > 0
    assert np.array_equal(p1, p0) and np.array_equal(f1, f0)

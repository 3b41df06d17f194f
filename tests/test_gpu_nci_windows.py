"""The near-contact pass on the grids where its row masks, brick ranges and windows can go wrong: sides
that are not multiples of 4 or 32, rows shorter than a mask word and than a window, window radii 1 to
3, and facing thresholds down to the ones that make a direction class hold every cell."""
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
    torch.cuda.set_device(0)
    return True


@pytest.mark.parametrize("dims", [(33, 17, 12), (97, 11, 9), (38, 9, 5), (31, 13, 6), (5, 7, 9), (3, 20, 33), (64, 16, 8),
                                  (66, 14, 10), (32, 8, 4), (37, 21, 1), (100, 40, 1), (6, 50, 1)])
@pytest.mark.parametrize("w,cos_opp", [(3, -0.8), (2, -0.8), (1, -0.3), (3, -0.95), (3, 0.1)])
def test_partners_on_ragged_grids(dims, w, cos_opp):
    """The pass over every tile against the oracle's brute-force search (partners equal but where the
    oracle's decision margin is below 1e-5), and the pass over the listed tiles, at t = 0 and after two
    steps, against the pass over every tile."""
    dim = 3 if dims[2] > 1 else 2
    cfg = W.base_config(dim, *dims, 19 if dim == 3 else 9, rho_g=0.1, w=w, cos_opp=cos_opp)
    phi, u = W.smooth_random_fields(cfg, seed=sum(dims) + w)
    sim = B.Lbm(cfg)
    sim.init_fields(W.to_q30_grid(phi), u)
    for steps in (0, 2):
        sim.step(steps)
        ph, _, _ = sim.read_fields()
        dl = sim.nci_diagnostics()
        part, frep = sim.read_nci()
        film = part[:, 0] != B.NO_PARTNER
        assert dl["V_film"] == film.sum()
        s = np.sqrt((frep[:, film] ** 2).sum(axis=0)).sum()
        assert abs(dl["sum_rep"] - s) <= 1e-6 * s
        assert not np.any(frep[:, ~film])
        P = O.make_params(cfg)
        P.decide_f32 = 1
        part_o, _, marg = O.nci(P, ph)
        mis = np.any(part != part_o, axis=1)
        assert np.all(marg[mis] < 1e-5)
    sim.close()

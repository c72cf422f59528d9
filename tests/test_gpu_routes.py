"""Rules that choose a step's form where a size in itself does not: on both sides the bits of the
generic fused step."""
import numpy as np
import pytest

from cases import mixture_dict, smooth_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fm():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2212_10680_gb300 import fmlbm
    return fmlbm


@pytest.mark.parametrize("n,precision,shape", [(2, "fp32", (36000, 40)), (3, "bf16dev", (65536, 16)),
                                               (2, "fp16dev", (43000, 50))])
def test_monitored_runs_of_wide_lattices(fm, n, precision, shape):
    # few long strips of a march: requests by fused sums (the last: by snapshot and reduction)
    mixd = mixture_dict(n, "pr", Tr=0.9, kappa_scale=0.3)
    rho = smooth_state(n, *shape, seed=7)
    out = []
    for tile_y in (8, 16):
        lat = fm.Lattice(fm.mixture_from_dict(mixd), *shape, 0.9, precision=precision)
        fm.fmlbm_set_tile_height(lat.h, tile_y)
        lat.init(rho)
        out.append(tuple(fm.fmlbm_step_diagnostics(lat.h, 3, n)) + lat.distributions())
        lat.close()
    assert all(np.array_equal(u, v) for u, v in zip(*out))

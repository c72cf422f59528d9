"""The split step (FP64 storage and ln f in double: two launches over scratch planes) against the
fused step of the same library, which 16-row tiles still run: same bits, at the edges of its
blocks and on both sides of its block-height rule, with and without a diagnostics request."""
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


def _run(fm, mixd, rho, precision, stencil, velocity, tile_y, monitored):
    n, ny, nx = rho.shape
    lat = fm.Lattice(fm.mixture_from_dict(mixd), nx, ny, 0.9, stencil, precision, velocity)
    fm.fmlbm_set_tile_height(lat.h, tile_y)
    lat.init(rho)
    rows = fm.fmlbm_step_diagnostics(lat.h, 3, n) if monitored else (lat.step(3),)
    out = lat.distributions() + tuple(rows)
    lat.close()
    return out


@pytest.mark.parametrize("precision,n,eos,stencil,velocity", [
    ("fp64", 2, "pr", "isotropic", "lagged"), ("fp64", 1, "vdw", "central", "current"),
    ("fp64", 4, "srk", "isotropic", "lagged"), ("bf16dev_lnf64", 3, "pr", "isotropic", "lagged"),
    ("fp16dev_lnf64", 2, "srk", "central", "current")])
@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (33, 7), (64, 16), (31, 19), (256, 256), (257, 256)])
def test_split_step_is_bit_identical_to_the_fused_step(fm, precision, n, eos, stencil, velocity, shape):
    nx, ny = shape
    mixd = mixture_dict(n, eos, Tr=0.9, kappa_scale=0.3, M=[1.0, 1.7, 0.6, 1.2][:n], kij=0.03)
    rho = smooth_state(n, nx, ny, seed=nx + ny)
    for monitored in (False, True):
        a = _run(fm, mixd, rho, precision, stencil, velocity, 8, monitored)
        b = _run(fm, mixd, rho, precision, stencil, velocity, 16, monitored)
        for u, v in zip(a, b):
            if u is not None:
                assert np.array_equal(u, v)

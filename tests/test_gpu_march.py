"""The packed and the marching step (float and 16-bit storage) against the generic fused step of the
same library, which 16-row tiles run: same bits, around the size rules between them, at widths and
heights that leave ragged strips, tiles and chunks, for every option, with and without a
diagnostics request."""
import numpy as np
import pytest

from cases import mixture_dict, smooth_state

pytestmark = pytest.mark.gpu

OPTIONS = {"pr": ("pr", "isotropic", "lagged"), "srk": ("srk", "central", "current"), "vdw": ("vdw", "isotropic", "current")}


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
    rows = ()
    lat.step(2)
    if monitored:
        rows = fm.fmlbm_step_diagnostics(lat.h, 3, n)
    else:
        lat.step(2)
    out = lat.distributions() + tuple(rows)
    lat.close()
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("n,option", [(2, "pr"), (2, "srk"), (3, "pr"), (3, "vdw")])
@pytest.mark.parametrize("shape", [(256, 255), (257, 256), (1024, 512), (3, 65536), (65536, 9), (727, 733), (29, 18101)])
def test_packed_and_marching_steps_are_bit_identical_to_the_fused_step(fm, precision, n, option, shape):
    eos, stencil, velocity = OPTIONS[option]
    nx, ny = shape
    mixd = mixture_dict(n, eos, Tr=0.9, kappa_scale=0.3, M=[1.0, 1.7, 0.6][:n], kij=0.03)
    rho = smooth_state(n, nx, ny, seed=nx + ny)
    for monitored in (False, True):
        a = _run(fm, mixd, rho, precision, stencil, velocity, 8, monitored)
        b = _run(fm, mixd, rho, precision, stencil, velocity, 16, monitored)
        for u, v in zip(a, b):
            assert np.array_equal(u, v)


def test_marching_step_without_l1_places_and_beyond_one_wave(fm):
    # a state larger than the L2 (two waves of chunks in 16-bit storage), and one above the FP32 bound
    for precision, nx, ny in (("bf16dev", 2900, 1501), ("fp32", 1900, 1811)):
        mixd = mixture_dict(2, "pr", Tr=0.9, kappa_scale=0.3)
        rho = smooth_state(2, nx, ny, seed=5)
        a = _run(fm, mixd, rho, precision, "isotropic", "lagged", 8, False)
        b = _run(fm, mixd, rho, precision, "isotropic", "lagged", 16, False)
        assert all(np.array_equal(u, v) for u, v in zip(a, b))


def test_a_bad_node_is_latched_by_the_marching_step(fm):
    mixd = mixture_dict(2, "pr", Tr=0.9, kappa_scale=0.3)
    rho = smooth_state(2, 1024, 600, seed=1)
    rho[1, 431, 1023] = -1e-3
    lat = fm.Lattice(fm.mixture_from_dict(mixd), 1024, 600, 1.0)
    lat.init(rho)
    lat.step(1)
    with pytest.raises(fm.FmlbmError) as e:
        lat.synchronize()
    assert e.value.status == fm.E_NONPHYSICAL
    assert fm.fmlbm_error_node(lat.h) == (1, 1023, 431)
    lat.close()

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


@pytest.mark.parametrize("precision,count,shape", [
    ("fp32", 64, (96, 96)),       # several packed launches of more than a wave each; single steps by the batch kernel
    ("bf16dev", 130, (33, 17)),   # small lattices in several launches: the batch kernel
    ("fp32", 17, (40, 33)),       # one launch with the larger parameters; single steps by the batch kernel
    ("fp16dev", 5, (50, 41))])    # one launch with the smaller ones
def test_batches_of_many_lattices(fm, precision, count, shape):
    # calls of one and of several steps in turn, so that packed and unpacked steps follow each other
    mixd = mixture_dict(n=2, Tr=1.05, kappa_scale=0.5)
    b = fm.fmlbm_batch_create(2, precision, count)
    L = fm.make_lattice(*shape, 0.9, precision=precision)
    rhos = [smooth_state(2, *shape, seed=k) for k in range(count)]
    slots = [fm.fmlbm_batch_add(b, fm.mixture_from_dict(mixd), L, r) for r in rhos]
    for n in (1, 3, 1, 2, 1):
        fm.fmlbm_batch_step(b, n)
    nx, ny = shape
    for k in sorted({0, count // 2, count - 1}):
        g, F = np.empty((2, 9, ny, nx)), np.empty((2, ny, nx))
        fm.fmlbm_batch_get_distributions(b, slots[k], g, F)
        lat = fm.Lattice(fm.mixture_from_dict(mixd), nx, ny, 0.9, precision=precision)
        fm.fmlbm_set_tile_height(lat.h, 16)
        lat.init(rhos[k])
        lat.step(8)
        want = lat.distributions()
        lat.close()
        assert np.array_equal(g, want[0]) and np.array_equal(F, want[1]), k
    fm.fmlbm_batch_destroy(b)


@pytest.mark.parametrize("precision,trials", [("fp32", 5), ("fp64", 8)])   # packed on 8-row tiles; never packed
def test_batch_autotune_tries_each_grid_once(fm, precision, trials):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    b = fm.fmlbm_batch_create(2, precision, 2)
    mix = fm.mixture_from_dict(mixture_dict(n=2, Tr=1.05, kappa_scale=0.5))
    slot = fm.fmlbm_batch_add(b, mix, fm.make_lattice(100, 70, 1.0, precision=precision), smooth_state(2, 100, 70))
    ty, blocks, _ = fm.fmlbm_batch_autotune(b, 3)
    assert fm.fmlbm_batch_slot_info(b, slot)[0] == trials * (1 + 3)
    tiles = 4 * 9   # of 32 x 8 nodes
    assert blocks == tiles if precision == "fp32" and ty == 8 else blocks in (sms, 2 * sms, 4 * sms, 8 * sms)
    fm.fmlbm_batch_destroy(b)

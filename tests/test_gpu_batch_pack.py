"""Packed batch steps: every lattice of a batch bit-identical to the same lattice alone, at the
edges of the groups of lattices that one launch takes, and under capture."""
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


def _add(fm, b, k, precision, options):
    nx, ny = 9 + 29 * k % 67, 8 + 13 * k % 41   # narrower than a tile, ragged, whole tiles
    eos, stencil, force = options
    mixd = mixture_dict(n=2, eos=eos, Tr=1.05, kappa_scale=0.5, M=[1.0, 1.0 + 0.01 * k])
    rho = smooth_state(2, nx, ny, seed=k)
    L = fm.make_lattice(nx, ny, 0.9, stencil, precision, force)
    return fm.fmlbm_batch_add(b, fm.mixture_from_dict(mixd), L, rho), mixd, rho, options


def _same(fm, b, case, precision, steps):
    slot, mixd, rho, (_, stencil, force) = case
    ny, nx = rho.shape[1:]
    g, F = np.empty((2, 9, ny, nx)), np.empty((2, ny, nx))
    fm.fmlbm_batch_get_distributions(b, slot, g, F)
    lat = fm.Lattice(fm.mixture_from_dict(mixd), nx, ny, 0.9, stencil, precision, force)
    fm.fmlbm_set_tile_height(lat.h, 16)
    lat.init(rho)
    lat.step(steps)
    gs, Fs = lat.distributions()
    lat.close()
    return np.array_equal(g, gs) and np.array_equal(F, Fs)


SPEC = ("pr", "isotropic", "lagged")


@pytest.mark.parametrize("precision,count", [("fp32", 1), ("fp32", 16), ("fp16dev", 17), ("bf16dev", 48), ("fp32", 49)])
def test_groups_of_lattices(fm, precision, count):
    b = fm.fmlbm_batch_create(2, precision, count + 2)
    cases = [_add(fm, b, k, precision, SPEC) for k in range(count)]
    fm.fmlbm_batch_step(b, 3)
    # a slot leaves and another joins at another count of steps
    if count > 1:
        fm.fmlbm_batch_set_active(b, cases[0][0], False)
    late = _add(fm, b, count, precision, SPEC)
    fm.fmlbm_batch_step(b, 4)
    assert _same(fm, b, late, precision, 4)
    for k, case in enumerate(cases):
        assert _same(fm, b, case, precision, 3 if k == 0 and count > 1 else 7), k
    fm.fmlbm_batch_destroy(b)


@pytest.mark.parametrize("precision", ["fp32", "fp16dev"])
def test_mixed_options(fm, precision):
    b = fm.fmlbm_batch_create(2, precision, 4)
    cases = [_add(fm, b, k, precision, o)
             for k, o in enumerate([SPEC, ("srk", "central", "current"), ("pr", "isotropic", "current")])]
    fm.fmlbm_batch_step(b, 5)
    for case in cases:
        assert _same(fm, b, case, precision, 5)
    fm.fmlbm_batch_destroy(b)


def test_captured_steps_replay(fm):
    # three replays of one captured step, between steps that are launched
    import torch
    s = torch.cuda.Stream()
    b = fm.fmlbm_batch_create(2, "fp32", 2, s.cuda_stream)
    case = _add(fm, b, 3, "fp32", SPEC)
    fm.fmlbm_batch_step(b, 1)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        fm.fmlbm_batch_step(b, 1)
    with torch.cuda.stream(s):
        for _ in range(3):
            graph.replay()
    fm.fmlbm_batch_step(b, 1)
    assert _same(fm, b, case, "fp32", 5)
    fm.fmlbm_batch_destroy(b)

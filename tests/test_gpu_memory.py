"""Device memory of a handle: what it holds, and that stepping takes none."""
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


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _lattice(fm, n, nx, ny, precision):
    lat = fm.Lattice(fm.mixture_from_dict(mixture_dict(n, Tr=0.9, kappa_scale=0.3)), nx, ny, 0.9, precision=precision)
    lat.init(smooth_state(n, nx, ny, seed=1))
    return lat


def _monitored(fm, lat, n):
    fm.fmlbm_diagnostics_wait(lat.h, fm.fmlbm_diagnostics_async(lat.h), n)
    t = fm.fmlbm_diagnostics_async(lat.h)
    lat.step(1)
    fm.fmlbm_diagnostics_wait(lat.h, t, n)
    lat.synchronize()


@pytest.mark.parametrize("n,precision,shape", [(2, "fp32", (2048, 1024)), (3, "bf16dev", (2048, 1024)),
                                               (2, "fp64", (512, 512))])
def test_a_monitored_step_allocates_nothing(fm, n, precision, shape):
    # the first lattice loads every kernel of the run; 16 MB and more in question for the second
    first, second = (_lattice(fm, n, *shape, precision) for _ in range(2))
    _monitored(fm, first, n)
    before = _free()
    _monitored(fm, second, n)
    assert _free() == before
    first.close()
    second.close()


@pytest.mark.parametrize("n,precision,shape", [(2, "fp64", (1024, 1024)), (3, "bf16dev_lnf64", (2048, 1024)),
                                               (2, "fp32", (4096, 2048)), (3, "fp16dev", (3000, 2001)),
                                               (2, "fp32", (512, 512))])
def test_lattice_bytes_cover_what_a_handle_holds(fm, n, precision, shape):
    _lattice(fm, n, *shape, precision).close()   # loads the kernels
    nbytes = fm.fmlbm_lattice_bytes(n, fm.make_lattice(*shape, 0.9, precision=precision))
    before = _free()
    lat = _lattice(fm, n, *shape, precision)
    # ten allocations, each rounded up to 2 MiB
    assert before - _free() <= nbytes + 10 * (2 << 20)
    lat.close()


def test_a_server_admits_by_what_its_batch_holds(fm):
    # FP64: a handle's eight scratch planes per node are no part of a served lattice
    L = fm.make_lattice(64, 64, 1.0, precision="fp64")
    rho = np.stack([np.full((64, 64), 1.0), np.full((64, 64), 0.8)])
    need = fm.fmlbm_lattice_bytes(2, L) - 8 * 8 * 64 * 64
    mix = fm.mixture_from_dict(mixture_dict(2, Tr=1.1, kappa_scale=0.5))
    for budget, accepted in ((need, True), (need - 1, False)):
        s = fm.fmlbm_server_create(2, "fp64", 2, 100, 1e-12, 1000, budget)
        if accepted:
            fm.fmlbm_server_submit(s, mix, L, rho)
        else:
            with pytest.raises(fm.FmlbmError):
                fm.fmlbm_server_submit(s, mix, L, rho)
        fm.fmlbm_server_destroy(s)


@pytest.mark.parametrize("n,precision,shape", [(2, "fp32", (4096, 2048)), (2, "fp64", (2048, 1024))])
def test_a_lattice_without_room_for_its_scratch_steps_all_the_same(fm, n, precision, shape):
    # device memory for all that the lattice needs, not for its second snapshot or scratch planes as well
    import torch
    mix = fm.mixture_from_dict(mixture_dict(n, Tr=0.9, kappa_scale=0.3))
    pinned = torch.from_numpy(smooth_state(n, *shape, seed=4)).pin_memory()   # read in place: no device copy
    out = []
    for short in (False, True):
        filler = None
        if short:
            L = fm.make_lattice(*shape, 0.9, precision=precision)
            scratch = (3 * n + 2) * 8 if precision == "fp64" else n * 4
            need = fm.fmlbm_lattice_bytes(n, L) - scratch * shape[0] * shape[1] + 10 * (2 << 20)
            torch.cuda.empty_cache()
            filler = torch.empty(_free() - need - (16 << 20), dtype=torch.uint8, device="cuda")
        lat = fm.Lattice(mix, *shape, 0.9, precision=precision)
        lat.init(pinned.numpy())
        rows = fm.fmlbm_step_diagnostics(lat.h, 3, n)
        del filler
        torch.cuda.empty_cache()
        out.append(tuple(rows) + lat.distributions())
        lat.close()
    assert all(np.array_equal(u, v) for u, v in zip(*out))


@pytest.mark.parametrize("n,precision,shape", [(2, "fp64", (2048, 2048)), (2, "fp32", (4096, 4096))])
def test_the_slabs_of_a_lattice_share_their_scratch(fm, n, precision, shape):
    # four slabs: what they need, the scratch planes of one (FP64), and no second snapshot of any
    nx, ny = shape
    mix = fm.mixture_from_dict(mixture_dict(n, Tr=0.9, kappa_scale=0.3))
    local = fm.make_lattice(nx, ny // 4 + 6, 0.9, precision=precision)
    scratch = ((3 * n + 2) * 8 if precision == "fp64" else n * 4) * nx * (ny // 4 + 6)
    need = 4 * (fm.fmlbm_lattice_bytes(n, local) - scratch) + (scratch if precision == "fp64" else 0)
    _lattice(fm, n, 64, 64, precision).close()
    before = _free()
    d = fm.Decomposition(mix, nx, ny, 0.9, 4, precision=precision)
    assert before - _free() <= need + 4 * 10 * (2 << 20)   # ten allocations a slab, rounded up to 2 MiB
    d.close()

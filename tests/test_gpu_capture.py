"""Steps captured into a graph and replayed between launched calls: the same state, diagnostics and
counts as stepping directly."""
import numpy as np
import pytest

from cases import mixture_dict, slab_state_binary, smooth_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fm():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2212_10680_gb300 import fmlbm
    return fmlbm


def _capture(stream, call):
    import torch
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        call()

    def replay(times=1):
        with torch.cuda.stream(stream):
            for _ in range(times):
                graph.replay()
        stream.synchronize()
    return replay


@pytest.mark.parametrize("precision,n,shape", [("fp32", 2, (1024, 512)), ("bf16dev", 3, (1024, 512)),
                                               ("fp32", 2, (300, 256)), ("fp64", 2, (70, 45))])
def test_requests_captured_and_launched_share_one_snapshot(fm, precision, n, shape):
    # every residual is taken against the state of the request before it, whether a replayed graph or a
    # launched step served that one (2^19 nodes: the marching step; then packed tiles and the split step)
    import torch
    nx, ny = shape
    mixd = mixture_dict(n, "pr", Tr=0.9, kappa_scale=0.3)
    rho = smooth_state(n, nx, ny, seed=3)

    def lattice(stream):
        lat = fm.Lattice(fm.mixture_from_dict(mixd), nx, ny, 0.9, "isotropic", precision, "lagged", stream=stream)
        lat.init(rho)
        fm.fmlbm_synchronize(lat.h)
        return lat

    ref, expect = lattice(0), []
    for _ in range(5):
        expect.append(ref.diagnostics()[:2])
        ref.step(2)
    s = torch.cuda.Stream()
    lat, got = lattice(s.cuda_stream), []

    def launched():
        t = fm.fmlbm_diagnostics_async(lat.h)
        lat.step(2)
        got.append(fm.fmlbm_diagnostics_wait(lat.h, t, n)[:2])
        fm.fmlbm_synchronize(lat.h)

    launched()
    ticket = fm.fmlbm_diagnostics_async(lat.h)
    replay = _capture(s, lambda: lat.step(2))

    def replayed():
        replay()
        got.append(fm.fmlbm_diagnostics_wait(lat.h, ticket, n)[:2])

    for serve in (replayed, launched, replayed, launched):
        serve()
    for k, ((mass, res), (mass_ref, res_ref)) in enumerate(zip(got, expect)):
        assert np.array_equal(mass, mass_ref) and res == res_ref, k
    for u, v in zip(lat.distributions(), ref.distributions()):
        assert np.array_equal(u, v)
    lat.close()
    ref.close()


def _batch(fm, stream, precision="fp32", shape=(70, 45)):
    mixd, rho = slab_state_binary(*shape, seed=3)
    L = fm.make_lattice(*shape, 1.0, precision=precision)
    b = fm.fmlbm_batch_create(2, precision, 3, stream.cuda_stream)
    return b, fm.fmlbm_batch_add(b, fm.mixture_from_dict(mixd), L, rho), (mixd, rho, precision)


def _after(fm, b, slot, case, steps):
    """Whether the slot's state, fields, phases and count are those of the same lattice after `steps` steps."""
    mixd, rho, precision = case
    n, ny, nx = rho.shape
    lat = fm.Lattice(fm.mixture_from_dict(mixd), nx, ny, 1.0, precision=precision)
    lat.init(rho)
    lat.step(steps)
    want = lat.distributions() + (lat.moments()[0],)
    lat.close()
    got = np.empty((n, 9, ny, nx)), np.empty((2, ny, nx)), np.empty((n, ny, nx))
    fm.fmlbm_batch_moments(b, slot, got[2])
    fm.fmlbm_batch_get_distributions(b, slot, *got[:2])
    liquid, vapour = fm.fmlbm_batch_phases(b, slot, n)
    return (all(np.array_equal(u, v) for u, v in zip(got, want)) and liquid.sum() > vapour.sum() and
            fm.fmlbm_batch_slot_info(b, slot)[0] == steps)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])   # packed tiles; the batch kernel alone
@pytest.mark.parametrize("rebuild", [False, True])
@pytest.mark.parametrize("replays", [0, 1, 2, 3])
def test_batch_counts_the_replays_of_captured_steps(fm, precision, rebuild, replays):
    import torch
    s = torch.cuda.Stream()
    b, slot, case = _batch(fm, s, precision)
    fm.fmlbm_batch_step(b, 1)
    s.synchronize()
    replay = _capture(s, lambda: fm.fmlbm_batch_step(b, 1))
    if rebuild:   # descriptors and counters are uploaded again
        fm.fmlbm_batch_set_active(b, slot, False)
        fm.fmlbm_batch_set_active(b, slot, True)
    fm.fmlbm_batch_step(b, 1)
    replay(replays)
    assert _after(fm, b, slot, case, 2 + replays)
    fm.fmlbm_batch_step(b, 1)
    replay()
    assert _after(fm, b, slot, case, 4 + replays)
    steps, _, _ = fm.fmlbm_batch_run(b, 3, max_steps=9 + replays, check_every=5, tol=0.0)
    assert steps[slot] == 9 + replays
    assert _after(fm, b, slot, case, 9 + replays)
    fm.fmlbm_batch_destroy(b)


@pytest.mark.parametrize("call", ["chunk", "run"])
def test_batch_runs_are_refused_under_capture_and_leave_no_trace(fm, call):
    import torch
    s = torch.cuda.Stream()
    b, slot, case = _batch(fm, s)
    fm.fmlbm_batch_step(b, 2)
    s.synchronize()

    def refused():
        with pytest.raises(fm.FmlbmError) as e:
            if call == "chunk":
                fm.fmlbm_batch_run_chunk(b, 3)
            else:
                fm.fmlbm_batch_run(b, 3, max_steps=5, check_every=3, tol=0.0)
        assert e.value.status == 3   # FMLBM_E_CUDA
        fm.fmlbm_batch_step(b, 1)   # the capture goes on

    replay = _capture(s, refused)
    assert _after(fm, b, slot, case, 2)
    replay()
    assert _after(fm, b, slot, case, 3)
    fm.fmlbm_batch_destroy(b)

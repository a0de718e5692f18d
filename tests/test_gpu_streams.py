"""Streams and threads.  Calls given another stream than the current one: arrays that the call
allocates (and clears) on the current stream, and the imaging chains, whose
transforms torch.fft runs on the current stream, are ordered between the two.
The current stream is held up ahead of each call (a bounded device-side delay
of some 20 ms), so that a missing wait shows as a wrong result."""
import numpy as np
import pytest
import torch

import synthetic as syn
from paper_2111_04141_gb300 import imaging

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)
DELAY = 40_000_000          # clock cycles, about 20 ms


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_04141_gb300 import build as b
    b.build()
    import paper_2111_04141_gb300 as gw
    return gw


def case(gw, n_w=1, n=256):
    obs = syn.small_case(n_ant=8, n_times=20, n_chan=2, npol=2, grid_n=n, s_min=5, s_max=5,
                         n_w=n_w, diameter_m=1500.0, seed=51)
    t = [torch.from_numpy(a).to(DEV) for a in (obs.uvw_m, obs.freq_hz, obs.vis)]
    return gw.Plan.from_observation(obs), obs, *t


def close(got, want):
    """Equal up to the order of the FP32 sums, on the central half of an image
    (the correction multiplies rounding at its border)."""
    n = want.shape[-1]
    a, b = (x[..., n // 4:-(n // 4), n // 4:-(n // 4)] for x in (got, want))
    return float(torch.linalg.vector_norm(a - b)) <= 1e-5 * float(torch.linalg.vector_norm(b))


def stale(shape, dtype):
    """Leaves the allocator a block that pending work of the current stream
    still fills with NaN."""
    x = torch.empty(shape, dtype=dtype, device=DEV)
    torch.cuda._sleep(DELAY)
    x.fill_(float("nan"))


@pytest.mark.parametrize("call", ["grid", "grid_compressed", "grid_wstack", "hybrid_grid", "degrid",
                                  "degrid_static", "hybrid_prune", "hybrid_image", "index"])
def test_arrays_allocated_for_another_stream(gw, call):
    plan, obs, uvw, freq, vis = case(gw)
    side = torch.cuda.Stream()
    with plan:
        model = plan.grid(uvw, freq, vis)
        fine = plan.hybrid_grid(uvw, freq, vis, 9)
        pruned = plan.hybrid_prune(9, fine)
        run = {
            "grid": lambda s: plan.grid(uvw, freq, vis, stream=s),
            "grid_compressed": lambda s: plan.grid_compressed(uvw, freq, vis, stream=s)[0],
            "grid_wstack": lambda s: plan.grid_wstack(uvw, freq, vis, 3, -50.0, 50.0, stream=s),
            "hybrid_grid": lambda s: plan.hybrid_grid(uvw, freq, vis, 9, stream=s),
            "degrid": lambda s: plan.degrid(uvw, freq, model, stream=s),
            "degrid_static": lambda s: plan.degrid_static(uvw, freq, model, stream=s),
            "hybrid_prune": lambda s: plan.hybrid_prune(9, fine, stream=s),
            "hybrid_image": lambda s: plan.hybrid_image(9, pruned, stream=s),
            "index": lambda s: plan.index(uvw, freq, stream=s)[0],
        }[call]
        want = run(None)
        torch.cuda.synchronize()
        stale(want.shape, want.dtype if want.dtype != torch.int32 else torch.float32)
        got = run(side)
        torch.cuda.synchronize()
        if call == "index":
            assert torch.equal(got, want)
        else:
            assert torch.isfinite(torch.view_as_real(got)).all()
            assert torch.linalg.vector_norm(got - want) <= 1e-5 * torch.linalg.vector_norm(want)


@pytest.mark.parametrize("chain", ["dirty", "weighted", "wstack", "hybrid", "model_vis"])
def test_imaging_on_another_stream(gw, chain):
    plan, obs, uvw, freq, vis = case(gw)
    weight = torch.from_numpy(syn.random_weights(obs)).to(DEV)
    side = torch.cuda.Stream()
    with plan:
        sky = torch.zeros((2, 256, 256), device=DEV)
        sky[:, 100:150:7, 90:160:9] = 1.0
        run = {
            "dirty": lambda v, w, x, s: imaging.dirty_image(plan, uvw, freq, v, stream=s),
            "weighted": lambda v, w, x, s: imaging.dirty_image(plan, uvw, freq, v, w, stream=s),
            "wstack": lambda v, w, x, s: imaging.dirty_image_wstack(plan, uvw, freq, v, 3, -50.0, 50.0,
                                                                    stream=s),
            "hybrid": lambda v, w, x, s: imaging.dirty_image_hybrid(plan, uvw, freq, v, 9, stream=s),
            "model_vis": lambda v, w, x, s: imaging.model_vis(plan, uvw, freq, x, stream=s),
        }[chain]
        want = run(vis, weight, sky, None)
        torch.cuda.synchronize()
        for _ in range(3):
            torch.cuda._sleep(DELAY)                 # the inputs are late on the current stream
            late = [t * 1.0 for t in (vis, weight, sky)]
            got = run(*late, side)
            del late                                 # their memory may be used again at once
            filler = [torch.full_like(t, float("nan")) for t in (vis, weight, sky)]
            got = got * 1.0                          # used without another wait
            torch.cuda.synchronize()
            del filler
            if chain == "model_vis":
                assert torch.linalg.vector_norm(got - want) <= 1e-6 * torch.linalg.vector_norm(want)
            else:
                assert close(got, want)


def test_threads_with_plans_of_different_sizes(gw):
    """Threads, each with its plan and stream, launch the same kernels with
    different amounts of shared memory: no launch may be refused."""
    import threading
    plans, failures = [], []
    for smax, n in ((5, 64), (71, 700), (5, 64), (71, 700)):
        obs = syn.small_case(n_ant=6, n_times=8, n_chan=1, npol=2, grid_n=n, s_min=5, s_max=smax,
                             n_w=3, beta=2, diameter_m=1500.0, seed=53)
        uvw, freq, vis = (torch.from_numpy(a).to(DEV) for a in (obs.uvw_m, obs.freq_hz, obs.vis))
        plan = gw.Plan.from_observation(obs)
        plan.set_tuning(grid_kernel=1, degrid_kernel=1)
        plans.append((plan, uvw, freq, vis, plan.grid(uvw, freq, vis)))
    torch.cuda.synchronize()

    def work(plan, uvw, freq, vis, model):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                first = plan.degrid(uvw, freq, model)
                for _ in range(1500):
                    v = plan.degrid(uvw, freq, model)
                torch.cuda.current_stream().synchronize()
                assert torch.linalg.vector_norm(v - first) <= 1e-5 * torch.linalg.vector_norm(first)
        except Exception as e:                       # reported by the main thread
            failures.append(e)

    threads = [threading.Thread(target=work, args=p) for p in plans]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for p in plans:
        p[0].close()
    assert not failures, failures

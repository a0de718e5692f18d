"""The choices a gridding call makes by its size (direct or binned, records per
work item) cost no accuracy against the binned gridder with long work items,
also where the visibilities are concentrated in a few tiles or on a few pixels
and where they are coherent (a source at the phase centre), so that the partial
sums grow with every one of them.

Errors are relative L2 against the FP64 oracle.  They are FP32 roundings in an
order that differs from run to run, so each is a mean of eight runs; where few
grid points carry the norm these scatter by a tenth and more, which counts with
three times the standard error of the difference.  A bin of short items adds to
the grid up to eight times where long ones add twice; six more roundings, each
about 0.4 of FP32's unit roundoff of a part of the total, are 3.4e-8 in
quadrature, on errors of 9e-8 and more 7 %.  So a call may show 1.1 times the error
of the long items plus 1e-8, beside the scatter."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.cgrid import Oracle
from oracle.wkernel import Params

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_04141_gb300 import build as b
    b.build()
    import paper_2111_04141_gb300 as gw
    return gw


def check(gw, scale, coherent, **kw):
    obs = syn.small_case(diameter_m=8.0 * kw["grid_n"], seed=61, **kw)
    obs.uvw_m[:, :2] *= scale
    if coherent:
        obs.vis[:] = 1.0 - 0.5j
    ref = Oracle(Params(**obs.plan_kwargs())).grid(obs.uvw_m, obs.freq_hz, obs.vis)
    uvw, freq, vis = (torch.from_numpy(a).to(DEV) for a in (obs.uvw_m, obs.freq_hz, obs.vis))

    def err(**tuning):
        plan.set_tuning(**tuning)
        e = [np.linalg.norm(plan.grid(uvw, freq, vis).cpu().numpy() - ref) for _ in range(8)]
        e = np.array(e) / np.linalg.norm(ref)
        return float(e.mean()), float(e.var(ddof=1) / e.size)

    with gw.Plan.from_observation(obs) as plan:
        (auto, va), (long, vl) = err(), err(grid_kernel=1, item_max=1024)
    print(f"auto {auto:.3e} long {long:.3e} scatter {np.sqrt(va + vl):.1e}")
    assert auto <= 1.1 * long + 1e-8 + 3 * np.sqrt(va + vl), (auto, long, va, vl)


# 16,080 visibilities, just below the most that are gridded directly, of supports
# beyond the limit on taps (2^22: 15 is within it)
@pytest.mark.parametrize("coherent", [False, True])
@pytest.mark.parametrize("scale", [1.0, 0.1, 0.01])
@pytest.mark.parametrize("npol,smin,smax", [(1, 17, 17), (1, 7, 33), (3, 31, 31)])
def test_direct_or_binned(gw, npol, smin, smax, scale, coherent):
    check(gw, scale, coherent, n_ant=16, n_times=134, n_chan=1, npol=npol, grid_n=1024, s_min=smin,
          s_max=smax, n_w=1 if smin == 17 else 8)


# calls that take items of 255 records (48 k) and of 510 (below 1.24 M pairs of a
# record and a tile on 152 SMs), spread over the grid, in a hundredth of its area
# (bins beyond eight such items) and on a few pixels
@pytest.mark.parametrize("coherent", [False, True])
@pytest.mark.parametrize("scale", [1.0, 0.1, 0.01])
@pytest.mark.parametrize("n_ant,n_times,npol,n,smin,smax", [
    (16, 100, 1, 512, 7, 31), (16, 250, 4, 256, 7, 9), (24, 300, 2, 512, 7, 21)])
def test_items_of_small_calls(gw, n_ant, n_times, npol, n, smin, smax, scale, coherent):
    check(gw, scale, coherent, n_ant=n_ant, n_times=n_times, n_chan=4, npol=npol, grid_n=n,
          s_min=smin, s_max=smax, n_w=8)

"""The choices a gridding call makes by its size (direct or binned, records per
work item) cost no accuracy against the binned gridder with long work items,
also where the visibilities are concentrated in a few tiles or on a few pixels
and where they are coherent (a source at the phase centre), so that the partial
sums grow with every one of them.

Errors are relative L2 against the FP64 oracle.  They are FP32 roundings in an
order that differs from run to run (repeats lie within some 3 %), so a call may
show 1.1 times the error of the long items plus 1e-8, a sixth of FP32's unit
roundoff."""
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
        e = [np.linalg.norm(plan.grid(uvw, freq, vis).cpu().numpy() - ref) for _ in range(3)]
        return float(np.mean(e) / np.linalg.norm(ref))

    with gw.Plan.from_observation(obs) as plan:
        auto, binned = err(), err(grid_kernel=1, item_max=1024)
    assert auto <= 1.1 * binned + 1e-8, (auto, binned)


# 16,080 visibilities, just below the most that are gridded directly, of supports
# beyond the limit on taps (2^22: 15 is within it)
@pytest.mark.parametrize("coherent", [False, True])
@pytest.mark.parametrize("scale", [1.0, 0.1, 0.01])
@pytest.mark.parametrize("npol,smin,smax", [(1, 17, 17), (1, 7, 33), (3, 31, 31)])
def test_direct_or_binned(gw, npol, smin, smax, scale, coherent):
    check(gw, scale, coherent, n_ant=16, n_times=134, n_chan=1, npol=npol, grid_n=1024, s_min=smin,
          s_max=smax, n_w=1 if smin == 17 else 8)

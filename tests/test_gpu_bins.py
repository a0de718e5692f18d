"""Bins counted by the index stage (into shared histograms or the bins'
counters) and by the binner, at the sizes where that changes: every bin holds
exactly the records that meet its tile (whole numbers: no tolerance)."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.index import index_vis
from oracle.wkernel import Params, plane_support

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


# records and bins: 76,000 over 128 (shared, several records a thread), 30,400
# over 512 (shared, few CTAs), 152,000, 30,400 (with footprints 19 pairs a bin,
# shared; with centres 7), 15,200 (10 and 4, the bins' counters) and 7,600 over
# 2,048 or 4,096, channels past the cached factors, and more bins than one kernel
# scans and scatters (8,192), with centres more than 16,384
@pytest.mark.parametrize("n,n_ant,n_times,n_chan,n_w", [
    (512, 20, 100, 4, 5), (1024, 20, 40, 4, 1), (2048, 20, 200, 4, 3), (2048, 20, 40, 4, 3),
    (2048, 20, 20, 4, 3), (2048, 20, 10, 4, 7), (512, 4, 3, 1500, 2), (4222, 20, 700, 4, 3)])
@pytest.mark.parametrize("mode", [0, 1])
def test_every_bin_holds_its_records(gw, n, n_ant, n_times, n_chan, n_w, mode):
    obs = syn.small_case(n_ant=n_ant, n_times=n_times, n_chan=n_chan, npol=1, grid_n=n, s_min=5,
                         s_max=15 if n_w > 1 else 5, n_w=n_w, beta=4, diameter_m=40.0 * n, seed=41)
    obs.uvw_m[::7] *= 1.5                                # some leave the grid
    prm = Params(**obs.plan_kwargs())
    ref = index_vis(obs.uvw_m, obs.freq_hz, prm)
    with gw.Plan.from_observation(obs) as plan:
        info = plan.info
        offs, ent = plan.debug_bins(torch.from_numpy(obs.uvw_m).to(DEV),
                                    torch.from_numpy(obs.freq_hz).to(DEV), mode=mode)
        work = plan.timing()
    tu, tv = (info.grid_tile_u, info.grid_tile_v) if mode == 0 else (info.degrid_tile,) * 2
    ntu, ntv = -(-n // tu), -(-n // tv)
    i = np.flatnonzero(ref["valid"])
    S = plane_support(prm)[ref["plane"][i]]
    h = S // 2 if mode == 0 else 0 * S
    ku, kv = ref["ku"][i].astype(np.int64), ref["kv"][i].astype(np.int64)
    u0, u1, v0, v1 = (ku - h) // tu, (ku + h) // tu, (kv - h) // tv, (kv + h) // tv
    pairs = [np.stack([(v0 + b) * ntu + u0 + a, i], 1)[(u0 + a <= u1) & (v0 + b <= v1)]
             for a in range(3) for b in range(3)]
    want = np.concatenate(pairs)
    want = want[np.lexsort((want[:, 1], want[:, 0]))]
    got = np.stack([np.repeat(np.arange(ntu * ntv), np.diff(offs)), np.asarray(ent[:offs[-1]])], 1)
    got = got[np.lexsort((got[:, 1], got[:, 0]))]
    assert np.array_equal(got, want)
    assert work["valid_vis"] == len(i) and work["taps"] == int(np.sum(S.astype(np.int64) ** 2))

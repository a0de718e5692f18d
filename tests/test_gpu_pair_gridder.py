"""The gridders over pair tables (16-bit tensor cores; FP32 with one or two
polarisations) at the edges of their tiles, blocks, groups and supports:
against the FP64 oracle run on exactly the stored values (the products of
16-bit values are exact in FP32, so only FP32 sums differ: relative L2 <= 1e-5,
the tolerance of every FP32 grid)."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.cgrid import Oracle
from oracle.precision import QuantisedTables
from oracle.wkernel import KernelTables, Params
from paper_2111_04141_gb300.plan import from_storage, to_storage

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)
TOL = 1e-5


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_04141_gb300 import build as b
    b.build()
    import paper_2111_04141_gb300 as gw
    return gw


def case(kind, npol, n, smin, smax, n_w, beta=8, n_times=10):
    obs = syn.small_case(n_ant=6, n_times=n_times, n_chan=3, npol=npol, grid_n=n, s_min=smin,
                         s_max=smax, n_w=n_w, beta=beta, diameter_m=1100.0, seed=21)
    prm = Params(**obs.plan_kwargs())
    vis = to_storage(torch.from_numpy(obs.vis), kind)
    held = from_storage(vis).numpy().astype(np.complex128)
    kt = KernelTables(prm)
    ref = Oracle(prm, kt if kind == "c64" else QuantisedTables(kt, kind)).grid(
        obs.uvw_m, obs.freq_hz, held)
    return obs, vis.to(DEV), ref


# grid sides off every tile and block multiple, supports from one tap to wider
# than a tile, every polarisation count, oversampling that is no power of two
@pytest.mark.parametrize("kind,npol,n,smin,smax,n_w,beta", [
    ("bf16", 1, 66, 1, 1, 1, 8), ("f16", 2, 98, 3, 5, 2, 6), ("bf16", 3, 130, 7, 15, 4, 8),
    ("f16", 4, 142, 5, 33, 3, 4), ("bf16", 4, 254, 15, 79, 5, 4), ("f16", 1, 190, 7, 65, 3, 2),
    ("c64", 1, 66, 1, 3, 2, 8), ("c64", 2, 98, 3, 5, 2, 6), ("c64", 1, 142, 5, 33, 3, 4),
    ("c64", 2, 254, 15, 79, 5, 4), ("c64", 1, 600, 41, 255, 3, 2)])
def test_grid_matches_oracle_on_stored_values(gw, kind, npol, n, smin, smax, n_w, beta):
    obs, vis, ref = case(kind, npol, n, smin, smax, n_w, beta)
    uvw, freq = torch.from_numpy(obs.uvw_m).to(DEV), torch.from_numpy(obs.freq_hz).to(DEV)
    with gw.Plan.from_observation(obs, table_dtype=kind, vis_dtype=kind) as plan:
        plan.set_tuning(grid_kernel=1)
        err = torch.zeros((npol, n, n), dtype=torch.complex64, device=DEV)
        comp = plan.grid(uvw, freq, vis, err=err)            # compensated commits
        plan.fold(comp, err)
        c = comp.cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(c - ref) / np.linalg.norm(ref) <= TOL
        # a buffer whose visibilities start one element (4 bytes) off, and a
        # grid on an odd 8-byte boundary: the narrow copies and commits
        # (FP32 pairs of polarisations have to start on 16 bytes)
        skip = 2 if kind != "c64" else int(npol == 1)
        buf = torch.empty(vis.numel() + skip, dtype=vis.dtype, device=DEV)
        odd = buf[skip:].view(vis.shape)
        odd.copy_(vis)
        room = torch.zeros(plan.npol * n * n + 1, dtype=torch.complex64, device=DEV)
        off = room[1:].view(plan.npol, n, n)
        for v, out in ((vis, None), (odd, None), (vis, off)):
            g = plan.grid(uvw, freq, v, out=out).cpu().numpy().astype(np.complex128)
            err = np.linalg.norm(g - ref) / np.linalg.norm(ref)
            assert err <= TOL, err
        plan.device_status()


def test_infinite_visibility_stays_near_its_footprint(gw):
    obs, vis, ref = case("bf16", 2, 256, 7, 7, 1, n_times=4)
    prm = Params(**obs.plan_kwargs())
    idx = Oracle(prm).index(obs.uvw_m, obs.freq_hz)
    i = int(np.flatnonzero(idx["valid"])[0])
    vis.view(-1, 2, 2)[i, 1, 0] = float("inf")
    uvw, freq = torch.from_numpy(obs.uvw_m).to(DEV), torch.from_numpy(obs.freq_hz).to(DEV)
    with gw.Plan.from_observation(obs, table_dtype="bf16", vis_dtype="bf16") as plan:
        plan.set_tuning(grid_kernel=1)
        g = plan.grid(uvw, freq, vis).cpu().numpy()
    ku, kv = int(idx["ku"][i]), int(idx["kv"][i])
    assert np.isfinite(g[0]).all()                      # the other polarisation
    assert not np.isfinite(g[1, kv, ku])
    far = np.ones((256, 256), dtype=bool)               # beyond the blocks it meets
    far[max(0, kv - 11):kv + 12, max(0, ku - 19):ku + 20] = False
    d = np.abs(g[1] - ref[1])[far]
    assert d.max() <= TOL * np.linalg.norm(ref[1])

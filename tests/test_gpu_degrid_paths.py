"""The degridder's paths at the sizes where they change: direct (small calls),
staged regions in one piece, staged regions in bands of rows (wide supports),
items longer than one chunk, and 16 x 16 against 32 x 32 centre tiles.  FP32
results against the FP64 oracle: relative L2 <= 1e-5, the tolerance of every
FP32 degridded visibility."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.cgrid import Oracle
from oracle.wkernel import Params

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


def degrid(gw, obs, grid, bands, **tuning):
    uvw, freq = torch.from_numpy(obs.uvw_m).to(DEV), torch.from_numpy(obs.freq_hz).to(DEV)
    g = torch.from_numpy(grid).to(DEV)
    with gw.Plan.from_observation(obs) as plan:
        plan.set_tuning(**tuning)
        # no stale value may survive, dropped visibilities read zero
        out = torch.full((obs.nrow, obs.nchan, obs.npol), float("nan"), dtype=torch.complex64, device=DEV)
        v, dropped = plan.degrid(uvw, freq, g, out=out, return_dropped=True)
        again = plan.degrid(uvw, freq, g)
        work = plan.timing()
    if not bands:
        assert torch.equal(v, again)                # sums in a fixed order
    else:
        # bands cut a record's sum where the item's region puts them, and the
        # order of a bin is free: each run is within the FP32 bound of check()
        assert torch.linalg.vector_norm(v - again) <= 2 * TOL * torch.linalg.vector_norm(v)
    return v.cpu().numpy().astype(np.complex128), dropped, work


def check(gw, obs, bands=False, **tuning):
    prm = Params(**obs.plan_kwargs())
    orc = Oracle(prm)
    rng = np.random.default_rng(3)
    shape = (obs.npol, obs.grid_n, obs.grid_n)
    grid = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(np.complex64)
    ref = orc.degrid(obs.uvw_m, obs.freq_hz, grid.astype(np.complex128))
    idx = orc.index(obs.uvw_m, obs.freq_hz)
    v, dropped, work = degrid(gw, obs, grid, bands, **tuning)
    v = v.reshape(ref.shape)
    assert np.linalg.norm(v - ref) / np.linalg.norm(ref) <= TOL
    assert dropped == int(np.sum(~idx["valid"]))
    assert np.all(v.reshape(-1, obs.npol)[~idx["valid"].reshape(-1)] == 0)
    assert work["valid_vis"] == 2 * int(np.sum(idx["valid"]))


def drop_some(obs):
    obs.uvw_m[::5] *= 1.4                           # off the grid at the upper channels
    return obs


@pytest.mark.parametrize("npol,n,smin,smax,n_w,beta", [
    (1, 66, 1, 1, 1, 8), (2, 98, 3, 5, 2, 6), (3, 130, 7, 15, 4, 8), (4, 142, 5, 33, 3, 4)])
@pytest.mark.parametrize("kernel", [0, 1, 2])
def test_direct_staged_and_gather(gw, npol, n, smin, smax, n_w, beta, kernel):
    obs = syn.small_case(n_ant=6, n_times=10, n_chan=3, npol=npol, grid_n=n, s_min=smin, s_max=smax,
                         n_w=n_w, beta=beta, diameter_m=1100.0, seed=23)
    check(gw, drop_some(obs), degrid_kernel=kernel)


# regions of several bands: 16 + 2 h (or 32 + 2 h) rows of 8 npol bytes a point
# beyond about 190 KB, down to bands of a few rows
@pytest.mark.parametrize("npol,n,smin,smax,n_w", [
    (4, 256, 15, 71, 4), (4, 400, 31, 127, 3), (3, 300, 9, 101, 4), (1, 600, 41, 255, 3)])
def test_regions_in_bands(gw, npol, n, smin, smax, n_w):
    obs = syn.small_case(n_ant=6, n_times=8, n_chan=2, npol=npol, grid_n=n, s_min=smin, s_max=smax,
                         n_w=n_w, beta=2, diameter_m=1000.0, seed=29)
    check(gw, obs, bands=True, degrid_kernel=1)


# the global gather at supports of several warps' widths
@pytest.mark.parametrize("npol,n,smin,smax,n_w", [(4, 400, 31, 127, 3), (2, 600, 41, 255, 3)])
def test_gather_of_wide_supports(gw, npol, n, smin, smax, n_w):
    obs = syn.small_case(n_ant=6, n_times=8, n_chan=2, npol=npol, grid_n=n, s_min=smin, s_max=smax,
                         n_w=n_w, beta=2, diameter_m=1000.0, seed=29)
    check(gw, drop_some(obs), degrid_kernel=2)


# thousands of records centred in a few tiles (dense: 16 x 16 tiles), with
# items of one chunk and of several
@pytest.mark.parametrize("smax", [9, 71])
@pytest.mark.parametrize("item_max", [0, 4096])
def test_dense_tiles_and_long_items(gw, smax, item_max):
    obs = syn.small_case(n_ant=10, n_times=100, n_chan=3, npol=4, grid_n=160, s_min=7, s_max=smax,
                         n_w=3, beta=4, diameter_m=1000.0, seed=31)
    obs.uvw_m[:, :2] *= 0.06
    check(gw, obs, bands=smax == 71, degrid_kernel=1, item_max=item_max)


# large grids with few records: centre tiles of 64 x 64 (17 k on 2900^2) and of
# 128 x 128 points, the last tile of a row cut off, in one piece and in bands
@pytest.mark.parametrize("npol,n,n_ant,n_times,smin,smax", [
    (1, 2900, 20, 30, 3, 17), (2, 2900, 20, 30, 5, 41), (1, 5830, 6, 9, 1, 9), (1, 5830, 6, 9, 9, 127)])
def test_sparse_inputs_take_large_tiles(gw, npol, n, n_ant, n_times, smin, smax):
    obs = syn.small_case(n_ant=n_ant, n_times=n_times, n_chan=3, npol=npol, grid_n=n, s_min=smin,
                         s_max=smax, n_w=3, beta=4, diameter_m=20.0 * n, seed=37)
    check(gw, obs, bands=smax > 17, degrid_kernel=1)


# wide supports, whose regions are served in bands: few visibilities take the
# direct kernel (here up to 8,192), and concentrated ones short items
@pytest.mark.parametrize("scale", [1.0, 0.1])
@pytest.mark.parametrize("n_times,n", [(96, 400), (272, 400), (274, 400), (100, 1600)])
def test_few_visibilities_of_wide_supports(gw, n_times, n, scale):
    obs = syn.small_case(n_ant=6, n_times=n_times, n_chan=2, npol=4, grid_n=n, s_min=9, s_max=101,
                         n_w=4, beta=2, diameter_m=2.5 * n, seed=33)
    obs.uvw_m[:, :2] *= scale
    check(gw, drop_some(obs), bands=True)


# a row count on the device: rows beyond it stay as they were, whichever kernel
# serves the count (the gather below 8,192 visibilities or more)
@pytest.mark.parametrize("npol,smin,smax", [(4, 9, 101), (4, 7, 33), (1, 5, 5)])
def test_device_counts(gw, npol, smin, smax):
    obs = syn.small_case(n_ant=10, n_times=110, n_chan=2, npol=npol, grid_n=500, s_min=smin, s_max=smax,
                         n_w=4, beta=2, diameter_m=1200.0, seed=35)
    prm = Params(**obs.plan_kwargs())
    rng = np.random.default_rng(3)
    shape = (npol, 500, 500)
    grid = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(np.complex64)
    ref = Oracle(prm).degrid(obs.uvw_m, obs.freq_hz, grid.astype(np.complex128))
    ref = ref.reshape(obs.nrow, obs.nchan, npol)
    uvw, freq = torch.from_numpy(obs.uvw_m).to(DEV), torch.from_numpy(obs.freq_hz).to(DEV)
    g = torch.from_numpy(grid).to(DEV)
    with gw.Plan.from_observation(obs) as plan:
        for rows in (0, 1, 100, 4095, 4096, obs.nrow, obs.nrow + 7):     # (at most all)
            out = torch.full(ref.shape, 7.0, dtype=torch.complex64, device=DEV)
            plan.degrid_devcount(uvw, freq, torch.tensor([rows], dtype=torch.int64, device=DEV), g, out)
            plan.device_status()
            v = out.cpu().numpy().astype(np.complex128)
            assert np.all(v[rows:] == 7.0)
            assert np.linalg.norm(v[:rows] - ref[:rows]) <= TOL * np.linalg.norm(ref[:rows])


# one launch for small calls against the staged kernel, both over a warp's
# flattened taps, at supports around its 32 lanes and every polarisation count.
# They fold the lanes' sums alike except for 3 polarisations and where bands cut
# a sum: a few roundings of 2^-24, 3e-7 of the root mean square
@pytest.mark.parametrize("npol,n,smin,smax,n_w", [
    (1, 130, 1, 1, 1), (2, 98, 5, 7, 2), (3, 142, 31, 33, 3), (4, 300, 5, 65, 4), (1, 600, 41, 255, 3)])
def test_direct_equals_staged(gw, npol, n, smin, smax, n_w):
    obs = drop_some(syn.small_case(n_ant=6, n_times=9, n_chan=3, npol=npol, grid_n=n, s_min=smin,
                                   s_max=smax, n_w=n_w, beta=4, diameter_m=1100.0, seed=43))
    rng = np.random.default_rng(5)
    shape = (npol, n, n)
    grid = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(np.complex64)
    direct, dropped, _ = degrid(gw, obs, grid, True, degrid_kernel=0)
    staged, again, _ = degrid(gw, obs, grid, True, degrid_kernel=1)
    assert dropped == again
    assert np.linalg.norm(direct - staged) <= 3e-7 * np.linalg.norm(staged)

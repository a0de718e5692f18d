"""Imaging pipeline on the GPU (imaging.py): dirty image and model
visibilities against the oracle, and the aliasing experiment R(X) of
Section 8 for X = 0..63 on a 128^2 image against the oracle's R(X).

Tolerances: before correction the GPU image (FP32 gridding and cuFFT) and
the oracle's (FP64) agree at every pixel (X, X) to 2e-6 of the image peak:
FP32 rounding, the same at the field edge as at the centre.  The correction
multiplies that difference by h(l_X) h(m_X), so the corrected values R(X)
agree within 2e-6 peak h(l_X)^2 (peak: the uncorrected image at the centre,
about 1 / h(0)^2)."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.cgrid import Oracle
from oracle.image import centred_dft, centred_idft, correct, point_source_vis
from oracle.wkernel import Params, corrector

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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def test_rx_matches_oracle(gw):
    from paper_2111_04141_gb300.imaging import dirty_image
    N = 128
    obs = syn.config_2d()
    prm = Params(grid_n=N, cell_rad=syn.fit_cell(obs.uvw_m, obs.freq_hz, N, 7), support_min=7,
                 support_max=7, oversample=128, n_wplanes=1, w_max_lambda=0.0, npol=1)
    orc = Oracle(prm)
    h = corrector(prm)
    idx = orc.index(obs.uvw_m, obs.freq_hz)
    nv = int(idx["valid"].sum())
    r_gpu, r_orc, raw_gpu, raw_orc = [], [], [], []
    with gw.Plan(grid_n=N, cell_rad=prm.cell_rad, support_min=7, support_max=7, oversample=128,
                 n_wplanes=1, w_max_lambda=0.0, npol=1) as plan:
        u, f = dev(obs.uvw_m), dev(obs.freq_hz)
        for x in range(64):
            v = point_source_vis(obs.uvw_m, obs.freq_hz, prm, x, x)
            vd = dev(v.reshape(obs.nrow, obs.nchan, 1).astype(np.complex64))
            img = dirty_image(plan, u, f, vd)
            r_gpu.append(abs(1.0 - float(img[0, N // 2 + x, N // 2 + x].real)))
            # the same transform without the correction step
            g = plan.grid(u, f, vd)
            plan.shift(g)
            raw = torch.fft.ifft2(g, norm="forward") / nv
            raw_gpu.append(complex(raw[0, N // 2 + x, N // 2 + x].item()))
            ref_raw = centred_idft(orc.grid(obs.uvw_m, obs.freq_hz, v, idx=idx)) / nv
            raw_orc.append(complex(ref_raw[0, N // 2 + x, N // 2 + x]))
            ref = correct(ref_raw, h)
            r_orc.append(abs(1.0 - ref[0, N // 2 + x, N // 2 + x].real))
    r_gpu, r_orc = np.array(r_gpu), np.array(r_orc)
    raw_gpu, raw_orc = np.array(raw_gpu), np.array(raw_orc)
    hx = h[N // 2 + np.arange(64)]
    peak = abs(raw_orc[0])
    print("R(X) gpu max central half %.3g, all %.3g; oracle %.3g, %.3g; raw max |diff| %.3g"
          " of the peak" % (r_gpu[:33].max(), r_gpu.max(), r_orc[:33].max(), r_orc.max(),
                             np.abs(raw_gpu - raw_orc).max() / peak))
    # the uncorrected transform agrees to FP32 rounding at every X, edge included
    assert np.all(np.abs(raw_gpu - raw_orc) <= 2e-6 * peak)
    # the corrected values differ by that, times the corrector
    assert np.all(np.abs(r_gpu - r_orc) <= 2e-6 * peak * hx ** 2 + 1e-7)


def test_dirty_image_and_model_vis_match_oracle(gw):
    from paper_2111_04141_gb300.imaging import dirty_image, model_vis
    obs = syn.small_case(n_ant=7, n_times=10, n_chan=3, npol=4, grid_n=128, s_min=7,
                         s_max=21, n_w=5, diameter_m=1500.0)
    prm = Params(**obs.plan_kwargs())
    orc = Oracle(prm)
    h = corrector(prm)
    N = prm.grid_n
    wt = syn.random_weights(obs)
    idx = orc.index(obs.uvw_m, obs.freq_hz)
    valid = idx["valid"]
    ref = correct(centred_idft(orc.grid(obs.uvw_m, obs.freq_hz, obs.vis, weight=wt)), h)
    ref = ref / wt.reshape(-1, prm.npol)[valid].sum(0)[:, None, None]
    rng = np.random.default_rng(2)
    model = np.zeros((prm.npol, N, N), dtype=np.complex64)
    c = slice(N // 4, 3 * N // 4)
    model[:, c, c] = (rng.normal(size=(prm.npol, N // 2, N // 2))).astype(np.complex64)
    ref_v = orc.degrid(obs.uvw_m, obs.freq_hz, centred_dft(correct(model.astype(np.complex128), h)))
    with gw.Plan.from_observation(obs) as plan:
        u, f = dev(obs.uvw_m), dev(obs.freq_hz)
        img = dirty_image(plan, u, f, dev(obs.vis), weight=dev(wt)).cpu().numpy()
        mv = model_vis(plan, u, f, dev(model)).cpu().numpy().reshape(ref_v.shape)
    assert rel_l2(img[:, c, c], ref[:, c, c]) <= 2e-5
    assert rel_l2(mv, ref_v) <= 2e-5


# finish_image against shift + correct + divide in FP64: sides with whole and
# odd halves of 16 bytes (pairs of pixels or single ones), an image off 16
# bytes, host and device scales.  At most six FP32 roundings a
# pixel (factors, scale and products): 6 x 2^-24.
@pytest.mark.parametrize("n,npol,shift", [(8, 1, 0), (10, 3, 0), (130, 2, 0), (256, 4, 0),
                                          (256, 1, 1), (1030, 1, 1)])
@pytest.mark.parametrize("device_scale", [False, True])
def test_finish_is_shift_correct_and_scale(gw, n, npol, shift, device_scale):
    rng = np.random.default_rng(n + npol)
    z = (rng.standard_normal((npol, n, n)) + 1j * rng.standard_normal((npol, n, n)))
    z = z.astype(np.complex64)
    buf = torch.empty(npol * n * n + shift, dtype=torch.complex64, device=DEV)
    img = buf[shift:].view(npol, n, n)
    img.copy_(torch.from_numpy(z))
    scale_dev = dev(rng.uniform(0.5, 2.0, npol).astype(np.float32)) if device_scale else None
    with gw.Plan(grid_n=n, cell_rad=1e-3, support_min=1, support_max=3, oversample=4,
                 n_wplanes=1, w_max_lambda=0.0, npol=npol) as plan:
        ones = plan.correct(torch.ones_like(img), direction=+1).cpu().numpy().astype(complex)
        out = plan.finish_image(img, scale=0.37, scale_dev=scale_dev).cpu().numpy()
    # correct(+1) holds the sign; its FP32 factors are taken as given
    ref = np.roll(z.astype(complex), (n // 2, n // 2), (1, 2)) * ones * np.float32(0.37)
    if device_scale:
        ref *= scale_dev.cpu().numpy()[:, None, None].astype(float)
    assert np.all(np.abs(out - ref) <= 6 * 2.0 ** -24 * np.abs(ref) + 1e-30)


def test_dirty_image_without_weight_is_zero(gw):
    from paper_2111_04141_gb300.imaging import dirty_image
    obs = syn.config_2d()
    n = 128
    with gw.Plan(grid_n=n, cell_rad=syn.fit_cell(obs.uvw_m, obs.freq_hz, n, 7), support_min=7,
                 support_max=7, oversample=128, n_wplanes=1, w_max_lambda=0.0, npol=1) as plan:
        v = torch.ones((obs.nrow, obs.nchan, 1), dtype=torch.complex64, device=DEV)
        w = torch.zeros((obs.nrow, obs.nchan, 1), dtype=torch.float32, device=DEV)
        img = dirty_image(plan, dev(obs.uvw_m), dev(obs.freq_hz), v, weight=w)
    assert torch.count_nonzero(torch.view_as_real(img)) == 0

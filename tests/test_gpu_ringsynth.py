"""The single-precision ring synthesis (power-of-two grids; interpolation on the cap rings) at the
sizes where its rules change: belts shorter than the smallest grid (Nside 1 .. 64) and just
on it (128), band limits that fold aliases in the caps and in the belt (above 2 Nside, up to 8 Nside), odd band
limits, bands that fill the grid up to its Nyquist frequency, and the rings that take two interleaved grids
(Nside 2048). Derivative maps of Eq. 4 against the oracle's per-ring library FFT (Naess & Louis
2013, Sec. II.B), and the lensed maps of the interleaved rows of the tensor-core stage.

Tolerance: the recurrence's single precision sets the level, as in test_gpu_ringfft.py (5e-5 relative RMS
per map); the synthesis itself adds float rounding (1e-7). Where only the caps of a large
sphere are compared, the same bound per ring."""
import numpy as np
import pytest
import torch

import oracle.healpix as hp
import oracle.lens as OL
from gpu_util import rel_rms, sky, to_dev

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")
TOL = 5e-5


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("nside,lmax,order", [(1, 8, 2), (2, 3, 6), (4, 31, 3), (16, 100, 4), (32, 256, 2), (64, 127, 5),
                                              (64, 190, 3), (128, 255, 2), (128, 257, 2), (256, 1100, 1)])
def test_derivs_spin0_vs_oracle(nside, lmax, order):
    s = sky(nside, lmax, pol=False, seeds=(11, 0, 1))
    ref = OL.derivative_maps(nside, lmax, order, alm_T=s["T"])["T"]
    out = api.synth_derivs(nside, lmax, order, to_dev(s)["T"], 0, api.MIXED_FP32).cpu().numpy()
    for i in range(ref.shape[0]):
        assert rel_rms(out[i], ref[i]) < TOL, (i, rel_rms(out[i], ref[i]))


def test_spin2_below_its_lowest_l_is_zero():
    """lmax 1 holds no spin-2 harmonics."""
    s = sky(2, 1, pol=True, seeds=(11, 12, 1))
    d = to_dev(s)
    out = api.synth_derivs(2, 1, 2, torch.cat([d["E"], d["B"]]), 2, api.MIXED_FP32)
    assert torch.count_nonzero(out) == 0


@pytest.mark.parametrize("nside,lmax,order", [(2, 2, 2), (2, 16, 3), (32, 75, 4), (64, 200, 2), (128, 300, 1)])
def test_derivs_spin2_vs_oracle(nside, lmax, order):
    s = sky(nside, lmax, pol=True, seeds=(11, 12, 1), b_scale=0.6)
    ref = OL.derivative_maps(nside, lmax, order, alm_E=s["E"], alm_B=s["B"])
    d = to_dev(s)
    out = api.synth_derivs(nside, lmax, order, torch.cat([d["E"], d["B"]]), 2, api.MIXED_FP32).cpu().numpy()
    K = ref["Q"].shape[0]
    for i in range(K):
        for f, o in (("Q", out[i]), ("U", out[K + i])):
            assert rel_rms(o, ref[f][i]) < TOL, (f, i, rel_rms(o, ref[f][i]))


@pytest.mark.parametrize("lmax", [4096, 6001])
def test_outer_cap_rings_nside2048_vs_ring_fft(lmax):
    """Rings near the cap's edge, whose band needs the two interleaved grids, and their folded form (lmax
    above 2 Nside), at order 1: against the oracle's coefficients and library FFT, ring by ring."""
    import oracle.sht as sht
    nside, order = 2048, 1
    s = sky(nside, lmax, pol=False, seeds=(13, 0, 1), damp_t=400.0)
    tab = hp.ring_table(nside)
    rings = [1200, 1561, 1700, 2046, 2047, 4 * nside - 2 - 1900]
    F = sht.ring_coeffs(lmax, order, tab["theta"][rings], alm_T=s["T"])["T"]
    out = api.synth_derivs(nside, lmax, order, to_dev(s)["T"], 0, api.MIXED_FP32)
    jk = OL.derivative_pairs(order)
    for q, r in enumerate(rings):
        a, n = int(tab["first"][r]), int(tab["nphi"][r])
        ref = OL.ring_synthesis(F[q], n, float(tab["phi0"][r]), jk)
        got = out[:, a:a + n].cpu().numpy()
        for i in range(len(jk)):
            assert rel_rms(got[i], ref[i]) < TOL, (r, jk[i], rel_rms(got[i], ref[i]))


def test_lens_interleaved_rows_above_the_grid():
    """The tensor-core stage's four-ring interleaved rows with folded aliases (lmax 2.5 Nside)."""
    nside, lmax, order = 32, 81, 4
    s = sky(nside, lmax, b_scale=0.4)
    ref = OL.lens(nside, lmax, order, s["T"], s["E"], s["B"], s["phi"])
    d = to_dev(s)
    out = api.lens(nside, lmax, order, d["T"], d["E"], d["B"], d["phi"], precision=api.MIXED_BF16x3).cpu().numpy()
    for i, f in enumerate("TQU"):
        assert rel_rms(out[i], ref[f]) < 1e-4, (f, rel_rms(out[i], ref[f]))

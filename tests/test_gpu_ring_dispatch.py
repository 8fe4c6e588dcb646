"""Which kernel forms a ring in single precision (Naess & Louis 2013, Sec. II.B): the general ring FFT for every
ring (TAYLENS_RING_FFT=shared), cap rings longer than the grid their band needs, and above Nside 2048 plans whose
belt and outer cap rings go to the general ring FFT and the others to the grids. Derivative maps (Eq. 4)
against the oracle's coefficients and library FFT, ring by ring, to the level of the float recurrence
(5e-5 relative RMS, as in test_gpu_ringfft.py)."""
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


def _check(nside, lmax, order, rings, damp=100.0):
    import oracle.sht as sht
    s = sky(nside, lmax, pol=False, seeds=(13, 0, 1), damp_t=damp)
    tab = hp.ring_table(nside)
    F = sht.ring_coeffs(lmax, order, tab["theta"][rings], alm_T=s["T"])["T"]
    out = api.synth_derivs(nside, lmax, order, to_dev(s)["T"], 0, api.MIXED_FP32)
    jk = OL.derivative_pairs(order)
    for q, r in enumerate(rings):
        a, n = int(tab["first"][r]), int(tab["nphi"][r])
        ref = OL.ring_synthesis(F[q], n, float(tab["phi0"][r]), jk)
        got = out[:, a:a + n].cpu().numpy()
        for i in range(len(jk)):
            assert rel_rms(got[i], ref[i]) < TOL, (r, n, jk[i], rel_rms(got[i], ref[i]))


@pytest.mark.parametrize("nside,lmax,order", [(16, 100, 3), (128, 300, 4), (512, 1024, 2)])
def test_general_ring_fft_in_float(nside, lmax, order, monkeypatch):
    monkeypatch.setenv("TAYLENS_RING_FFT", "shared")
    rings = [2, nside // 3, nside // 2 - 1, nside - 2, nside, 2 * nside - 1, 4 * nside - 2 - nside // 3]
    _check(nside, lmax, order, rings)


@pytest.mark.parametrize("nside,lmax,order", [(512, 128, 3), (1024, 33, 4), (2048, 400, 2)])
def test_cap_rings_longer_than_their_grid(nside, lmax, order):
    _check(nside, lmax, order, [nside // 8, nside // 2, nside - 3, nside - 2, 4 * nside - 2 - nside // 2, 2 * nside])


@pytest.mark.parametrize("lmax", [2000, 6001])
def test_both_kernels_in_one_plan_nside4096(lmax):
    """lmax 2000: the belt alone on the general ring FFT, cap rings of up to 16380 pixels on the grids;
    6001: the outer cap rings too (bands above 4095), others on two interleaved grids."""
    nside = 4096
    _check(nside, lmax, 1, [600, 1500, 2050, 3300, 4000, 4094, 5001, 8191, 4 * nside - 2 - 4000], damp=800.0)


def test_interleaved_rows_with_both_kernels_nside4096():
    """The tensor-core stage's rows for a plan that mixes the kernels, against the float stage's."""
    nside, lmax, order = 4096, 1500, 3
    d = to_dev(sky(nside, lmax, pol=False, damp_t=400.0))
    out = {}
    for precision in (api.MIXED_FP32, api.MIXED_BF16x3):
        plan = api.Plan(nside, lmax, order, pol=False, precision=precision)
        out[precision] = plan.lens(d["T"], None, None, d["phi"]).cpu().numpy()
        torch.cuda.synchronize()
        plan.close()
    a, b = out[api.MIXED_BF16x3], out[api.MIXED_FP32]
    n = 2 * nside * (nside - 1)  # pixels of a cap
    for part in (slice(0, n), slice(n, -n), slice(-n, None)):
        assert rel_rms(a[..., part], b[..., part]) < 1e-4, (part, rel_rms(a[..., part], b[..., part]))

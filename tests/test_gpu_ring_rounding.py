"""Float rounding of the ring synthesis by itself: coefficient rows given directly (launch_ringfft_planes, the
stage's own entry; Naess & Louis 2013, Sec. II.B), against each ring's sum in double precision.

The bound is what packed pairs of maps with Bluestein's convolution measure on these rings: 1.8 to 2.6e-7
relative RMS over the phi-derivatives 0 .. 4 of a row, here 2.6e-7 for the caps and 1.6e-7 for the belt. The rows
rise as (m + 1)^p towards the top of the band, where the interpolation amplifies rounding; the
rings lie just below and above the bands where a larger grid takes over, at odd and folded
bands, and where two interleaved grids are used."""
import ctypes

import numpy as np
import pytest
import torch

import oracle.healpix as hp

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")
_lib = pytest.importorskip("paper_1307_0719_gb300._lib")

LAUNCH = "_ZN2tl21launch_ringfft_planesEPK7tl_planPKPKvPKNS_6MapJobEiP11CUstream_st"
BANDS = "_ZN2tl15host_ring_bandsEiiiPKdS1_Pi"


class MapJob(ctypes.Structure):
    _fields_ = [("plane", ctypes.c_int), ("j", ctypes.c_int), ("k", ctypes.c_int), ("div_sint", ctypes.c_int),
                ("scale", ctypes.c_double), ("out", ctypes.c_void_p), ("tile", ctypes.c_longlong), ("il", ctypes.c_int)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _bands(nside, lmax):
    tab = hp.ring_table(nside)
    th = np.asarray(tab["theta"], dtype=np.float64)
    z, s, out = np.cos(th), np.sin(th), np.zeros(4 * nside - 1, np.int32)
    dp = ctypes.POINTER(ctypes.c_double)
    getattr(_lib.lib(), BANDS)(nside, lmax, 32, s.ctypes.data_as(dp), z.ctypes.data_as(dp),
                               out.ctypes.data_as(ctypes.POINTER(ctypes.c_int)))
    return tab, out


@pytest.mark.parametrize("p", [0, 2])
@pytest.mark.parametrize("nside,lmax,rings", [
    (64, 128, [4, 20, 40, 62, 100]),
    (512, 1024, [50, 280, 300, 350, 380, 500, 1000]),
    (512, 1301, [200, 350, 480, 900]),
    (1024, 2048, [300, 560, 640, 700, 1020, 2000]),
    (2048, 3000, [399, 900, 1650, 1730, 1760, 2040, 4000]),
    (2048, 4096, [1300, 2046]),
])
def test_rounding_of_a_ring(nside, lmax, rings, p):
    K = 5
    tab, mcut = _bands(nside, lmax)
    m = np.arange(lmax + 1)
    rng = np.random.default_rng(7)
    F = np.zeros((4 * nside - 1, lmax + 1), np.complex64)
    for r in rings:
        row = (rng.standard_normal(lmax + 1) + 1j * rng.standard_normal(lmax + 1)) * ((m + 1.0) / (lmax + 1)) ** p
        row[mcut[r] + 1:] = 0  # (functions beyond are held at zero)
        F[r] = row
    plan = api.Plan(nside, lmax, 4, pol=False, precision=api.MIXED_FP32)
    try:
        rows = torch.from_numpy(F).cuda()
        out = torch.zeros(K, 12 * nside * nside, dtype=torch.float32, device="cuda")
        planes = (ctypes.c_void_p * 4)(*[rows.data_ptr()] * 4)
        jobs = (MapJob * K)(*[MapJob(0, 0, k, 0, 1.0, out[k].data_ptr(), 0, 0) for k in range(K)])
        torch.cuda.synchronize()
        assert getattr(_lib.lib(), LAUNCH)(ctypes.c_void_p(getattr(plan._h, "value", plan._h)), planes, jobs, K,
                                           ctypes.c_void_p(0)) == 0
        torch.cuda.synchronize()
    finally:
        plan.close()
    for r in rings:
        n, a = int(tab["nphi"][r]), int(tab["first"][r])
        err = []
        for k in range(K):
            g = F[r].astype(complex) * (1j * m / (lmax + 1)) ** k * np.exp(1j * m * float(tab["phi0"][r]))
            c = np.zeros(n, complex)
            np.add.at(c, m % n, g * np.where(m > 0, 2, 1))
            ref = (np.fft.ifft(c) * n).real
            err.append(np.mean((out[k, a:a + n].double().cpu().numpy() - ref) ** 2) / np.mean(ref ** 2))
        bound = 1.6e-7 if n == 4 * nside else 2.6e-7
        assert np.sqrt(np.mean(err)) < bound, (r, n, int(mcut[r]), np.sqrt(err))

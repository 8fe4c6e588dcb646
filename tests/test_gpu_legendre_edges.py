"""The Legendre kernels at the edges of their loops (Naess & Louis 2013, Sec. II.B): l ranges of one step up
to just over the staged 32, units of fewer 8-l blocks than parts (four, two or one by order and form),
every order, and spheres whose polar rings are cut in m. Each against the FP64 kernels, which the
other tests hold to the oracle.

Tolerances, as where these forms meet the oracle: 5e-5 relative RMS per derivative map for the float
recurrence (test_gpu_ringfft.py), 1e-4 for lensed maps of the split-precision contractions (test_gpu_parity.py), 1e-5
for the analysis (test_gpu_analysis.py), 5e-6 for the gradients of T, E and B
(test_gpu_adjoint.py) and 3e-5 for the potential's, which amplifies the maps' float error (6e-7) up to fifty times."""
import numpy as np
import pytest
import torch

from gpu_util import rel_rms, sky, to_dev

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def _cmp(a, b):
    return rel_rms(torch.view_as_real(a).cpu().numpy(), torch.view_as_real(b).cpu().numpy())


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("nside,lmax,order", [(16, 2, 0), (16, 3, 1), (8, 31, 6), (16, 32, 5), (32, 33, 2), (32, 65, 3),
                                              (256, 400, 1)])
def test_float_recurrence(nside, lmax, order, spin):
    d = to_dev(sky(nside, lmax, pol=True, seeds=(11, 12, 1), b_scale=0.6))
    alm = torch.cat([d["E"], d["B"]]) if spin else d["T"]
    ref = api.synth_derivs(nside, lmax, order, alm, spin, api.FP64).cpu().numpy()
    out = api.synth_derivs(nside, lmax, order, alm, spin, api.MIXED_FP32).cpu().numpy()
    for i in range(ref.shape[0]):
        if np.any(ref[i]):
            assert rel_rms(out[i], ref[i]) < 5e-5, (i, rel_rms(out[i], ref[i]))


@pytest.mark.parametrize("precision", ["MIXED_BF16x3", "MIXED_TF32x3"])
@pytest.mark.parametrize("nside,lmax,order", [(16, 2, 4), (16, 9, 4), (16, 17, 1), (32, 26, 5), (32, 33, 6), (64, 150, 2)])
def test_tensor_core_parts(nside, lmax, order, precision):
    skies = [to_dev(sky(nside, lmax, pol=True, seeds=(11 + i, 12 + i, 1 + i), b_scale=0.6)) for i in range(3)]
    plan = api.Plan(nside, lmax, order, pol=True, precision=getattr(api, precision))
    out = [o.cpu().numpy() for o in plan.lens_batch(skies)]
    plan.check_device_error()
    plan.close()
    for s, o in zip(skies, out):
        ref = torch.stack(list(api.lens(nside, lmax, order, s["T"], s["E"], s["B"], s["phi"]))).cpu().numpy()
        for f in range(3):
            assert rel_rms(o[f], ref[f]) < 1e-4, (f, rel_rms(o[f], ref[f]))


@pytest.mark.parametrize("nside,lmax", [(8, 2), (8, 15), (16, 16), (16, 33), (64, 63), (128, 256)])
def test_float_analysis(nside, lmax):
    g = torch.Generator(device="cuda").manual_seed(nside + lmax)
    maps = torch.randn(3, 12 * nside * nside, dtype=torch.float32, device="cuda", generator=g)
    res = []
    for precision in (api.FP64, api.MIXED_FP32):
        plan = api.Plan(nside, lmax, 0, pol=True, precision=precision)
        m = maps.to(plan.dtype)
        res.append(plan.map2alm(m[0].contiguous(), m[1].contiguous(), m[2].contiguous()))
        torch.cuda.synchronize()
        plan.close()
    for f in "TEB":
        assert _cmp(res[1][f], res[0][f]) < 1e-5, (f, _cmp(res[1][f], res[0][f]))


@pytest.mark.parametrize("nside,lmax,order", [(8, 15, 5), (16, 17, 3), (16, 33, 1)])
def test_float_gradient(nside, lmax, order):
    d = to_dev(sky(nside, lmax, pol=True, b_scale=0.5))
    g = torch.Generator(device="cuda").manual_seed(nside + order)
    maps = torch.randn(3, 12 * nside * nside, dtype=torch.float32, device="cuda", generator=g)
    res = []
    for precision in (api.FP64, api.MIXED_FP32):
        plan = api.Plan(nside, lmax, order, pol=True, precision=precision)
        m = maps.to(plan.dtype)
        res.append(plan.lens_adjoint(d["T"], d["E"], d["B"], d["phi"], m[0].contiguous(), m[1].contiguous(),
                                     m[2].contiguous()))
        torch.cuda.synchronize()
        plan.close()
    for f, tol in (("T", 5e-6), ("E", 5e-6), ("B", 5e-6), ("phi", 3e-5)):
        assert _cmp(res[1][f], res[0][f]) < tol, (f, _cmp(res[1][f], res[0][f]))

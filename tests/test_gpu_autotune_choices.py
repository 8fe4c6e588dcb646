"""The batch autotuner times only what reaches a kernel: up to Nside 2048 no tensor-core plan's rings take the
general ring FFT, so its batching keeps the automatic value (0), and where tensor memory holds one CTA
per SM there is one grid. With the general ring FFT for every ring there is a batching to choose. The choice
is read back from the tuning cache, one line '<key> <grid> <batching of each group>'."""
import pytest
import torch

from gpu_util import rel_rms, sky, to_dev

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")

NSIDES, LMAXS = [16, 32, 16], [32, 64, 32]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("order,ring_fft,grids,batchings", [(4, None, (1,), {0}), (1, None, (1, 2), {0}),
                                                            (4, "shared", (1,), {1, 4})])
def test_choices(order, ring_fft, grids, batchings, tmp_path, monkeypatch):
    cache = tmp_path / "tune"
    monkeypatch.setenv("TAYLENS_TUNE_CACHE", str(cache))
    if ring_fft:
        monkeypatch.setenv("TAYLENS_RING_FFT", ring_fft)
    skies = [to_dev(sky(ns, lm, pol=True, seeds=(5 + i, 6 + i, 7 + i), b_scale=0.3))
             for i, (ns, lm) in enumerate(zip(NSIDES, LMAXS))]
    b = api.Batch(NSIDES, LMAXS, order, pol=True, precision=api.MIXED_BF16x3)
    try:
        outs = b.outputs()
        b.autotune(skies, outs)
        b.lens(skies, outs, "graph")
        ref = b.outputs()
        b.lens(skies, ref, "loop")
        torch.cuda.synchronize()
        for o, r in zip(outs, ref):
            for f in range(3):
                assert rel_rms(o[f].cpu().numpy(), r[f].cpu().numpy()) < 1e-6
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        words = cache.read_text().split()
        assert int(words[1]) == b.grid and b.grid in [k * sms for k in grids]
        assert len(words) == 2 + b.groups and {int(w) for w in words[2:]} <= batchings
    finally:
        torch.cuda.synchronize()
        b.close()

"""The persistent Legendre launch at the orders whose basis tiles have two buffers per part (1 to 3 in
BF16x3, 1 in 3xTF32): the barriers are initialised anew between items, so every commit of an
item has to have arrived before. Against the per-realisation loop, and replay against replay bit for
bit (Naess & Louis 2013, Eq. 4). Band limits from one 8-l block up, so that units of one hand-off
and of two occur."""
import pytest
import torch

from gpu_util import rel_rms, sky, to_dev

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")

NSIDES = [16, 32, 64, 16, 32]
LMAXS = [9, 33, 100, 40, 64]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("order,precision", [(1, "MIXED_BF16x3"), (2, "MIXED_BF16x3"), (3, "MIXED_BF16x3"),
                                             (1, "MIXED_TF32x3")])
def test_persistent_units_with_two_buffers(order, precision):
    skies = [to_dev(sky(ns, lm, pol=True, seeds=(20 + i, 30 + i, 40 + i), b_scale=0.3))
             for i, (ns, lm) in enumerate(zip(NSIDES, LMAXS))]
    b = api.Batch(NSIDES, LMAXS, order, pol=True, precision=getattr(api, precision))
    try:
        ref = b.outputs()
        b.lens(skies, ref, "loop")
        first = None
        for rep in range(20):
            outs = b.outputs()
            b.lens(skies, outs, "persistent")
            if first is None:
                first = outs
                for o, r in zip(outs, ref):
                    for f in range(3):
                        assert rel_rms(o[f].cpu().numpy(), r[f].cpu().numpy()) < 1e-6
            for o, r in zip(outs, first):
                assert torch.equal(o, r), rep
    finally:
        torch.cuda.synchronize()
        b.close()

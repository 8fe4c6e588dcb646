"""Replays of a captured batch on small spheres, whose ring groups are all resident at once: a group that
was not ordered before the gather would show as maps of the replay before. The skies change between replays in
the same buffers, and every replay of a sky has to give the same bits (Naess & Louis 2013, Eq. 4)."""
import pytest
import torch

from gpu_util import rel_rms, sky, to_dev

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")

NSIDES = [16, 32, 64, 16, 64]
LMAXS = [40, 64, 100, 40, 100]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def test_replays_follow_their_inputs():
    sets = [[to_dev(sky(ns, lm, pol=True, seeds=(200 + i + k, 300 + i + k, 400 + i + k), b_scale=0.3))
             for i, (ns, lm) in enumerate(zip(NSIDES, LMAXS))] for k in (0, 50)]
    buf = [{f: t.clone() for f, t in s.items()} for s in sets[0]]
    b = api.Batch(NSIDES, LMAXS, 4, pol=True, precision=api.MIXED_BF16x3)

    def load(k):
        for d, s in zip(buf, sets[k]):
            for f in d:
                d[f].copy_(s[f])

    try:
        ref = []
        for k in (0, 1):
            load(k)
            outs = b.outputs()
            b.lens(buf, outs, "loop")
            torch.cuda.synchronize()
            ref.append([o.clone() for o in outs])
        outs = b.outputs()
        first = [None, None]
        for rep in range(60):
            k = rep & 1
            load(k)
            b.lens(buf, outs, "graph")
            now = [o.clone() for o in outs]
            if first[k] is None:
                first[k] = now
                for o, r in zip(now, ref[k]):
                    for f in range(3):
                        assert rel_rms(o[f].cpu().numpy(), r[f].cpu().numpy()) < 1e-6
            else:
                for o, r in zip(now, first[k]):
                    assert torch.equal(o, r), rep
    finally:
        torch.cuda.synchronize()
        b.close()

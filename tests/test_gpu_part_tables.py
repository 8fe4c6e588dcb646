"""Memory of the tensor-core start tables: a plan holds a part table for every part after the first that its
kernels split a unit's l range into, and none where a unit is one part. At order 5 a BF16x3 unit is two parts and a
3xTF32 unit one (tensor memory: 6 x 64 accumulator columns, 48 or 96 columns of basis tiles per part);
everything else of the two plans has the same size, so they differ by one table of T and one of Q/U.
The same with the tables read: both against the float maps (Naess & Louis 2013, Eq. 4)."""
import pytest
import torch

from gpu_util import rel_rms, sky, to_dev

pytestmark = pytest.mark.gpu

api = pytest.importorskip("paper_1307_0719_gb300.api")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("nside,lmax", [(64, 128), (128, 300)])
def test_part_tables_at_order_5(nside, lmax):
    order = 5
    d = to_dev(sky(nside, lmax, pol=True, b_scale=0.3))
    ref = api.lens(nside, lmax, order, d["T"], d["E"], d["B"], d["phi"], precision=api.MIXED_FP32).cpu().numpy()
    size = {}
    for name in ("MIXED_BF16x3", "MIXED_TF32x3"):
        plan = api.Plan(nside, lmax, order, pol=True, precision=getattr(api, name))
        size[name] = plan.workspace_bytes
        out = plan.lens(d["T"], d["E"], d["B"], d["phi"]).cpu().numpy()
        plan.close()
        for f in range(3):
            assert rel_rms(out[f], ref[f]) < 1e-4, (name, f)
    blocks = -(-2 * nside // 128) + -(-2 * nside // 64)  # of T and of Q/U, per m
    table = (lmax + 1) * blocks * (2 * (order + 1) + 1) * 128 * 4
    assert size["MIXED_BF16x3"] - size["MIXED_TF32x3"] == table

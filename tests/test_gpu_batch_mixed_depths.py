"""Batches that mix systems with and without light cells (sparse trees of at
least 64^3 cells beside others) run merged, each system as by itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMM, FMMBatch, inputs  # noqa: E402


@pytest.mark.parametrize("periodic,continuous", [(True, True), (False, False)])
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
def test_light_and_other_systems_merge(precision, periodic, continuous):
    pos, q, offs, boxes, counts = inputs.batch_systems(5, 44, lo=3000, hi=30000)
    depths = np.array([3, 6, 5, 6, 2])
    kw = dict(periodic=periodic, continuous=continuous, precision=precision)
    bt = FMMBatch(boxes, depths, 4, max_n=counts, sync=True, **kw)
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    for _ in range(2):  # recorded and tuned, then replayed
        r = bt.eval(P, Q, offs)
        st = bt.stats()
        assert st["merged"] and st["lanes"] == 0
    for i in range(5):
        a, b = offs[i], offs[i + 1]
        plan = FMM(tuple(boxes[i]), int(depths[i]), 4, max_n=int(counts[i]), **kw)
        s = plan.eval(P[a:b].contiguous(), Q[a:b].contiguous())
        for k in ("potential", "forces"):
            assert torch.equal(r[k][a:b], s[k]), (i, k)
        assert r["energy"][i] == s["energy"][0]
        plan.close()
    bt.close()

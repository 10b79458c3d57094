"""Systems that do not start at row 0 of the caller's arrays: calls with equal
counts and other first rows (windows of one trajectory array) evaluate and write
the rows that their offsets name."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMM, FMMBatch, inputs  # noqa: E402


@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "fp64"])
def test_windows_of_one_array(precision):
    pos, q, offs, boxes, counts = inputs.batch_systems(4, 43, lo=1024, hi=5000)
    N, frames, kw = len(q), 3, dict(periodic=True, continuous=True, precision=precision)
    g = torch.Generator().manual_seed(9)
    P, Q = torch.rand(frames * N, 3, generator=g).cuda(), torch.from_numpy(np.tile(q, frames)).cuda()
    dt = torch.float64 if precision == "fp64" else torch.float32
    want = []
    for i in range(4):
        plan = FMM(tuple(boxes[i]), 3, 4, max_n=int(counts[i]), **kw)
        want.append([])
        for f in range(frames):
            a, b = f * N + int(offs[i]), f * N + int(offs[i + 1])
            want[i].append({k: v.clone() for k, v in plan.eval(P[a:b].contiguous(), Q[a:b].contiguous()).items()})
        plan.close()
    bt = FMMBatch(boxes, [3] * 4, 4, max_n=counts, sync=True, **kw)
    out = {"potential": torch.empty(frames * N, dtype=dt, device="cuda"),
           "forces": torch.empty(frames * N, 3, dtype=dt, device="cuda")}
    for f in (0, 2, 1, 0):  # the same arrays throughout; then arrays of the call's own
        for o in (out, None):
            if o is not None:
                for v in o.values():
                    v.fill_(float("nan"))
            r = bt.eval(P, Q, offs + f * N, out=o)
            for i in range(4):
                a, b = f * N + int(offs[i]), f * N + int(offs[i + 1])
                for k in ("potential", "forces"):
                    assert torch.equal(r[k][a:b], want[i][f][k]), (f, i, k)
                assert r["energy"][i] == want[i][f]["energy"][0]
            if o is not None:  # and no row outside the window is written
                for v in o.values():
                    assert torch.isnan(v[: f * N]).all() and torch.isnan(v[(f + 1) * N:]).all()
    bt.close()

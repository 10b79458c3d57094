"""Workspaces between fmm_workspace_minimum and fmm_workspace_size: FP32 plans
take FP32 multiply-adds in them, single and batched alike; fewer bytes are refused;
the package falls back to them where device memory does not hold the full size."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2212_13080_gb300 as pkg  # noqa: E402
from paper_2212_13080_gb300 import FMM, FMMBatch, FmmError, inputs  # noqa: E402
from paper_2212_13080_gb300 import _binding as B  # noqa: E402


def _bytes(n):
    ws = torch.empty(n + 256, dtype=torch.uint8, device="cuda")
    return ws[(-ws.data_ptr()) % 256:][:n]


def test_sizes_by_precision():
    for precision, p, smaller in (("fp32", 6, True), ("fp32", 7, False), ("tf32x3", 6, False), ("fp64", 4, False)):
        plan = FMM((0, 0, 0, 1), 5, p, precision=precision, max_n=20000)
        size, least = plan.workspace_size(20000), B.fmm_workspace_minimum(plan._h, 20000)
        assert least < size if smaller else least == size, precision
        plan.close()


@pytest.mark.parametrize("p", [3, 4, 5, 6])
def test_batch_in_the_smallest_workspace(p):
    pos, q, offs, boxes, counts = inputs.batch_systems(4, 45, lo=1024, hi=9000)
    depths = np.array([3, 4, 5, 2])
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    bt = FMMBatch(boxes, depths, p, periodic=True, max_n=counts, sync=True)
    size, least = B.fmm_batch_workspace_size(bt._h, counts), B.fmm_batch_workspace_minimum(bt._h, counts)
    assert least < size
    N = len(q)
    phi, E = torch.empty(N, device="cuda"), torch.empty(4, dtype=torch.float64, device="cuda")
    F = torch.empty(N, 3, device="cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (P, Q, phi, E, F)]
    ws = _bytes(size)
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    with pytest.raises(FmmError) as e:
        B.fmm_batch_eval(bt._h, offs, *ptr, ctypes.c_void_p(ws.data_ptr()), least - 256, st)
    assert e.value.code == B.FMM_ERR_WORKSPACE
    for nbytes in (least, size, least):  # one batch object, in turn
        B.fmm_batch_eval(bt._h, offs, *ptr, ctypes.c_void_p(ws.data_ptr()), nbytes, st)
        assert bt.stats()["merged"]
        for i in range(4):
            a, b = offs[i], offs[i + 1]
            plan = FMM(tuple(boxes[i]), int(depths[i]), p, periodic=True, max_n=int(counts[i]))
            m = B.fmm_workspace_minimum(plan._h, int(counts[i]))
            full = plan.workspace_size(int(counts[i]))
            r = plan.eval(P[a:b].contiguous(), Q[a:b].contiguous(), workspace=_bytes(m if nbytes == least else full))
            assert torch.equal(phi[a:b], r["potential"]) or (m == full and nbytes == least), (nbytes == least, i)
            plan.close()
    bt.close()


def test_package_falls_back(monkeypatch):
    pos, q, box = inputs.uniform_pm1(9001, 46)
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    plan = FMM(box, 5, 6, max_n=len(q))
    size, least = plan.workspace_size(len(q)), B.fmm_workspace_minimum(plan._h, len(q))
    want = plan.eval(P, Q, workspace=_bytes(least))["potential"].clone()
    other = plan.eval(P, Q, workspace=_bytes(size))["potential"].clone()
    assert not torch.equal(want, other)
    empty, asked = torch.empty, []

    def short(*a, **k):
        if k.get("dtype") == torch.uint8:
            asked.append(a[0])
            if a[0] > least + 256:
                raise torch.cuda.OutOfMemoryError("no room")
        return empty(*a, **k)

    monkeypatch.setattr(pkg.torch, "empty", short)
    for n in (len(q), len(q), 5000):
        r = plan.eval(P[:n].contiguous(), Q[:n].contiguous())["potential"]
        if n == len(q):
            assert torch.equal(r, want)
    assert asked == [size + 256, least + 256]  # tried once, and the smaller one kept
    plan.close()
    tc = FMM(box, 5, 6, precision="tf32x3", max_n=len(q))
    with pytest.raises(torch.cuda.OutOfMemoryError):  # no smaller form
        tc.eval(P, Q)
    tc.close()

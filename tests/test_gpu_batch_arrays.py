"""A batch's captured graph serves any arrays: calls with other inputs and
outputs, queued without waiting, give what each would give alone."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMMBatch, inputs  # noqa: E402


@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "fp64"])
def test_other_arrays_every_call(precision):
    pos, q, offs, boxes, counts = inputs.batch_systems(5, 41, lo=1024, hi=6000)
    mk = dict(periodic=True, continuous=True, precision=precision, max_n=counts)
    P = [torch.rand(len(q), 3, generator=torch.Generator().manual_seed(k)).cuda() for k in range(3)]
    Q = [torch.from_numpy(q).cuda() * (k + 1) for k in range(3)]
    want = []
    for k in range(3):  # a batch object of its own for every set of arrays
        bt = FMMBatch(boxes, [3] * 5, 4, sync=True, **mk)
        want.append({n: v.clone() for n, v in bt.eval(P[k], Q[k], offs).items()})
        if k == 2:  # energies alone take the potential-only kernels
            want_energy = bt.eval(P[k], Q[k], offs, potential=False, forces=False)["energy"].clone()
        bt.close()
    bt = FMMBatch(boxes, [3] * 5, 4, sync=False, **mk)
    got = [(k, bt.eval(P[k], Q[k], offs)) for k in (0, 1, 2, 1, 0)]
    # fewer outputs: another graph
    only = bt.eval(P[2], Q[2], offs, potential=False, forces=False)
    again = bt.eval(P[1], Q[1], offs)
    torch.cuda.synchronize()
    for k, r in got + [(1, again)]:
        for n in want[k]:
            assert torch.equal(r[n], want[k][n]), (k, n)
    assert only["potential"] is None and torch.equal(only["energy"], want_energy)
    bt.close()

"""Near field of sparse deep trees in single precision: cells with few charges
take their pairs one-sided, the others in mutual form.  Compared with the FP64
plan (mutual form throughout) where light, dense and empty cells mix."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMM, inputs  # noqa: E402

TOL_FP32 = 1e-6


def _mixed(n, seed):
    """Uniform background and a dense ball: cells of 0 to several hundred charges."""
    rng = np.random.default_rng(seed)
    a = rng.random((n // 2, 3))
    b = 0.4 + 0.05 * rng.standard_normal((n - n // 2, 3))
    pos = np.clip(np.concatenate([a, b]), 0.0, 0.999999).astype(np.float32)
    q = np.ones(n, np.float32)
    q[::2] = -1.0
    return pos, rng.permutation(q), (0.0, 0.0, 0.0, 1.0)


CASES = [("open_plain", dict(), 3), ("open_cont", dict(continuous=True), 4),
         ("periodic_odd", dict(continuous=True, periodic=True), 3),
         ("inverse_square", dict(kernel="inverse_square"), 3)]


@pytest.mark.parametrize("forces", [True, False])
@pytest.mark.parametrize("name,kw,p", CASES, ids=[c[0] for c in CASES])
def test_light_and_dense_cells(name, kw, p, forces):
    pos, q, box = _mixed(300001, 5)
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    out = []
    for precision in ("fp64", "fp32"):
        plan = FMM(box, 6, p, precision=precision, max_n=len(q), **kw)
        r = plan.eval(P, Q, forces=forces)
        out.append({k: v.double().clone() for k, v in r.items() if v is not None})
        plan.close()
    for k in out[0]:
        if k == "energy":
            continue  # a small difference of large sums here
        assert float((out[1][k] - out[0][k]).norm() / out[0][k].norm()) < TOL_FP32, k


def test_coincident_and_split_charges_of_light_cells():
    """Pairs of coincident particles contribute nothing, in light cells too."""
    rng = np.random.default_rng(6)
    pos = rng.random((20000, 3)).astype(np.float32)
    pos = np.concatenate([pos, pos[:500], pos[:500]])
    q = rng.uniform(-1, 1, len(pos)).astype(np.float32)
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    out = []
    for precision in ("fp64", "fp32"):
        plan = FMM((0, 0, 0, 1), 6, 5, precision=precision, continuous=True, max_n=len(q))
        out.append({k: v.double().clone() for k, v in plan.eval(P, Q).items()})
        plan.close()
    assert torch.isfinite(out[1]["forces"]).all()
    for k in ("potential", "forces"):
        assert float((out[1][k] - out[0][k]).norm() / out[0][k].norm()) < TOL_FP32, k

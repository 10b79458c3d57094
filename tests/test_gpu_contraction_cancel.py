"""Sums over the interaction list whose terms cancel: a periodic box whose octants
are charged in turn.  At level 1 every source cell appears as 27 images of one sign;
the order in which a target's 189 offsets are added decides how large the partial
sums become, and every rounding of a term counts against a small result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMM  # noqa: E402


def _octants(n, seed):
    rng = np.random.default_rng(seed)
    pos = rng.random((n, 3)).astype(np.float32)
    q = np.where((pos >= 0.5).sum(1) & 1, -1.0, 1.0) * (0.5 + rng.random(n))
    return torch.from_numpy(pos).cuda(), torch.from_numpy((q - q.mean()).astype(np.float32)).cuda()


@pytest.mark.parametrize("depth", [2, 4])  # levels whose offsets are split over blocks
@pytest.mark.parametrize("p", [4, 5, 6])
def test_alternating_octants_keep_fp32_errors(p, depth):
    P, Q = _octants(4096, p)
    phi = {}
    for precision in ("fp64", "fp32", "tf32x3"):
        plan = FMM((0, 0, 0, 1), depth, p, periodic=True, precision=precision, max_n=len(Q))
        full = plan.workspace_size(len(Q))
        ws = torch.empty(full + 512, dtype=torch.uint8, device="cuda")
        ws = ws[(-ws.data_ptr()) % 256:]
        # FP32 plans: the split form, and with the smaller workspace FP32 multiply-adds
        for name, size in ((precision, full), ("simt", full - 256))[: 2 if precision == "fp32" else 1]:
            phi[name] = plan.eval(P, Q, forces=False, workspace=ws[:size])["potential"].double().clone()
        plan.close()
    err = {k: float((v - phi["fp64"]).norm() / phi["fp64"].norm()) for k, v in phi.items()}
    ulps = 2 * 2.0 ** -24
    # as many roundings at the size of the terms as the multiply-adds have: the same
    # error, and a sample's scatter
    assert err["fp32"] <= 1.25 * err["simt"] + ulps, err
    # no compensation of the sum: a second rounding per term, at the size of partial
    # sums of a term or two
    assert err["tf32x3"] <= 2.0 * err["simt"] + ulps, err

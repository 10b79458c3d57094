"""Digits of the split contraction of FP32 plans (p = 3..6) where the interaction
list's terms cancel: on average over systems as many as FP32 multiply-adds keep."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMM  # noqa: E402

SYSTEMS = 16


@pytest.mark.parametrize("p", [3, 4, 5, 6])
def test_mean_error_is_that_of_fp32_multiply_adds(p):
    n = 4096
    ref = FMM((0, 0, 0, 1), 2, p, periodic=True, precision="fp64", max_n=n)
    plan = FMM((0, 0, 0, 1), 2, p, periodic=True, max_n=n)
    full = plan.workspace_size(n)
    ws = torch.empty(full + 512, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    ratio = []
    for seed in range(SYSTEMS):
        rng = np.random.default_rng(seed)
        pos = rng.random((n, 3)).astype(np.float32)
        q = np.where((pos >= 0.5).sum(1) & 1, -1.0, 1.0) * (0.5 + rng.random(n))  # octants charged in turn
        P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy((q - q.mean()).astype(np.float32)).cuda()
        want = ref.eval(P, Q, forces=False)["potential"]
        # the split form; with the smaller workspace the multiply-adds
        e = [float((plan.eval(P, Q, forces=False, workspace=ws[:k])["potential"].double() - want).norm())
             for k in (full, full - 256)]
        ratio.append(e[0] / e[1])
    # both round every term once, at its own size: a ratio of 1.  A system's ratio
    # scatters by some 5% (its error is a few large, correlated roundings), the mean
    # of 16 by an 80th: three of those
    assert np.exp(np.mean(np.log(ratio))) <= 1.0 + 3 * 0.05 / np.sqrt(SYSTEMS), ratio
    plan.close()
    ref.close()

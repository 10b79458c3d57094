"""Plans of one process on several devices: what a kernel needs to be launched
with is set on the plan's own device."""
import glob
import os
import re

import pytest

torch = pytest.importorskip("torch")

from paper_2212_13080_gb300 import FMM, inputs  # noqa: E402

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2212_13080_gb300", "csrc")


def test_no_process_wide_once_flags():
    """A function attribute belongs to the device that was current when it was
    set: no launch hides it behind a flag of the process."""
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"\bstatic\s+bool\s+\w+\s*=", open(f).read()), f


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
def test_second_device_evaluates(precision):
    if torch.cuda.device_count() < 2:
        pytest.skip("one device")
    pos, q, box = inputs.uniform_pm1(4096, 3)
    got = []
    for d in (0, 1):
        dev = torch.device("cuda", d)
        with torch.cuda.device(dev):
            plan = FMM(box, 3, 4, precision=precision, max_n=len(q), device=dev)
            r = plan.eval(torch.from_numpy(pos).to(dev), torch.from_numpy(q).to(dev))
            got.append({k: v.cpu().clone() for k, v in r.items()})
            plan.close()
    for k in got[0]:
        assert torch.equal(got[0][k], got[1][k]), k

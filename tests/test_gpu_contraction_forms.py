"""The two forms of the far-field contraction of FP32 plans (p = 3..6): split
half-precision operands on the tensor cores (a full workspace) and FP32
multiply-adds (a workspace that holds no operand copy).  Both are compared with
the FP64 plan over the forms a plan accepts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2212_13080_gb300 import FMM, FmmError, inputs  # noqa: E402


def _system(dist, n, seed):
    if dist == "water":
        return inputs.water(n // 3, seed)
    if dist == "plummer":
        return inputs.plummer(n, seed)
    return inputs.uniform_cont(n, seed) if dist == "cont" else inputs.uniform_pm1(n, seed)


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


# depth 2 and 3: only levels whose offsets are split over blocks; 4: the finest
# level too; 5: box tiles, and gathered tiles of a clustered system
FORMS = [("uniform", 257, 2, dict()), ("cont", 3001, 3, dict(continuous=True)),
         ("water", 3000, 2, dict(periodic=True, continuous=True)),
         ("water", 24000, 4, dict(periodic=True, continuous=True)),
         ("plummer", 30001, 5, dict()), ("uniform", 250000, 5, dict()),
         ("cont", 9001, 4, dict(continuous=True, force_mode="kernel")),
         ("uniform", 9001, 4, dict(kernel="inverse_square")), ("uniform", 9001, 4, dict(grid_scale=1 / 1.2))]


@pytest.mark.parametrize("p", [3, 4, 5, 6])
@pytest.mark.parametrize("dist,n,depth,kw", FORMS, ids=["%s%d" % (f[0], f[1]) for f in FORMS[:6]] +
                         ["force_kernel", "inverse_square", "reduced"])
def test_split_form_is_as_accurate_as_fp32(dist, n, depth, kw, p):
    pos, q, box = _system(dist, n, 31)
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    ref = FMM(box, depth, p, precision="fp64", max_n=len(q), **kw)
    r64 = ref.eval(P, Q)
    plan = FMM(box, depth, p, max_n=len(q), **kw)
    full = plan.workspace_size(len(q))
    ws = torch.empty(full + 512, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    got = {}
    for form, size in (("split", full), ("fp32", full - 256)):
        try:
            r = plan.eval(P, Q, workspace=ws[:size])
        except FmmError:
            assert form == "fp32"  # its scratch is the larger one here: a workspace always holds the split form's
            assert _rel(got["split"]["potential"], r64["potential"]) < 1e-6
            return
        got[form] = {k: v.clone() for k, v in r.items()}
    assert not torch.equal(got["split"]["potential"], got["fp32"]["potential"])  # both forms ran
    for k in ("potential", "forces"):
        e_split, e_fp32 = _rel(got["split"][k], r64[k]), _rel(got["fp32"][k], r64[k])
        # two samples of rounding errors of the same size, and two units in the
        # last place that both share
        assert e_split <= 1.5 * e_fp32 + 2 * 2.0 ** -24, (k, e_split, e_fp32)
    plan.close()
    ref.close()


@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "tf32x1"])
@pytest.mark.parametrize("p", [3, 6])
def test_scaled_charges_scale_the_result(p, precision):
    """The halves' scaling is exact: charges times 2^k give potentials times 2^k,
    bit for bit, far outside the half type's own range."""
    pos, q, box = inputs.uniform_pm1(6000, 32)
    plan = FMM(box, 4, p, precision=precision, max_n=len(q))
    P, Q = torch.from_numpy(pos).cuda(), torch.from_numpy(q).cuda()
    phi = plan.eval(P, Q, energy=False, forces=False)["potential"].clone()
    for k in (-60, -30, 30, 60):
        r = plan.eval(P, Q * 2.0 ** k, energy=False, forces=False)["potential"]
        assert torch.equal(r, phi * 2.0 ** k), k
    # one cell's charges far above all others: the others keep their digits
    big = Q.clone()
    big[(P < 1 / 16).all(1)] *= 2.0 ** 40
    r64 = FMM(box, 4, p, precision="fp64", max_n=len(q))
    far = (P > 0.5).all(1)
    a = plan.eval(P, big, energy=False, forces=False)["potential"][far]
    b = r64.eval(P, big, energy=False, forces=False)["potential"][far]
    assert _rel(a, b) < (1e-3 if precision == "tf32x1" else 1e-5)
    plan.close()
    r64.close()


def test_nonfinite_charges_stay_visible():
    pos, q, box = inputs.uniform_pm1(4000, 33)
    plan = FMM(box, 3, 4, max_n=len(q))
    P = torch.from_numpy(pos).cuda()
    for bad in (float("nan"), float("inf")):
        Q = torch.from_numpy(q).cuda()
        Q[7] = bad
        phi = plan.eval(P, Q, energy=False, forces=False)["potential"]
        assert not torch.isfinite(phi[torch.arange(len(q), device="cuda") != 7]).any()
    plan.close()

"""The order in which the tensor-core contraction walks a target's interaction
list (§2.2 step 3): by source parity, then by the source's coarse shift.  A
restatement of the walk, checked to be the list of every target parity."""
import itertools

import pytest


def walk(par):
    b = (par & 1, (par >> 1) & 1, par >> 2)
    out = []
    for sp in range(8):
        s = (sp & 1, (sp >> 1) & 1, sp >> 2)
        for dz, dy, dx in itertools.product((-1, 0, 1), repeat=3):
            o = tuple(2 * d + s[a] - b[a] for a, d in enumerate((dx, dy, dz)))
            if max(map(abs, o)) > 1:
                out.append((o, sp, (dx, dy, dz)))
    return out


@pytest.mark.parametrize("par", range(8))
def test_walk_is_the_interaction_list(par):
    b = (par & 1, (par >> 1) & 1, par >> 2)
    want = {o for o in itertools.product(*[range(-2 - x, 4 - x) for x in b]) if max(map(abs, o)) > 1}
    got = walk(par)
    assert len(got) == 189 and {o for o, _, _ in got} == want
    for o, sp, d in got:  # the source cell: target (coarse X, parity b) + o
        for a in range(3):
            assert 2 * d[a] + ((sp >> a) & 1) == b[a] + o[a]
    assert [sp for _, sp, _ in got] == sorted(sp for _, sp, _ in got)
    # runs of 21 offsets (small levels) and thirds (depth 4) tile the list
    assert 189 % 9 == 0 and 189 % 3 == 0

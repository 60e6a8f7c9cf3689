"""The level analysis at rows whose number of dependencies lies around the few
that are looked at together, on earlier chunks of 32 rows, on the row's own
chunk and on both, against the CPU oracle (whole numbers: equal)."""
import numpy as np
import pytest

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu


def _system(n, outside, inside, seed):
    rng = np.random.default_rng(seed)
    rp, ci = [0], []
    for i in range(n):
        c = i // 32 * 32
        far = rng.choice(c, size=min(outside[i % len(outside)], c), replace=False) if c else np.zeros(0, int)
        near = c + rng.choice(i - c, size=min(inside[i % len(inside)], i - c), replace=False) if i > c else np.zeros(0, int)
        ci += [*np.sort(np.concatenate([far, near])).astype(int).tolist(), i]
        rp.append(len(ci))
    return S.CSR(n, np.array(rp, np.int32), np.array(ci, np.int32), np.ones(len(ci)))


@pytest.mark.parametrize("outside", [(0,), (1, 3, 4, 5), (7, 8, 9, 12, 13), (31, 32, 33, 40)])
@pytest.mark.parametrize("inside", [(0,), (1,), (0, 3, 4, 5, 31)])
@pytest.mark.parametrize("n", [33, 4099])
def test_levels(n, outside, inside):
    import paper_2609_40159_gb300 as P
    A_h = _system(n, outside, inside, seed=n + len(outside))
    an, ref = P.analyze(P.Matrix.from_host(A_h)), oracle.analyze(A_h)
    assert an.nlevels == ref["nlevels"]
    assert np.array_equal(an.lev.cpu().numpy(), ref["lev"])
    assert np.array_equal(an.perm.cpu().numpy(), ref["perm"])
    assert P.handle().status() == 0

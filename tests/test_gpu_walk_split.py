"""Groups of bodies walked by one, four or eight warps, against the oracle's tree."""
import numpy as np
import pytest

import oracle
from paper_1211_2292_gb300 import inputs, nbody
from helpers import host, relerr_per_body, to_dev

pytestmark = pytest.mark.gpu

# On 152 SMs: groups of 64 take 8 warps below 1216 groups, 4 below 6080;
# groups of 32 take 8 below 3040.  Bounds of the float32 walk: rms 1e-5, max
# 1e-4 of |a| per body; lists (cells, bodies) exact.
CASES = [
    # (n, theta, leaf_cap, group); the first two open so many cells that the
    # warps' segments of the shared frontier (256 nodes) overflow
    (12000, 0.15, 1, 64),
    (12000, 0.15, 1, 32),
    (77823, 0.8, 32, 64),   # 1216 groups: the first size with 4 warps
    (77824 - 64, 0.8, 32, 64),  # 1215 groups
    (97280, 0.8, 32, 32),   # 3040 groups of 32: one warp
    (31, 0.5, 4, 64),
]


@pytest.mark.parametrize("n,theta,leaf_cap,group", CASES)
def test_lists_and_forces_match_the_oracle(cuda, n, theta, leaf_cap, group):
    b = inputs.plummer(n, seed=n)
    ref, stats, cnt_ref = oracle.bh_forces(b.pos, b.mass, 1.0, 0.01, theta, leaf_cap, group,
                                           counts=True)
    with nbody.NBody(n, "fp32_comp") as nb:
        x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
        a, cnt = nb.tree_forces(x, m, 1.0, 0.01, theta, leaf_cap, counts=True, group=group)
        again = nb.tree_forces(x, m, 1.0, 0.01, theta, leaf_cap, group=group)
        nb.sync()
    assert np.array_equal(host(cnt), cnt_ref)
    assert np.array_equal(host(a), host(again))
    err = relerr_per_body(host(a), ref)
    assert np.sqrt(np.mean(err ** 2)) <= 1e-5 and err.max() <= 1e-4


def test_more_groups_than_one_wave_of_small_walks(cuda):
    # 6250 groups, one warp each: the sums do not depend on the schedule
    b = inputs.two_plummer(200000, seed=5)
    x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
    with nbody.NBody(b.n, "fp32_comp") as nb:
        dyn = host(nb.tree_forces(x, m, 1.0, 0.002, 0.7, 16))
        nb.tree_schedule("static")
        assert np.array_equal(host(nb.tree_forces(x, m, 1.0, 0.002, 0.7, 16)), dyn)

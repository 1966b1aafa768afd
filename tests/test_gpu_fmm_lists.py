"""FMM list and work-item passes at the sizes where they take another turn."""
import numpy as np
import pytest

import oracle
from paper_1211_2292_gb300 import inputs, nbody
from helpers import host, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,theta,leaf_cap,order", [
    (20000, 0.75, 1, 2),   # more leaves than one tile (8192) of the work items' scan
    (9000, 0.4, 8, 3),     # cells with candidates for all eight warps, leaves in several slices
    (64, 0.6, 64, 4),      # one leaf, nothing handed down
])
def test_lists_and_items_match_the_oracle(cuda, n, theta, leaf_cap, order):
    # counts exact; forces within the float32 form's 1e-4 of the rms (and 1e-5 rms)
    b = inputs.plummer(n, seed=n)
    ref, stats, cref = oracle.fmm_forces(b.pos, b.mass, 1.0, 0.01, theta, order, leaf_cap,
                                         counts=True)
    with nbody.NBody(n, "fp32_comp") as nb:
        x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
        a, cnt = nb.fmm_forces(x, m, 1.0, 0.01, theta, order, leaf_cap, counts=True)
        again = nb.fmm_forces(x, m, 1.0, 0.01, theta, order, leaf_cap)
        nb.sync()
    assert np.array_equal(host(cnt), cref)
    assert np.array_equal(host(a), host(again))
    d = np.linalg.norm(host(a) - ref, axis=1) / np.sqrt(np.mean(np.sum(ref ** 2, axis=1)))
    assert np.sqrt(np.mean(d ** 2)) <= 1e-5 and d.max() <= 1e-4

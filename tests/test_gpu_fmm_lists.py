"""FMM list and work-item passes at the sizes where they take another turn."""
import numpy as np
import pytest
import torch

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


def test_calls_on_other_streams_and_contexts(cuda):
    # the expansions run on a stream of the context's own: calls in a row on
    # another stream than the arrays', and of two contexts at once
    sys_ = [inputs.plummer(n, seed=n) for n in (3000, 20011)]
    dev = [(to_dev(b.pos, cuda), to_dev(b.mass, cuda)) for b in sys_]
    want = []
    for b, (x, m) in zip(sys_, dev):
        with nbody.NBody(b.n, "fp32_comp") as nb:
            want.append(host(nb.fmm_forces(x, m, 1.0, 0.01, 0.6, 4, 32)))
            st = nb.tree_stats()
            assert (st["nodes"], st["leaves"]) == tuple(nb.fmm_stats()[k] for k in ("nodes", "leaves"))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for s in streams:
        s.wait_stream(torch.cuda.current_stream())
    nbs = [nbody.NBody(20011, "fp32_comp", stream=s) for s in streams]
    outs = [torch.empty_like(dev[1][0]) for _ in range(4)]
    small = [torch.empty_like(dev[0][0]) for _ in nbs]
    for r in range(2):
        for q, nb in enumerate(nbs):  # the small system in between, then the large one
            nb.fmm_forces(*dev[0], 1.0, 0.01, 0.6, 4, 32, out=small[q])
            nb.fmm_forces(*dev[1], 1.0, 0.01, 0.6, 4, 32, out=outs[2 * r + q])
    for nb in nbs:
        nb.sync()
        nb.close()
    for o in small:
        assert np.array_equal(host(o), want[0])
    for o in outs:
        assert np.array_equal(host(o), want[1])

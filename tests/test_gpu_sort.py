"""The radix sort behind the spatial orders: exact orders at the edges of its tiles."""
import numpy as np
import pytest
import torch

from paper_1211_2292_gb300 import nbody

pytestmark = pytest.mark.gpu

# one tile is 1024 keys up to 2^16 of them, 4096 beyond; up to 64 tiles sum
# their counts themselves, more are scanned by a launch of their own
SIZES = [1, 31, 1023, 1024, 1025, 65536, 65537, 262144, 262145, 300001]


@pytest.mark.parametrize("n", SIZES)
def test_orders_are_exact_and_stable(cuda, n):
    rng = np.random.default_rng(n)
    ids = rng.choice(1 << 31, size=n, replace=False).astype(np.int64)
    rank = rng.integers(0, 64, n).astype(np.int32)
    pos = rng.normal(size=(n, 3))
    t = lambda a: torch.as_tensor(a, device=cuda).contiguous()  # noqa: E731
    x, v, m, i = t(pos), t(pos * 2.0), t(pos[:, 0] ** 2), t(ids)
    with nbody.NBody(n, "fp32_comp") as nb:
        want = np.argsort(ids, kind="stable")  # four passes over the whole key
        for _ in range(2):
            got = nb.orb_order(x, v, m, i)
            assert np.array_equal(got[3].cpu().numpy(), ids[want])
            assert np.array_equal(got[0].cpu().numpy(), pos[want])
        want = np.argsort(rank, kind="stable")  # one pass with many equal keys
        got = nb.orb_pack(t(rank), 64, x, v, m, i)
        assert np.array_equal(got[3].cpu().numpy(), ids[want])
        assert np.array_equal(got[4], np.bincount(rank, minlength=64))

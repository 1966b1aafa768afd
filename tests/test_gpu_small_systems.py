"""Direct sums of small systems: the team kernels, and j-splits of equal body counts."""
import numpy as np
import pytest
import torch

import oracle
from paper_1211_2292_gb300 import inputs, nbody
from helpers import host, relerr_per_body, to_dev

pytestmark = pytest.mark.gpu

# float32 pair terms, compensated sums: the mode's bounds, rms 1e-5 and max 1e-4
BOUND = (1e-5, 1e-4)


def _check(a, b, eps):
    err = relerr_per_body(host(a), oracle.accel(b.pos, b.mass, 1.0, eps))
    assert np.sqrt(np.mean(err ** 2)) <= BOUND[0] and err.max() <= BOUND[1]


@pytest.mark.parametrize("variant", [-2, -1])  # the table's last two: 64 and 128 bodies per block
@pytest.mark.parametrize("n", [1, 7, 63, 64, 65, 129, 2047, 2048, 2049, 4096, 4097, 5003])
def test_team_kernels_at_tile_and_cluster_edges(cuda, variant, n):
    # 4096 bodies is the largest system read straight from float64
    b = inputs.random_system(n, seed=n)
    v = len(nbody.variants(nbody.KIND_FORCE, "fp32_comp")) + variant
    x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
    with nbody.NBody(n, "fp32_comp") as nb:
        for eps, split in ((0.02, 0), (0.02, 1), (0.0, 2), (0.02, 8)):
            nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, v, split)
            a = nb.forces(x, m, 1.0, eps)
            again = nb.forces(x, m, 1.0, eps)
            nb.sync()
            assert np.array_equal(host(a), host(again))
            if n > 1:
                _check(a, b, eps)
            else:
                assert np.array_equal(host(a), np.zeros((1, 3)))


def test_output_may_overlap_the_positions(cuda):
    # acc written over pos: the bodies are packed before anything is written
    b = inputs.plummer(700, seed=3)
    x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
    with nbody.NBody(b.n, "fp32_comp") as nb:
        want = host(nb.forces(x, m, 1.0, 0.01))
        got = host(nb.forces(x, m, 1.0, 0.01, out=x))
    assert np.array_equal(got, want)


@pytest.mark.parametrize("variant", [5, 21, 22])  # 21, 22 split by bodies, 5 by tiles
@pytest.mark.parametrize("n", [65, 4097, 9001, 16411])
def test_even_splits_and_their_merge(cuda, variant, n):
    b = inputs.plummer(n, seed=n)
    x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
    with nbody.NBody(n, "fp32_comp") as nb:
        nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, 0)
        a = nb.forces(x, m, 1.0, 0.01)
        _check(a, b, 0.01)
        # three steps (merges fused with the next kick) against three calls of
        # one step (merges of their own): the same operations
        run = []
        for calls in ([3], [1, 1, 1]):
            p, v, acc = to_dev(b.pos, cuda), to_dev(b.vel, cuda), a.clone()
            for k in calls:
                nb.step(p, v, m, 1.0, 0.01, 1e-3, k, acc, acc_valid=True)
            run.append((host(p), host(v), host(acc)))
        nb.sync()
    for p, q in zip(*run):
        assert np.array_equal(p, q)


def test_masses_in_the_log_domain(cuda):
    # variant 8 takes every pair as 2^(log2 m - 1.5 log2 r^2): masses over many
    # binades, zero and subnormal ones among them
    n = 600
    b = inputs.random_system(n, seed=4)
    rng = np.random.default_rng(5)
    mass = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-30, 30, n)
    mass[:3] = [0.0, 5e-310, 1.0]
    ref = oracle.accel(b.pos, mass, 1.0, 0.05)
    with nbody.NBody(n, "fp32_comp") as nb:
        nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, 8, 0)
        a = nb.forces(to_dev(b.pos, cuda), torch.as_tensor(mass, device=cuda), 1.0, 0.05)
        nb.sync()
    err = relerr_per_body(host(a), ref)
    assert np.sqrt(np.mean(err ** 2)) <= BOUND[0] and err.max() <= BOUND[1]


def test_packed_pairs_at_every_exponent(cuda):
    # pairs of bodies a 2^-8 of their coordinates apart, coordinates of both
    # signs with all 53 bits over 110 octaves and some zero: their difference is
    # only as good as x = h + l, so a wrong bit of either half shows
    rng = np.random.default_rng(11)
    npair = 512
    e = rng.integers(-50, 60, (npair, 1)).astype(float)
    p = rng.choice([-1.0, 1.0], (npair, 3)) * (1.0 + rng.integers(0, 1 << 52, (npair, 3)) * 2.0 ** -52)
    p *= 2.0 ** e
    p[::7, 1] = 0.0
    q = p + rng.choice([-1.0, 1.0], (npair, 3)) * 2.0 ** (e - 8) * rng.uniform(0.5, 1.0, (npair, 3))
    pos = np.stack([p, q], 1).reshape(-1, 3)
    mass = np.repeat(2.0 ** (2 * e[:, 0]), 2)  # accelerations of order 1
    with nbody.NBody(2 * npair, "fp32_comp") as nb:
        nb.batch_plan(np.arange(0, 2 * npair + 1, 2))
        a = host(nb.forces_batched(to_dev(pos, cuda), to_dev(mass, cuda), 1.0, 0.0))
        nb.sync()
    d = q - p
    want = mass[::2, None] * d / ((d * d).sum(1) ** 1.5)[:, None]
    # coordinates to 2^-48 of themselves, 2^-40 of the difference; the pair in float32
    for got, w in ((a[::2], want), (a[1::2], -want)):
        assert (np.abs(got - w).max(1) <= 1e-5 * np.abs(w).max(1)).all()


@pytest.mark.parametrize("variant,split,parts", [
    (5, 5, 5), (21, 5, 5), (22, 5, 5), (22, 20, 20)])  # splits by tiles and by bodies
def test_merging_splits_rounds_no_more_than_float64(cuda, variant, split, parts):
    # one body with mass in each part of the j range, so that every part's sum
    # is one float32 pair term, which a call with only that body's mass shows:
    # their sum must be as good as parts - 1 float64 additions (terms over 28
    # octaves, whose sum takes more bits than two float32 hold)
    n = 5120
    rng = np.random.default_rng(variant)
    b = inputs.random_system(n, seed=7)
    at = ((np.arange(parts) + 0.5) * n / parts).astype(int)
    mass = np.zeros(n)
    mass[at] = 2.0 ** -rng.uniform(0, 28, parts)
    x = to_dev(b.pos, cuda)
    with nbody.NBody(n, "fp32_comp") as nb:
        nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, split)
        got = host(nb.forces(x, to_dev(mass, cuda), 1.0, 0.05)).astype(np.longdouble)
        want, size = np.zeros_like(got), np.zeros_like(got)
        for k in at:
            one = np.zeros(n)
            one[k] = mass[k]
            t = host(nb.forces(x, to_dev(one, cuda), 1.0, 0.05)).astype(np.longdouble)
            assert np.array_equal(t, t.astype(np.float32))
            want += t
            size += np.abs(t)
        nb.sync()
    assert (np.abs(got - want) <= (parts - 1) * 2.0 ** -53 * size).all()


@pytest.mark.parametrize("prec", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("variant,split,n", [(23, 1, 500), (24, 8, 5003), (5, 16, 5003), (21, 9, 5003),
                                             (22, 20, 9001), ("batch", 0, 61)])
def test_sums_past_float32_of_parts_within_it(cuda, prec, variant, split, n):
    # two clouds pull at one another with sums of up to 6e38, above float32's range
    # (3.4e38), of which each of four parts or more (splits, warps or lanes, the
    # bodies in random order) adds a fourth or so; G brings them back to 6e8
    rng = np.random.default_rng(n)
    pos = rng.uniform(-0.5, 0.5, (n, 3))
    pos[: n // 2, 0] += 3.0
    pos = pos[rng.permutation(n)]
    mass = rng.uniform(0.5, 1.5, n)
    mass *= 6e38 / np.abs(oracle.accel(pos, mass, 1.0, 1.0)).max()
    x, m = to_dev(pos, cuda), to_dev(mass, cuda)
    with nbody.NBody(n, prec) as nb:
        if variant == "batch":
            nb.batch_plan([0, n])
            a = host(nb.forces_batched(x, m, 1e-30, 1.0))
        else:
            nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, split)
            a = host(nb.forces(x, m, 1e-30, 1.0))
        nb.sync()  # raises if anything is not finite
    err = relerr_per_body(a, oracle.accel(pos, mass, 1e-30, 1.0))
    assert np.sqrt(np.mean(err ** 2)) <= BOUND[0] and err.max() <= BOUND[1]


@pytest.mark.parametrize("prec", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("variant,split,n", [(23, 8, 1280), (24, 8, 5120), (21, 9, 7680), (22, 7, 7680), (5, 5, 7600)])
def test_a_body_next_to_the_origin_without_softening(cuda, prec, variant, split, n):
    # the slots past the end of a part of the j range hold massless bodies, which
    # must not lie so close to a body that 1 / r^3 overflows: one body 3e-20 from the
    # origin, its tile's coordinates relative to the origin itself (bodies in
    # opposite pairs)
    rng = np.random.default_rng(8)
    half = rng.uniform(-1.0, 1.0, (n // 2, 3))
    pos = np.stack([half, -half], 1).reshape(-1, 3)
    pos[0], pos[1] = (3e-20, 0.0, 0.0), (0.3, -0.2, 0.4)
    mass = rng.uniform(0.5, 1.5, n) / n
    with nbody.NBody(n, prec) as nb:
        nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, split)
        a = host(nb.forces(to_dev(pos, cuda), to_dev(mass, cuda), 1.0, 0.0))
        nb.sync()
    err = relerr_per_body(a, oracle.accel(pos, mass, 1.0, 0.0))
    assert np.sqrt(np.mean(err ** 2)) <= BOUND[0] * 10


@pytest.mark.parametrize("prec,variant", [("fp32_comp", 22), ("fp32", 21)])
def test_records_between_the_two_half_kicks(cuda, prec, variant):
    # with split forces a launch ends one step and opens the next: what it records
    # in between is the state that single-step calls return
    n, dt = 9001, 1e-3
    b = inputs.plummer(n, seed=12)
    m = to_dev(b.mass, cuda)
    with nbody.NBody(n, prec) as nb:
        nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, 0)
        x, v, acc = to_dev(b.pos, cuda), to_dev(b.vel, cuda), torch.empty_like(to_dev(b.pos, cuda))
        rx, rv = (torch.empty((4, n, 3), dtype=torch.float64, device=cuda) for _ in range(2))
        nb.rollout(x, v, m, 1.0, 0.01, dt, 3, acc, 1, rx, rv)
        p, q, a = to_dev(b.pos, cuda), to_dev(b.vel, cuda), torch.empty_like(acc)
        for k in range(4):
            assert np.array_equal(host(rx[k]), host(p)) and np.array_equal(host(rv[k]), host(q))
            if k < 3:
                nb.step(p, q, m, 1.0, 0.01, dt, 1, a, acc_valid=k > 0)
        assert np.array_equal(host(x), host(p)) and np.array_equal(host(acc), host(a))
        nb.sync()

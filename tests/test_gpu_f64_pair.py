"""float64 forces: the integer pair terms at the edges of their ranges; j-splits of equal body counts."""
import numpy as np
import pytest

import oracle
from paper_1211_2292_gb300 import inputs, nbody
from helpers import host, relerr_per_body, to_dev

pytestmark = pytest.mark.gpu


def _exact(pos, mass, eps):
    """Extended-precision sums and, per body, the sum of the terms' magnitudes."""
    p, m, e = pos.astype(np.longdouble), mass.astype(np.longdouble), np.longdouble(eps)
    d = p[None, :, :] - p[:, None, :]
    r2 = (d * d).sum(2) + e * e
    own = r2 == e * e if eps == 0.0 else np.zeros_like(r2, dtype=bool)
    s2 = np.where(own, np.longdouble(1), r2)
    t = np.where(own, 0, m[None, :] / (s2 * np.sqrt(s2)))[:, :, None] * d
    return t.sum(1), np.abs(t).sum(1)


def _check(cuda, pos, mass, eps, split=0, variant=0):
    n = len(mass)
    x, m = to_dev(pos, cuda), to_dev(mass, cuda)
    with nbody.NBody(n, "fp64") as nb:
        nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, split)
        a = host(nb.forces(x, m, 1.0, eps))
        nb.sync()
    ref, size = _exact(pos, mass, eps)
    # a pair's term: differences and r^2 3 x 2^-53 (1.5 fold for the power), the
    # factor and its product below 5 x 2^-53; n additions of 2^-53 each
    assert (np.abs(a - ref) <= (n + 10) * 2.0 ** -53 * size).all()


@pytest.mark.parametrize("variant", range(4))
@pytest.mark.parametrize("n", [1, 2, 15, 17, 127, 129, 257, 400])
def test_even_splits_and_tile_edges(cuda, n, variant):
    b = inputs.random_system(n, seed=n)
    for eps, split in ((0.01, 0), (0.0, 0), (0.01, 1), (0.0, 3)):
        _check(cuda, b.pos, b.mass, eps, split, variant)


@pytest.mark.parametrize("scale", [0, -329, -331, 328, 331])
@pytest.mark.parametrize("rel", [0.0, 1e-6, 1.0, 1e5])
def test_exponents_of_differences_and_softening(cuda, scale, rel):
    # separations over 80 octaves, equal and zero coordinates, massless and
    # negative masses, around the exponents at which the general form takes over
    rng = np.random.default_rng(5)
    n = 70
    pos = rng.uniform(-1, 1, (n, 3)) * np.ldexp(1.0, -rng.integers(0, 80, (n, 3)))
    pos[:10, 1] = 0.0
    pos[10:20, 2] = pos[5, 2]
    pos[20] = pos[21]
    mass = rng.uniform(0.1, 1.0, n)
    mass[::7] = 0.0
    mass[3] = -mass[3]
    # |a| ~ m 2^(-2 scale): scaled so that the sums stay in range
    mass = np.ldexp(mass, scale)
    _check(cuda, np.ldexp(pos, scale), mass, float(np.ldexp(rel, scale)))


@pytest.mark.parametrize("variant", range(3))
@pytest.mark.parametrize("n", [2, 15, 127, 129, 257, 3001])
def test_double_float_even_splits(cuda, n, variant):
    # the mode's bound, 1e-12 per body
    b = inputs.random_system(n, seed=n)
    x, m = to_dev(b.pos, cuda), to_dev(b.mass, cuda)
    for eps, split in ((0.05, 0), (0.05, 1), (0.05, 3)):
        with nbody.NBody(n, "df64") as nb:
            nb.tune_set(nbody.KIND_FORCE, 0, 1 << 40, variant, split)
            a = host(nb.forces(x, m, 1.0, eps))
            nb.sync()
        assert relerr_per_body(a, oracle.accel(b.pos, b.mass, 1.0, eps)).max() <= 1e-12


def test_many_small_terms_beside_a_large_one(cuda):
    # 1e5 terms of one sign, 2^-28 of the largest: rounded to 2^-55 of it at most
    # each (300 units of 2^-54 together by chance, 1.6e-14); a quarter of a unit
    # in one direction would make 1.4e-12
    rng = np.random.default_rng(3)
    n = 100001
    pos = rng.uniform(-0.2, 0.2, (n, 3)) + np.array([1.0, 1.0, 1.0])
    pos[0], pos[1] = 0.0, 2.0 ** -14 * np.array([0.6, 0.5, 0.7])
    mass = rng.uniform(0.5, 1.5, n)
    x, m = to_dev(pos, cuda), to_dev(mass, cuda)
    with nbody.NBody(n, "fp64") as nb:
        a = host(nb.forces(x, m, 1.0, 0.0))[0]
        nb.sync()
    d, w = pos[1:].astype(np.longdouble), mass[1:].astype(np.longdouble)
    r2 = (d * d).sum(1)
    t = (w / (r2 * np.sqrt(r2)))[:, None] * d
    assert (np.abs(a - t.sum(0)) <= 1e-13 * np.abs(t).max(0)).all()


def test_large_terms_that_cancel(cuda):
    # 40 bodies, each between two others at the same distance on either side,
    # whose terms (2^28 and more) cancel to the bit; then 1e5 others.  Only the
    # terms of the pairs' own tile (128 bodies) are rounded to 2^-55 of the
    # largest: 0.29 x 2^-55 rms each, so 128 of them 2^-53.3, six times that
    # 2^-50.7.  The others' own errors lie far below: 1e5 terms of some 1 each, to
    # 2^-53 of themselves and, in 800 tiles, of their sum, 2^-11 of a pair's term.
    rng = np.random.default_rng(9)
    k, n = 40, 100001
    mid = rng.integers(1 << 19, 1 << 20, (k, 3)) * 2.0 ** -20
    d = rng.integers(1 << 11, 1 << 12, (k, 3)) * 2.0 ** -26 * rng.choice([-1.0, 1.0], (k, 3))
    pos = rng.uniform(-1.5, -0.5, (n, 3))
    mass = rng.uniform(0.5, 1.5, n)
    pos[0:3 * k:3], pos[1:3 * k:3], pos[2:3 * k:3] = mid - d, mid, mid + d
    mass[0:3 * k:3] = mass[2:3 * k:3] = rng.uniform(1.0, 2.0, k)
    with nbody.NBody(n, "fp64") as nb:
        a = host(nb.forces(to_dev(pos, cuda), to_dev(mass, cuda), 1.0, 0.0))
        nb.sync()
    p, m = pos.astype(np.longdouble), mass.astype(np.longdouble)
    for i in range(1, 3 * k, 3):
        s = np.delete(p, i, 0) - p[i]
        r2 = (s * s).sum(1)
        t = (np.delete(m, i) / (r2 * np.sqrt(r2)))[:, None] * s
        big = np.abs(t[i - 1])
        rest = np.delete(t, [i - 1, i], 0).sum(0)
        assert (np.abs(a[i] - rest) <= 2.0 ** -50.7 * big).all()

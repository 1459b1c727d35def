"""CPU check of the bounds behind the Jacobian walk's loops (SlabRay::t0, t1).

Each axis' crossings are walked in a loop of its own, and a pair of crossings is seen
in two loops: crossing k of a minor axis as a position along the dominant axis (or the
other minor one), and the other's crossing as a coordinate of the minor axis.  Both are
sums of 32.32 fixed-point starts and steps, rounded differently.  A pair whose minor
crossing lies further than t0 (t1) from the other axis' plane has to be ordered alike
in both; closer ones are settled from FP64 positions.  Replayed here in integers
against exact fractions, with the start and step formulas of slab_setup, over random
rays and over the largest counts and spacings that the walk takes."""
import random
from fractions import Fraction as Fr

import pytest

ONE = 1 << 32


def mul_frac(x, m):  # x (0.32) times m (32.32), as two rounded-down halves
    return x * (m >> 32) + ((x * (m & (ONE - 1))) >> 32)


def case(rng, most):
    r20 = Fr(1) if rng.random() < 0.1 else Fr(rng.choice([1, 3, 10, 1000, 60000])) * Fr(rng.randrange(10**8, 10**9), 10**8) / 10 + 1
    r20 = min(r20, Fr(65535))
    E0, E2 = (Fr(rng.randrange(ONE * 4096), ONE * 4096) for _ in range(2))
    cnt2 = rng.randrange(1, most)
    return r20, E0, E2, max(1, min(most, int(cnt2 / r20))), cnt2


@pytest.mark.parametrize("most", [8, 600, 8000])
def test_two_views_of_a_pair_differ_by_less_than_the_bound(most):
    rng = random.Random(most)
    far = Fr(3 * most, 4096)
    for _ in range(1500):
        r20, x0, x2, cnt0, cnt2 = case(rng, most)
        off = rng.randrange(-1, 2)  # float-float start values: 2^-32 voxel either way
        E0, E2 = max(int(x0 * ONE) + off, 0), max(int(x2 * ONE) - off, 0)
        mdX, dy = round(r20 * ONE), int(ONE / r20)
        dy = min(dy, ONE - 1)
        t0 = int(2 * (cnt2 + 16 + far) * r20 + cnt0 + 16 + far)
        mX = E2 + (mdX - mul_frac(E0, mdX))
        Y = E0 + (dy - ((E2 * dy) >> 32))
        for k in {0, cnt0 - 1, rng.randrange(cnt0)}:
            # the dominant plane next to the crossing, and the crossing as that plane sees it
            exact = x2 + r20 * (1 - x0 + k)
            for q in {int(exact), int(exact) + 1}:
                m = q - 1  # dominant crossing
                if not 0 <= m < cnt2:
                    continue
                pos = mX + k * mdX - q * ONE           # of the crossing after the plane, in the minor loop
                seen = (k + 1) * ONE - (Y + m * dy)    # of the plane before the crossing, in voxels
                if abs(pos) >= t0:
                    assert (pos > 0) == (seen > 0), (r20, x0, x2, k, q)
                    assert (pos > 0) == (exact > q)

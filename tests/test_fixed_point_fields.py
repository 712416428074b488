"""The integer arithmetic of staged fields (csrc/pic_fixed64.cuh, pic_field64.cuh) in
exact integers, on the CPU: the conversion of doubles at a tile's or block's scale, of
offsets at 2^63, the range of the gather's sums at 60 bits, the range and the error of
the smoothing, and the rounding of one term of a difference to the other's scale.
"""
import random
import struct
from fractions import Fraction as F

from .test_fixed_point_split import mul, spline, split

BITS, MIN_EXP = 60, 82


def bits(v):
    return struct.unpack("<q", struct.pack("<d", v))[0]


def field_fixed(v, emax):
    b = bits(v)
    e = (b >> 52) & 0x7FF
    m = (b & 0xFFFFFFFFFFFFF) | 0x10000000000000
    assert m << 8 < 1 << 64
    X = (m << 8) >> min(emax - e, 63)
    X = 0 if e == 0 else (X + 1) >> 1
    return -X if b < 0 else X


def test_staged_fields_round_to_nearest_at_the_scale_of_the_largest():
    rng = random.Random(1)
    for emax in (MIN_EXP, 200, 1023, 1700, 2046):
        k = BITS - 1 + 1023 - emax
        assert -966 <= k <= 1000
        for drop in (0, 1, 6, 7, 8, 9, 30, 59, 60, 61, 62, 63, 70):
            for frac in (0, 1, (1 << 52) - 1, rng.randrange(1 << 52)):
                e = emax - drop
                v = struct.unpack("<d", struct.pack("<q", (e << 52) | frac))[0]
                want = F(v) * F(2) ** k
                for s in (1, -1):
                    got = field_fixed(s * v, emax)
                    assert abs(got) <= 1 << BITS
                    assert abs(got - s * want) <= F(1, 2)
                    if drop <= 7:  # 53 bits fit
                        assert got == s * want
        assert field_fixed(0.0, emax) == field_fixed(-0.0, emax) == field_fixed(5e-324, emax) == 0


def test_offsets_are_cut_at_the_last_unit():
    for o in (0.0, 5e-324, 2.0 ** -64, 2.0 ** -63, 1.5 * 2.0 ** -62, 0.1, 0.5, 1 - 2.0 ** -53):
        b = bits(o)
        got = (((b & 0xFFFFFFFFFFFFF) | 0x10000000000000) << 10) >> min(1022 - (b >> 52), 63)
        assert got == F(o) * 2 ** 63 // 1 and 0 <= got < 1 << 63


def gather(xs, wde):
    """One node of the third axis as gather64 forms it; the accumulators' range is checked."""
    H, M, N = 0, 1 << 30, 0
    for i in range(16):
        (xh, xl), (wh, wl) = split(xs[i]), split(wde[i])
        H, M, N = H + xh * wh, M + xh * wl, N + xl * wh
        assert max(abs(H), abs(M), abs(N)) < 1 << 63
        if i % 8 == 7:
            H, M = H + (M >> 32), M & 0xFFFFFFFF
    assert abs(M + N) < 1 << 63
    return 2 * H + ((M + N) >> 31)


def test_gather_sums_at_60_bits():
    rng = random.Random(2)
    big = 1 << BITS
    for trial in range(300):
        a, b = (spline(rng.randrange((1 << 63) - 1024) - (1 << 62), 63) for _ in range(2))
        wde = [2 * mul(x, y) for x in a for y in b]
        assert sum(split(w)[0] for w in wde) <= (1 << 31) + 16
        xs = [rng.choice((-big, big)) if trial % 3 == 0 else rng.randrange(-big, big + 1) for _ in wde]
        # 16 dropped products of at most a quarter unit (half at twice the scale) and the shift
        assert abs(gather(xs, wde) - F(sum(x * w for x, w in zip(xs, wde)), 1 << 63)) <= 9
        assert gather([0] * 16, wde) == 0
    # the largest cross sums that splits of these sizes can have
    for xh, wl in ((1 << 28, -(1 << 31)), (-(1 << 28), (1 << 31) - 1)):
        assert abs((1 << 30) + 8 * xh * wl) < 1 << 63 and abs((1 << 32) + 8 * xh * wl) < 1 << 63
    assert (1 << 32) + (1 << 31) * ((1 << 31) + 16) < 1 << 63
    assert 4 * (1 << 28) * (1 << 31) + (1 << 31) * ((1 << 31) + 4) + (1 << 30) < 1 << 63  # over the third axis


def smoothing(rb, rc):
    """Weights of the 3x3 smoothing: centre, two pairs of edges, corners."""
    g = rb * rc / 48
    b1, b2 = rb / 8 - 2 * g, rc / 8 - 2 * g
    return 1 - 2 * b1 - 2 * b2 - 4 * g, b1, b2, g


def test_smoothing_stays_in_range_and_close_to_exact():
    rng = random.Random(3)
    big = 1 << BITS
    for rb, rc in ((F(1), F(1)), (F(1), F(1, 9)), (F(1, 10 ** 6), F(1, 10 ** 6)), (F(1, 64), F(1, 64))):
        ws = [int(w * (1 << 62)) for w in smoothing(rb, rc)]
        for weights in (ws, [1 << 62, 0, 0, 0]):
            for trial in range(200):
                s = rng.choice((-1, 1))
                x = [s * big] * 9 if trial < 20 else [rng.randrange(-big, big + 1) for _ in range(9)]
                terms = [x[0], x[1] + x[2], x[3] + x[4], sum(x[5:])]
                H, M, l = 0, 1 << 28, 0
                for t, w in zip(terms, weights):
                    (th, tl), (wh, wl) = split(t), split(w)
                    H, M = H + th * wh, M + th * wl + tl * wh
                    l += (tl >> 17) * (wl >> 17)
                    assert abs(M) < 1 << 63 and abs(l) <= 1 << 30
                M += 4 * l
                got = (H << 3) + (M >> 29)
                assert abs(M) < 1 << 63 and abs(got) <= 1 << 61  # at twice the scale of x
                want = F(sum(t * w for t, w in zip(terms, weights)), 1 << 61)
                # the shift; four low products with 15 of 32 bits each: 2^-14 of at most 2 units
                assert abs(got - want) <= F(1, 2) + F(1, 1 << 10)


def test_products_with_the_step_per_cell():
    rng = random.Random(4)
    for K, xmax, wmax in ((1, 1 << 62, 1 << 62), (2, 1 << 61, 1 << 62)):  # magnetic, electric
        for _ in range(2000):
            x, w = rng.randrange(-xmax, xmax + 1), rng.randrange(wmax + 1)
            if rng.random() < 0.1:
                x, w = rng.choice((-xmax, xmax)), wmax
            (xh, xl), (wh, wl) = split(x), split(w)
            H, M = xh * wh, (1 << (31 - K)) + xh * wl + xl * wh
            assert abs(M) < 1 << 63
            got = (H << K) + (M >> (32 - K))
            assert abs(got) <= 1 << 61
            assert abs(got - F(x * w, 1 << (64 - K))) <= F(1, 2) + F(1 << K, 4)  # the shift and the dropped product


def coarser(a, sh):
    r = min(sh, 62)
    x = a + ((1 << r) >> 1)
    assert abs(x) < 1 << 63
    return x >> r


def test_the_finer_term_of_a_difference_rounds_to_nearest():
    rng = random.Random(5)
    top = (1 << 61) - 1
    for sh in (0, 1, 2, 20, 59, 60, 61, 62, 63, 900):
        for a in (0, 1, -1, top, -top, rng.randrange(-top, top), rng.randrange(-top, top)):
            assert abs(coarser(a, sh) - F(a, 1 << sh)) <= F(1, 2)
    errs = [coarser(a, 20) - a / 2 ** 20 for a in (rng.randrange(-(1 << 40), 1 << 40) for _ in range(20000))]
    assert abs(sum(errs) / len(errs)) < 0.02  # 0.29 / sqrt(20000) = 0.002

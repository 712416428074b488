"""The arithmetic of the FP64 push (csrc/pic_fixed64.cuh) in exact integers, on
the CPU: centred splits at 32 bits, the range of the cross products' sum, the
error of products, the shape factors, and the sums of current words.
"""
import random
from fractions import Fraction as F

M64 = 1 << 64
THIRD = (0x55555555, 0x55555555)


def signed(v, bits=64):
    v &= (1 << bits) - 1
    return v - (1 << bits) if v >> (bits - 1) else v


def split(x):
    hi, lo = signed(((x + 0x80000000) % M64) >> 32, 32), signed(x, 32)
    assert (hi << 32) + lo == x
    return hi, lo


def dot(pairs, rounding):
    """sum x w / 2^64 and the largest |M| seen."""
    H, M = 0, rounding
    for x, w in pairs:
        (xh, xl), (wh, wl) = split(x), split(w)
        H += xh * wh
        M += xh * wl + xl * wh
        assert abs(M) < 1 << 63
    return H + (M >> 32), 2 * H + (M >> 31)


def mul(x, w):
    return dot([(x, w)], 0)[0]


def spline(U, K):
    one48 = 192153584101141163 if K == 63 else 96076792050570581
    sh = 63 - K
    q = mul(U, U)
    c = mul(U, q)
    c3 = mul(c, (THIRD[0] << 32) + THIRD[1])
    e, u3 = q >> (sh + 1), U >> (3 + sh)
    e0, e1 = one48 + e, (1 << (K - 1)) - one48 - e
    o0, o1 = u3 + (c3 if sh else 2 * c3), u3 + (U >> (1 + sh)) - (c if sh else 2 * c)
    return [e0 - o0, e1 - o1, e1 + o1, e0 + o0]


def exact_spline(t):
    s = 1 - t
    return [s ** 3 / 6, F(2, 3) - t * t + t ** 3 / 2, F(2, 3) - s * s + s ** 3 / 2, t ** 3 / 6]


def test_shape_factors_are_within_a_few_units_and_sum_to_one():
    rng = random.Random(1)
    top = (1 << 63) - 1024  # the largest double below one
    ts = [0, 1, 1 << 20, 1 << 62, (1 << 62) - 1, top, top - 1024] + [rng.randrange(top) for _ in range(2000)]
    for T in ts:
        for K in (62, 63):
            w = spline(T - (1 << 62), K)
            assert sum(w) == 1 << K
            # four truncated products and shifts of at most one unit each, twice where doubled
            assert max(abs(F(a) - b * (1 << K)) for a, b in zip(w, exact_spline(F(T, 1 << 63)))) <= 8


def test_gather_sums_stay_in_range_and_close_to_exact():
    rng = random.Random(2)
    for trial in range(300):
        t = [rng.randrange((1 << 63) - 1024) for _ in range(2)]
        a, b = (spline(v - (1 << 62), 63) for v in t)
        wde = [2 * mul(x, y) for x in a for y in b]
        big = (1 << 58) - 1
        xs = [rng.choice((-big, big)) if trial % 3 == 0 else rng.randrange(-big, big + 1) for _ in wde]
        got = dot(list(zip(xs, wde)), 1 << 30)[1]
        want = F(sum(x * w for x, w in zip(xs, wde)), 1 << 63)
        # 16 dropped products of at most a quarter unit (half at twice the scale) and the shift
        assert abs(got - want) <= 9
        assert dot([(0, w) for w in wde], 1 << 30)[1] == 0


def test_products_of_current_and_factors_round_without_bias():
    rng = random.Random(3)
    errs = []
    for _ in range(20000):
        P, A = rng.randrange(-(1 << 63) // 1001 * 1000, (1 << 63) // 1001 * 1000), rng.randrange(1 << 62)
        x = dot([(P, A)], 1 << 31)[0]
        errs.append(float(x - F(P * A, M64)))
    assert max(map(abs, errs)) <= 1.0
    assert abs(sum(errs) / len(errs)) < 0.02  # uniform on half a unit either way: sigma 0.29 / sqrt(20000) = 0.002
    assert dot([(0, 1 << 61)], 1 << 31)[0] == 0


def test_current_words_give_back_the_exact_sum():
    rng = random.Random(4)
    for n, top in ((1, 1 << 61), (2304, (1 << 62) // 2304), (2304, 1 << 40), (5, 3)):
        for sign in (-1, 1, 0):
            xs = [rng.randrange(-top, top + 1) if not sign else sign * rng.randrange(top + 1) for _ in range(n)]
            w = [sum(x >> s for x in xs) % (1 << 32) for s in (0, 20, 40)]
            a = signed(w[2], 32) << 20
            b = a + (w[1] - a) % (1 << 32)
            c = b << 20
            assert c + (w[0] - c) % (1 << 32) == sum(xs)
    # FP32: T >> 12 and T mod 2^32, n < 2^20 adds, |sum| < 2^42
    for n, top in ((6000, (1 << 42) // 6000), (7, 1 << 39)):
        ts = [rng.randrange(-top, top + 1) for _ in range(n)]
        hi, lo = signed(sum(t >> 12 for t in ts), 32), sum(ts) % (1 << 32)
        assert hi * 4096 + (lo - (hi << 12)) % (1 << 32) == sum(ts)

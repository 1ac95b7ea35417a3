"""Host model of the Montgomery arithmetic of csrc/field.cuh and of the NTT's lazy words.

Restates the kernels' PTX carry chains on 32-bit words with an explicit carry
flag and checks, on random and extreme words, that each gives the exact residue
and that no word the chains assume not to wrap does: the Montgomery tail after
a product and after a lazy sum, the fold of a small top word, the seventh-root
scaling identity of the chain, and the three-word values of csrc/ntt.cu.
"""
import random

P = 2**64 - 2**32 + 1
R = 2**64
RI = pow(R, -1, P)
M = 0xFFFFFFFF


def adc(a, b, c=0):
    s = a + b + c
    return s & M, s >> 32


def sbb(a, b, c=0):
    d = a - b - c
    return d & M, 1 if d < 0 else 0


def sar(x, n):
    x &= M
    return ((x - (1 << 32) if x >> 31 else x) >> n) & M


def words(x, n):
    return [(x >> (32 * k)) & M for k in range(n)]


def mont_tail(r, any_sum=False):
    m, e = adc(r[1], r[0])
    me, wrap = adc(m, 0, e)
    assert not wrap
    lo, f = adc(r[1], r[2], e)
    if any_sum:
        h, b = sbb(r[3], me)
        k = -b
        h, c = adc(h, f)
        k += c
    else:
        t, wrap = adc(r[3], 0, f)
        assert not wrap
        h, b = sbb(t, me)
        k = -b
    assert k in (-1, 0)
    lo, b = sbb(lo, k & M)
    h, _ = sbb(h, 0, b)
    return (h << 32) | lo


def fold_small(w0, w1, h):
    u, k = adc(w1, h)
    g = h + k
    u += k
    assert u <= M
    lo, b = sbb(w0, g)
    u, b = sbb(u, 0, b)
    assert not b
    return (u << 32) | lo


EDGE = [0, 1, 2, 3, M - 1, M, M + 1, P - 1, P, P + 1, R - 1, R - 2, R - M, R - M - 1, 1 << 63, (1 << 63) - 1,
        0x5555555555555555, 0xFFFFFFFF00000000]


def pairs(n=20000):
    rng = random.Random(5)
    yield from ((a, b) for a in EDGE for b in EDGE)
    for _ in range(n):
        yield rng.getrandbits(64), rng.getrandbits(64)
    for _ in range(n):  # both near 2^64: the tail's largest top words
        yield R - 1 - rng.getrandbits(rng.randint(1, 34)), R - 1 - rng.getrandbits(rng.randint(1, 34))


def test_montgomery_tail_of_a_product():
    for a, b in pairs():
        v = mont_tail(words(a * b, 4))
        assert v < R and v % P == a * b * RI % P


def test_montgomery_tail_of_a_sum():
    rng = random.Random(6)
    xs = [(1 << 128) - 1 - e for e in EDGE] + [rng.getrandbits(128) for _ in range(20000)]
    xs += [((1 << 128) - 1) ^ (rng.getrandbits(32) << (32 * rng.randrange(4))) for _ in range(20000)]
    for x in xs:
        v = mont_tail(words(x, 4), True)
        assert v < R and v % P == x * RI % P


def test_fold_of_a_small_top_word():
    rng = random.Random(7)
    for lo, h in pairs():
        h %= 1 << rng.randint(1, 31)
        v = fold_small(lo & M, lo >> 32, h)
        assert v < R and v % P == (lo + h * R) % P


def test_seventh_root_scaling():
    e = next(k for k in range(1, 8 * (P - 1), P - 1) if k % 7 == 0) // 7
    rng = random.Random(8)
    r6 = pow(R, 6, P)
    for _ in range(50):
        beta, nxt, z = (rng.randrange(1, P) for _ in range(3))
        lam = pow(nxt * beta * r6 % P, e, P)
        # f(lambda z) = lambda' beta z^7, f(x) = x^7 R^-6
        assert pow(lam * z, 7, P) * pow(r6, -1, P) % P == nxt * beta * pow(z, 7, P) % P


# three-word values l0 + l1 2^32 + t 2^64, t signed
def value(a):
    t = a[2] - (1 << 32) if a[2] >> 31 else a[2]
    return a[0] + (a[1] << 32) + t * R


def lz_reduce(a):
    l0, l1, t = a
    s = sar(t, 31)
    l1, c = adc(l1, t)
    k = (s + c) & M
    l1, g = (l1 + k) & M, (t + k) & M
    lo, b = sbb(l0, g)
    hi, _ = sbb(l1, sar(g, 31), b)
    return (hi << 32) | lo


def funnel_r(lo, hi, n):
    return (((hi << 32) | lo) >> n) & M


def lz_m48(a):
    w1, hl, e0 = (a[0] << 16) & M, funnel_r(a[0], a[1], 16), funnel_r(a[1], a[2], 16)
    q0, c = adc(hl, e0)
    q1 = (sar(a[2], 16) + c) & M
    w1, w2 = adc(w1, hl)
    w0, b = sbb(0, q0)
    w1, b = sbb(w1, q1, b)
    return w0, w1, (w2 - sar(q1, 31) - b) & M


def lz_m72(a):
    hl, hh, k = (a[0] << 8) & M, funnel_r(a[0], a[1], 24), funnel_r(a[1], a[2], 24)
    q0, c = adc(hl, hh)
    k1 = (k + c) & M
    w0, b = sbb(0, q0)
    w1, b = sbb(hl, k1, b)
    return w0, w1, (0 - sar(k1, 31) - b) & M


def lazies(bits, n=20000):
    rng = random.Random(9)
    lows = [0, 1, M, M << 32, R - 1, R - 2, 1 << 32, 1 << 63, 0xFFFF, 0xFFFF0000, (1 << 48) - 1, (1 << 48)]
    tops = [0, 1, -1, 2, -2, (1 << bits) - 1, -(1 << bits) + 1]
    for lo in lows:
        for t in tops:
            yield lo & M, lo >> 32, t & M
    for _ in range(n):
        lo = rng.choice(lows) ^ rng.getrandbits(rng.randint(1, 64))
        yield lo & M, lo >> 32, rng.randint(-(1 << bits) + 1, (1 << bits) - 1) & M


def test_lazy_reduction():
    for a in lazies(30):
        assert lz_reduce(a) % P == value(a) % P


def test_lazy_shift_products():
    for a in lazies(30):
        r = lz_m48(a)
        assert value(r) % P == value(a) * (1 << 48) % P and abs(value(r) >> 64) <= 2
    for a in lazies(22):
        r = lz_m72(a)
        assert value(r) % P == value(a) * (1 << 72) % P and abs(value(r) >> 64) <= 2

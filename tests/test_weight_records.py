"""The bound on the integer weight records (CPU, a model of the protocol): no lane
copy's record may hold more than 65,535 products.  Eight warps add batches of up
to 4,096 products to one record (one lane copy, every pair in one bin), each looks
at the record's counter when another batch would take it past its share, and
flushes when the counter says more than is left over.  A scheduler that may stop
any warp between any two of its shared-memory operations for as long as it likes
must not bring a record past the bound; taking the counters of all entries before
their records, as a flush in two passes does, must.  No product is lost: a flush may
take a quad's counts and leave its products, added later, to a flush that finds no
count beside them."""

import random
from fractions import Fraction

import pytest

LIMIT, WARPS, QUAD, BATCH_QUADS = 65535, 8, 256, 16      # one lane copy: 32 lanes x 8 pairs a quad
KEEP = LIMIT // 4                                        # what a look may leave
SHARE = (LIMIT - KEEP) // WARPS
FULL = KEEP - 2 * QUAD * WARPS                           # flush past it (16 slots a lane in flight)
CLAIM = 1 << 24


class Cta:
    def __init__(self):
        self.count = self.record = self.most = 0
        self.counts_out = self.products_out = 0


def _warp(c, two_passes):
    """One step per yield: a quad's counters, a quad's products, a look, and the
    operations of a flush."""
    share = 0
    while True:
        share += QUAD * BATCH_QUADS
        if share > SHARE:
            look = c.count & (CLAIM - 1)
            yield
            if look > FULL:
                if two_passes:
                    n, c.count = c.count, 0
                    for _ in range(100):                  # the other entries' counters
                        yield
                    c.products_out += c.record
                    c.record = 0
                    c.counts_out += n
                else:
                    n = c.count
                    c.count += CLAIM
                    n = 0 if n >= CLAIM else n
                    yield
                    c.products_out += c.record
                    c.record = 0
                    yield
                    c.count -= CLAIM + n
                    c.counts_out += n
                yield
            share = QUAD * BATCH_QUADS
        for _ in range(BATCH_QUADS):
            c.count += QUAD
            yield
            c.record += QUAD
            c.most = max(c.most, c.record)
            yield


def _run(seed, two_passes, steps=60_000):
    rng = random.Random(seed)
    c = Cta()
    warps = [_warp(c, two_passes) for _ in range(WARPS)]
    asleep = [0] * WARPS
    for t in range(steps):
        w = rng.randrange(WARPS)
        while asleep[w] > t and any(a <= t for a in asleep):
            w = (w + 1) % WARPS
        next(warps[w])
        if rng.random() < 0.02:
            asleep[w] = t + int(rng.expovariate(1.0 / 400.0))
    return c


@pytest.mark.parametrize("seed", range(12))
def test_no_record_passes_the_bound(seed):
    c = _run(seed, two_passes=False)
    assert c.most <= LIMIT
    assert c.products_out > 20 * LIMIT                     # it flushed many times
    # what was taken out and what is left agree, but for the quads in flight
    assert abs((c.counts_out + (c.count & (CLAIM - 1))) - (c.products_out + c.record)) <= QUAD * WARPS + LIMIT


@pytest.mark.parametrize("seed", range(40))
def test_no_product_is_lost(seed):
    """A rare entry of a histogram that is flushed for others: one quad's counts and
    products, flushes in between at any step, the last one after all warps stopped."""
    rng = random.Random(seed)
    c = Cta()

    def quads(k):
        for _ in range(k):
            c.count += QUAD
            yield
            c.record += QUAD
            yield

    def flush():
        if c.count == 0 and c.record == 0:                 # nothing to take
            return
        n = c.count
        c.count += CLAIM
        n = 0 if n >= CLAIM else n
        yield
        c.products_out += c.record
        c.record = 0
        yield
        c.count -= CLAIM + n
        c.counts_out += n

    total = rng.randint(1, 3)
    live = [quads(1) for _ in range(total)] + [flush() for _ in range(3)]
    while live:
        g = rng.choice(live)
        if next(g, "done") == "done":
            live.remove(g)
    for _ in flush():
        pass
    assert c.products_out == total * QUAD and c.counts_out == total * QUAD
    assert c.count == c.record == 0


def test_the_bound_of_the_constants():
    assert BATCH_QUADS * QUAD <= SHARE and KEEP + WARPS * SHARE <= LIMIT
    assert LIMIT * 0xFFFF < 2 ** 32                        # 16-bit pieces
    assert LIMIT * 2 ** 16 < 2 ** 32                       # top piece of products up to 2^48
    assert LIMIT * 2 ** 48 < 2 ** 64                       # the record's sum
    assert LIMIT + WARPS * 2 * QUAD < CLAIM


def test_counters_taken_before_the_records_pass_it():
    assert max(_run(seed, two_passes=True).most for seed in range(12)) > LIMIT


def test_exact_sums_without_carries():
    """A CTA's sums: low + high 2^32 in two 64-bit words that wrap on their own;
    products may be taken off again.  The conversion rounds at most twice."""
    m64, rng = 2 ** 64 - 1, random.Random(3)

    def signed(v):
        return v - 2 ** 64 if v >> 63 else v

    for _ in range(200):
        f, exact = [0, 0], 0
        for _ in range(rng.randint(1, 400)):
            t = rng.randint(0, LIMIT * 2 ** 48 * 32 if rng.random() < 0.5 else 2 ** 48)
            sign = -1 if t < 2 ** 48 and exact > t and rng.random() < 0.5 else 1
            lo, hi = t & 0xFFFFFFFF, t >> 32
            f[0], f[1] = (f[0] + sign * lo) & m64, (f[1] + sign * hi) & m64
            exact += sign * t
        lo = signed(f[0])
        hi = signed(f[1]) + (lo >> 32)
        assert hi >= 0 and (hi << 32) + (lo & 0xFFFFFFFF) == exact
        w = Fraction(float(Fraction(float(hi)) * 2 ** 32 + (lo & 0xFFFFFFFF)))
        assert abs(w - exact) <= Fraction(exact, 2 ** 52)

"""CPU model of the strided sweeps' input ring: for every line length, segment
cut, window and chunk length, each position the segment solve reads is inside
the line's loaded range, its chunk has been waited for, and its slot has not
been given to a later chunk; an aligned ring's output chunk reads exactly one
chunk.  And the FP64 kick's nearer sine and cosine series against 50-digit
values: within a quarter of the unit roundoff over their range, not at four
times it."""
import pytest


def ring(n, tb, te, W, B):
    """One segment [tb, te) of a line of n interior nodes; the calls are solve_segment's."""
    lead = 2 * W + 4
    aligned = -lead % B <= 4
    chunks = 3 if aligned else 4
    e, tw = min(te + W, n), tb - (W + 1) if tb > W + 1 else 0
    first, limit = tw - 1, e + 2
    s0 = first
    if aligned:
        s0 = tb + W + 2 - -(-lead // B) * B
        if first > s0:
            s0 += (first - s0) // B * B
    issued, ready, loaded = 0, 0, set()

    def fill(upto):
        nonlocal issued
        while issued < upto and s0 + issued * B < limit:
            loaded.update(p for p in range(s0 + issued * B, s0 + (issued + 1) * B) if max(first, 0) <= p < n)
            issued += 1

    def need(end):
        nonlocal ready
        c = (end - 1 - s0) // B
        if c < ready:
            return
        assert c < issued <= c + 4
        ready = c + 1
        fill(c + 3)

    def val(p):
        c = (p - s0) // B
        assert 0 <= c < ready and c > issued - 1 - chunks, (n, tb, te, W, B, p)
        assert not 0 <= p < n or p in loaded

    fill(3)
    if tw > 0:
        need(tw)
        val(tw - 1)
    need(tw + 1)
    val(tw)
    need(tw + 2)
    val(tw + 1)
    for t in range(tw, tb):
        need(t + 3)
        val(t + 2)
    for q in range(min(W, e - tb)):
        need(tb + q + 3)
        val(tb + q + 2)
    t0 = tb
    while t0 + B + W <= e:
        need(t0 + W + 2 + B)
        assert not aligned or (t0 + W + 2 - s0) % B == 0
        for q in range(B):
            val(t0 + W + 2 + q)
        t0 += B
    need(e + 2)
    for q in range(W, min(B + W, e - t0)):
        val(t0 + q + 2)


@pytest.mark.parametrize("W", [4, 8, 16])
@pytest.mark.parametrize("B", [8, 16])
def test_ring_reads_what_is_loaded(W, B):
    for n in list(range(1, 70)) + [126, 127, 128, 158, 318, 478]:
        ring(n, 0, n, W, B)
        for seg in (1, 3, 5, 8, 9, 13, 16, 24, 64, 104, 128):
            for tb in range(0, n, seg):
                ring(n, tb, min(n, tb + seg), W, B)


def test_near_series_bounds():
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 50
    quarter = mp.mpf(2) ** -55

    def worst(bound):
        sn = cs = mp.mpf(0)
        for i in range(1, 201):
            x = mp.mpf(bound) * i / 200
            s = sum((-1) ** k * x ** (2 * k + 1) / mp.factorial(2 * k + 1) for k in range(4))  # through x^7
            c = sum((-1) ** k * x ** (2 * k) / mp.factorial(2 * k) for k in range(4))  # through x^6
            sn, cs = max(sn, abs(s / mp.sin(x) - 1)), max(cs, abs(c - mp.cos(x)))
        return sn, cs

    assert max(worst("0.03")) <= quarter
    assert max(worst("0.12")) > quarter

"""CPU model of the row passes' butterfly assignment (mirror pairs in registers).

For every row length the first-stage and last-stage butterflies of the threads
must cover the stage once, and a butterfly and its mirror must be in one thread
or in one warp, so that each pair of columns meets in registers exactly once.
"""

import pytest

LENGTHS = [64, 128, 256, 512, 1024, 2048, 4096, 8192]


def radix(L, ns):
    return 16 if L // ns >= 16 else L // ns


def last_ns(L):
    ns = 1
    while ns * radix(L, ns) < L:
        ns *= radix(L, ns)
    return ns


def neg(T, g):
    """Butterfly of thread g such that t and T - t share a warp."""
    if T < 32:
        return g
    w, l = divmod(g, 32)
    return 16 * w + l if l < 16 else (T // 2 if g == 16 else T + 16 - 16 * w - l)


def neg_source(T, g):
    if T < 32:
        return (g & ~(T - 1)) | ((T - g) & (T - 1))
    return g if g in (0, 16) else g ^ 16


def rev(T, g):
    if T < 32:
        return g
    w, l = divmod(g, 32)
    return 16 * w + l if l < 16 else T + 15 - 16 * w - l


@pytest.mark.parametrize("L", LENGTHS)
def test_mirror_lanes(L):
    for T in {L // 16, last_ns(L)} & {L // 16}:
        assert sorted(neg(T, g) for g in range(T)) == list(range(T))
        assert sorted(rev(T, g) for g in range(T)) == list(range(T))
        for g in range(T):
            src = neg_source(T, g)
            assert src // 32 == g // 32 and neg(T, src) == (T - neg(T, g)) % T
            partner = g ^ (16 if T >= 32 else T - 1)
            assert partner // 32 == g // 32 and rev(T, partner) == T - 1 - rev(T, g)


@pytest.mark.parametrize("L", LENGTHS)
def test_forward_columns_meet_once(L):
    ns = last_ns(L)
    R, tps = radix(L, ns), L // 16
    nb = 16 // R
    written = []
    for g in range(tps):
        if nb == 1:
            t = neg(ns, g)
            other = neg(ns, neg_source(ns, g))
            for m in range(8):
                mirror = other + ns * (((16 - m) & 15) if t == 0 else 15 - m)
                c = t + ns * m
                assert mirror == (L - c) % L
                written += [c] if c == 0 else [c, mirror]
            written += [L // 2] if t == 0 else []
            continue
        for i in range(nb // 2):
            t = g + i * tps
            u = ns - t if t else ns // 2
            A = [t + ns * m for m in range(R)]
            B = [u + ns * m for m in range(R)]
            half = A[R // 2]
            if t == 0:  # both are their own mirrors: regrouped
                A, B = A[:R // 2] + B[:R // 2], B[R // 2:] + A[R // 2 + 1:] + A[:1]
            for h in range(2):
                base = t if h == 0 else (ns // 2 if t == 0 else t + L // 2)
                for m in range(R // 2):
                    c = base + ns * m
                    assert A[h * (R // 2) + m] == c and B[R - 1 - h * (R // 2) - m] == (L - c) % L
                    written += [c] if c == 0 else [c, L - c]
            written += [half] if t == 0 else []
    assert sorted(written) == list(range(L))


@pytest.mark.parametrize("L", LENGTHS)
def test_inverse_points_and_pairs_meet_once(L):
    T = L // 16
    points = []
    for g in range(T):  # preprocess: the thread's own points, and the mirrors it is sent
        t = neg(T, g)
        other = neg(T, neg_source(T, g))
        mine = [t + T * j for j in range(8)] + [None] * 8
        for j in range(8):
            mine[15 - j] = (L - (other + T * j)) % L
        if t == 0:
            mine[9:16] = mine[8:15]
            mine[8] = L // 2
        assert mine == [t + T * j for j in range(16)]
        points += mine
    assert sorted(points) == list(range(L))

    ns = last_ns(L)
    R, nb = radix(L, ns), 16 // radix(L, ns)
    pairs = []
    for g in range(T):  # pairing: (p, L - 1 - p), p < L / 2
        if nb == 1:
            t, other = rev(ns, g), rev(ns, g ^ (16 if ns >= 32 else ns - 1))
            pairs += [(t + ns * m, other + ns * (15 - m)) for m in range(8)]
            continue
        for i in range(nb // 2):
            t = g + i * T
            u = ns - 1 - t
            for m in range(R // 2):
                pairs += [(t + ns * m, u + ns * (R - 1 - m)), (u + ns * m, t + ns * (R - 1 - m))]
    assert sorted(p for p, _ in pairs) == list(range(L // 2)) and all(p + q == L - 1 for p, q in pairs)


@pytest.mark.parametrize("N", [64, 128, 256, 512, 1024, 2048, 4096])
def test_axis_pass_lanes(N):
    """The axis-0 pass: every butterfly of every sequence once, its mirror 16 lanes away."""
    T = N // 16
    NP = 1 if T >= 128 else min(16, 128 // T)
    GW = 32 // NP
    H = GW // 2

    def butterfly(g):
        w, sl = divmod(g, GW)
        t0 = H * w + sl % H
        return t0 if sl < H else (T - t0 if t0 else T // 2)

    assert T % GW == 0 and sorted(butterfly(g) for g in range(T)) == list(range(T))
    for g in range(T):
        for pi in range(NP):
            thread = g * NP + pi
            t = butterfly(g)
            other = thread if t in (0, T // 2) else thread ^ 16
            assert other // 32 == thread // 32 and other % NP == pi and butterfly(other // NP) == (T - t) % T

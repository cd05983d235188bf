"""The SM-pair GEMM's item numbers on a CPU model of its arithmetic (gemm_crt.cu): divisions by multiplication, and the
counter's jump over runs of tiles below the diagonal of an integral block."""
import random

import pytest


def fast_div(d):
    """FastDiv: (multiplier, shift) -> quotient of 0 <= n < 2^31."""
    s = 0
    while d > 1 and (2 << s) < d:
        s += 1
    mul = ((1 << (32 + s)) + d - 1) // d if d > 1 else 0
    assert mul < 1 << 32
    return lambda n: n if d == 1 else ((n * mul) >> 32) >> s


def test_division_by_multiplication():
    rng = random.Random(1)
    top = 2**31 - 1
    ds = list(range(1, 600)) + [rng.randrange(1, 2**31) for _ in range(2000)]
    ds += [2**k + e for k in range(1, 31) for e in (-1, 0, 1)]
    for d in ds:
        f = fast_div(d)
        near = [q * d + e for q in (1, top // d, rng.randrange(top // d + 1)) for e in (-1, 0, 1)]
        for n in [0, 1, top - 1, top] + near:
            if 0 <= n <= top:
                assert f(n) == n // d, (n, d)


@pytest.mark.parametrize("v,ab,nb,nm,ks,pairs", [(1, 1, 1, 1, 1, 76), (17, 16, 17, 2, 1, 7), (33, 28, 31, 2, 2, 1),
                                                 (64, 34, 53, 1, 1, 7), (137, 24, 60, 2, 1, 76), (160, 39, 55, 1, 1, 76),
                                                 (200, 30, 31, 2, 1, 7), (301, 12, 56, 1, 2, 76)])
@pytest.mark.parametrize("group", [8, 16])
def test_every_kept_tile_is_handed_out_once(v, ab, nb, nm, ks, pairs, group):
    M, N = ab * v, nb * v
    tm, tn, units = (M + 255) // 256, (N + 255) // 256, (N + 31) // 32
    ub, ur, g0 = units // tn, units % tn, min(tm, group)
    total = tm * tn * ks * nm

    def place(i):
        t = i % (tm * tn * ks) % (tm * tn)
        g, inside = divmod(t, g0 * tn)
        return inside, g * g0, min(tm - g * g0, g0)

    def skipped(i):
        inside, first, gm = place(i)
        j = inside // gm
        m0, n0, w = 256 * (first + inside % gm), 32 * (j * ub + min(j, ur)), 32 * (ub + (j < ur))
        return min(N - 1, n0 + w - 1) // v < m0 // v

    def after_skipped(i):
        inside, first, gm = place(i)
        amin = first * 256 // v
        end = lambda j: min(N, 32 * ((j + 1) * ub + min(j + 1, ur)))  # noqa: E731
        j = max(0, amin * v // 32 // (ub + 1) - 1)
        assert j == 0 or (end(j - 1) - 1) // v < amin
        while j < tn and (end(j) - 1) // v < amin:
            j += 1
        return max(i + 1, i - inside + j * gm)

    rng = random.Random(v)
    counter, got, current, live = 0, [], list(range(pairs)), list(range(pairs))
    while live:
        q = rng.choice(live)
        i = current[q]
        if i >= total:
            live.remove(q)
            continue
        if skipped(i):
            to = after_skipped(i)
            assert all(skipped(x) for x in range(i, min(to, total)))
            if to > i + 1:
                counter = max(counter, to - pairs)
        else:
            got.append(i)
        current[q] = pairs + counter
        counter += 1
    assert sorted(got) == [i for i in range(total) if not skipped(i)]

"""The room that h-support alone takes for its balls is an upper bound of what they need.

Balls are stored as an n-bit set (W words, padded to four) or, where that takes at most W words, as a
(word index, word) pair for every word that holds a member.  The bound knows only degrees: |B(x,1)|
is the degree plus one, |B(x,r)| at most the sum of |B(y,r-1)| over the neighbours y (one without
any), sums cut off at the padded row, and a pair for every member.  Both are restated here; the
kernels that compute the bound are k_ball_bound and k_bound_words."""

import numpy as np
import pytest

from synth import barabasi_albert, erdos_renyi_gnm, rmat


def adjacency(n, s, d):
    adj = [set() for _ in range(n)]
    for u, v in zip(s.tolist(), d.tolist()):
        if u != v:
            adj[u].add(v)
            adj[v].add(u)
    return adj


def stored_words(ball, W, Wpad):
    nz = len({x >> 5 for x in ball})
    return Wpad if 2 * nz > W else (2 * nz + 3) & ~3


def bounds(adj, h, Wpad):
    b = [min(len(a) + 1, Wpad) for a in adj]
    for _ in range(h - 1):
        b = [min(max(sum(b[y] for y in a), 1), Wpad) for a in adj]
    return [min(Wpad, (2 * x + 3) & ~3) for x in b]


def graphs():
    yield "isolated", 70, np.zeros(0, np.int32), np.zeros(0, np.int32)
    x = np.arange(300)
    yield "path", 300, x[:-1], x[1:]
    yield "star", 513, np.zeros(512, np.int64), np.arange(1, 513)
    # a star in few words of many, and in one word of one, two, three and four
    for n in (31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 2000):
        yield f"star{n}", n, np.zeros(9, np.int64), np.arange(1, 10)
    yield "er", 600, *erdos_renyi_gnm(600, 900, 1)
    yield "er2", 400, *erdos_renyi_gnm(400, 4000, 2)
    yield "rmat", 512, *rmat(9, 4, 0.57, 0.19, 0.19, 3)
    yield "ba", 500, *barabasi_albert(500, 3, 4)
    yield "scattered", 6000, *(29 * a for a in erdos_renyi_gnm(200, 500, 5))


@pytest.mark.parametrize("h", [1, 2, 3, 4])
def test_bound_covers_every_ball(h):
    for name, n, s, d in graphs():
        adj = adjacency(n, np.asarray(s), np.asarray(d))
        W = (n + 31) // 32
        Wpad = (W + 3) & ~3
        ball = [a | {x} for x, a in enumerate(adj)]
        first = list(ball)
        for _ in range(h - 1):
            ball = [set().union(b, *(first[y] for y in b)) for b in ball]
        for x, (b, top) in enumerate(zip(ball, bounds(adj, h, Wpad))):
            assert stored_words(b, W, Wpad) <= top <= Wpad, f"{name}, vertex {x}"

"""Models of the tridiagonalisation's exchange and buffers (no GPU), following k_tridiag.

Between blocks: column j is owned by block j mod G.  Step k has slots of its own, (S, C) pairs for the entries
t < N - k - 1, empty until their owner writes each word once: the owner of column j >= k + 1 writes S of entry
j - k - 1, the owner of column k + 1 every C.  A block reads all of step k before it writes anything of step k + 1,
and leaves once it owns no column >= k + 2, unless it owns the last column.  Random interleavings of single words
check that every word is written once, read only as its own step's, and that the exchange completes.

Within a block: three barriers a step (A after the polls, B, C) and warps that run freely between them, so the column
passes of step k and the polls of step k + 1 overlap.  Two warps may not touch the same part of a buffer between
the same two barriers if one of them writes, unless every thread keeps to its own entries.
"""
import random

import pytest


def slot_offset(N, k):
    return k * (N - 1) - k * (k - 1) // 2


@pytest.mark.parametrize("N,G", [(3, 1), (3, 2), (8, 2), (8, 4), (17, 4), (40, 9), (41, 21), (96, 12)])
def test_every_word_is_written_once_and_read_as_its_own(N, G):
    base = [2 * slot_offset(N, k) for k in range(N - 1)]
    assert all(b + 2 * (N - k - 1) <= (base[k + 1] if k + 2 < N else N * (N + 1)) for k, b in enumerate(base))

    def writes(b, k):                              # block b's words of step k, in any order
        w = [base[k] + 2 * (j - k - 1) for j in range(k + 1, N) if j % G == b]
        if (k + 1) % G == b:
            w += [base[k] + 2 * t + 1 for t in range(N - k - 1)]
        return w

    def program(b):
        acts = [("w", 0, w) for w in writes(b, 0)]
        last = b + G * ((N - 1 - b) // G)
        for k in range(N - 2):
            if b != (N - 1) % G and last < k + 2:
                break
            acts += [("r", k, base[k] + i) for i in range(2 * (N - k - 1))]
            if k + 3 < N:
                acts += [("w", k + 1, w) for w in writes(b, k + 1)]
        return acts

    for seed in range(5):
        rng = random.Random(seed)
        slots, progs, pos = {}, [program(b) for b in range(G)], [0] * G
        running = [b for b in range(G) if progs[b]]
        idle = 0
        while running:
            b = rng.choice(running)
            kind, k, word = progs[b][pos[b]]
            if kind == "w":
                assert word not in slots, (b, k, word)
                slots[word] = k
            elif word not in slots:                # still empty: poll again
                idle += 1
                assert idle < 50 * N * N * G, "the exchange did not complete"
                continue
            else:
                assert slots[word] == k, (b, k, word)
            pos[b] += 1
            if pos[b] == len(progs[b]):
                running.remove(b)


def conflicts(nc, np_, steps=9):
    """Pairs of accesses that race, with nc column buffers and np_ product buffers."""
    # access: (interval, warp, writes, own entries only, buffer part); intervals are numbered by the barrier before
    acc = []
    for k in range(steps):
        c, cn, p = f"c{k % nc}", f"c{(k + 1) % nc}", f"p{k % np_}"
        a, b, d = 3 * k, 3 * k + 1, 3 * k + 2      # the intervals after A, B and C of step k; polls: after C of k - 1
        for w in range(4):
            def put(i, wr, own, *parts):
                acc.extend((i, w, wr, own, x) for x in parts)
            put(a - 1, True, True, cn + "[0]", cn + "[1]", cn + "[2:]", p)          # (1) polls, q' from own entries
            put(a - 1, False, True, c + "[2:]", p)
            put(a - 1, True, True, "red")
            put(a, True, True, cn + "[0]", cn + "[1]", cn + "[2:]", p)              # (2) p and C - gamma tau p
            put(a, False, False, c + "[1]", c + "[2:]", "bc0-6", "S0C0")            #     v of owned columns, scalars
            put(b, True, True, cn + "[0]", cn + "[1]", cn + "[2:]")                 # (3) c_{k+1}
            put(b, False, False, c + "[1]", c + "[2:]", "bc5", "q", "e1h1")
            put(d, False, False, c + "[1]", c + "[2:]", cn + "[2:]", p, "q", "e1h1")     # (4) column passes
        acc.append((a - 1, 0, True, False, "S0C0"))
        acc.append((a, 3, True, False, "e1h1"))
        w4 = [(a, False, "red"), (a, True, "q"), (d, False, cn + "[0]"), (d, False, cn + "[1]"), (d, False, cn + "[2:]"),
              (d, True, "bc0-6"), (d, True, "bc5"), (d, True, cn + "[1]"), (d, False, c + "[1]"), (d, False, c + "[2:]")]
        acc.extend((i, 4, wr, False, x) for i, wr, x in w4)                         # sums, scalars, (5) the reflector
    out = set()
    by = {}
    for x in acc:
        by.setdefault((x[0], x[4]), []).append(x)
    for (i, part), xs in by.items():
        for x in xs:
            for y in xs:
                if x[1] < y[1] and (x[2] or y[2]) and not (x[3] and y[3]):
                    out.add(part[0] if part[0] in "cp" else part)
    return out


def test_three_column_buffers_and_two_product_buffers_are_enough():
    assert conflicts(3, 2) == set()


def test_fewer_buffers_would_race():
    assert "c" in conflicts(2, 2)
    assert "p" in conflicts(3, 1)

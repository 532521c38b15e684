"""Host restatements of the 3D order-3 FP32 star kernels' schemes: the blocked storage of a star's inverse with
the products of its blocks, and the way in which the consumer warps of the ring leave it after a timeout."""
import itertools

import numpy as np
import pytest

K, S1, SB = 3, 5, 15
NS, SN = 375, 125
SQ1, SQ2 = 30, 27


def _block_of(b, nbr, noff):
    if b >= noff:
        return b - noff, b - noff
    i = 0
    while b >= nbr - 1 - i:
        b -= nbr - 1 - i
        i += 1
    return i, i + 1 + b


def _box(kind):
    """Offsets of the free nodes along an axis: 0 interior vertex, -1 / 1 on the lower / upper boundary."""
    return {0: range(5), -1: range(3, 5), 1: range(0, 2)}[kind]


@pytest.mark.parametrize("kinds,m", [((0, 0, 0), 375), ((0, -1, 0), 150), ((1, 0, -1), 60), ((-1, 1, 1), 24)])
def test_blocked_star_storage_and_product(kinds, m):
    """Every entry of the free dofs' inverse is stored once, in 15 x 15 blocks interleaved by quads, and the two
    products of each block add up to the star's product; 24 free dofs leave a partial block."""
    entry = [c * SN + x + S1 * y + S1 * S1 * z for c in range(3) for z in _box(kinds[2]) for y in _box(kinds[1])
             for x in _box(kinds[0])]
    assert len(entry) == m and entry == sorted(entry)
    rng = np.random.default_rng(m)
    A = rng.standard_normal((NS, NS))
    A = A + A.T
    nbr = -(-m // SB)
    nblk, noff = nbr * (nbr + 1) // 2, nbr * (nbr - 1) // 2
    store = np.full(4 * (SQ1 * nblk + SQ2 * noff), np.nan)
    seen = set()
    for p in range(store.size):              # the packing kernel's map from a place to an entry
        second = p >= 4 * SQ1 * nblk
        w, n = ((p - 4 * SQ1 * nblk) >> 2, noff) if second else (p >> 2, nblk)
        q, b = divmod(w, n)
        e = 4 * (q + SQ1 if second else q) + (p & 3)
        I, J = _block_of(b, nbr, noff)
        if I != J:
            rr, cc = divmod(e, SB)
        else:
            rr = 0
            while rr + 1 < SB and e >= (rr + 1) * SB - (rr + 1) * rr // 2:
                rr += 1
            cc = rr + e - (rr * SB - rr * (rr - 1) // 2)
        i, j = SB * I + rr, SB * J + cc
        store[p] = 0.0
        if rr < SB and i < m and j < m:
            assert i <= j and (i, j) not in seen
            seen.add((i, j))
            store[p] = A[entry[i], entry[j]]
    assert len(seen) == m * (m + 1) // 2
    r = np.zeros(nbr * SB)
    r[:m] = rng.standard_normal(m)
    part = np.full((nbr * SB, nbr), np.nan)
    for b in range(nblk):                    # the products of block b
        I, J = _block_of(b, nbr, noff)
        rI, rJ = r[SB * I:SB * I + SB], r[SB * J:SB * J + SB]
        yI, yJ = np.zeros(SB), np.zeros(SB)
        for q in range(SQ1 + (SQ2 if I != J else 0)):
            at = 4 * (q * nblk + b) if q < SQ1 else 4 * SQ1 * nblk + 4 * ((q - SQ1) * noff + b)
            for k in range(4):
                e, v = 4 * q + k, store[at + k]
                if I != J:
                    if e < SB * SB:
                        rr, cc = divmod(e, SB)
                        yI[rr] += v * rJ[cc]
                        yJ[cc] += v * rI[rr]
                else:
                    rr = max(x for x in range(SB) if e >= x * SB - x * (x - 1) // 2)
                    cc = rr + e - (rr * SB - rr * (rr - 1) // 2)
                    yI[rr] += v * rI[cc]
                    if cc != rr:
                        yI[cc] += v * rI[rr]
        part[SB * I:SB * I + SB, J] = yI
        if I != J:
            part[SB * J:SB * J + SB, I] = yJ
    y = part.sum(axis=1)[:m]
    ref = A[np.ix_(entry, entry)] @ r[:m]
    assert np.abs(y - ref).max() <= 1e-11 * np.abs(ref).max()


def _leaves(vote, order, items=3):
    """Two consumers and a producer that sets the failure flag, stepped in the given order and then in turn.  A
    consumer's item: barrier, [read the flag,] barrier, [read the flag], go on or leave.  Returns whether all end."""
    flag = [False]
    waiting, votes, verdict = {}, {}, {}

    def consumer(me):
        for it in range(items):
            yield ("bar", 2 * it)
            mine = flag[0]
            yield
            votes.setdefault(it, {})[me] = mine
            yield ("bar", 2 * it + 1)
            if any(votes[it].values()) if vote else flag[0]:
                return
            yield

    def producer():
        flag[0] = True
        yield

    procs = {0: consumer(0), 1: consumer(1), 2: producer()}

    def step(k):
        if k not in procs:
            return False
        if k in waiting:                      # at a barrier until the other consumer is at the same one
            if waiting.get(1 - k) != waiting[k] and verdict.get((1 - k, waiting[k])) is None:
                return False
            verdict[(k, waiting[k])] = True
            del waiting[k]
        try:
            got = next(procs[k])
        except StopIteration:
            del procs[k]
            return True
        if got:
            waiting[k] = got[1]
        return True

    for k in order:
        step(k)
    while procs:
        if not any([step(k) for k in (0, 1, 2)]):
            return False
    return True


def test_ring_consumers_leave_together():
    """A flag that is read after the barrier can be seen by one consumer and not by the other, which then waits at a
    barrier that is never completed; a vote at the barrier cannot."""
    orders = list(itertools.product((0, 1, 2), repeat=9))
    assert all(_leaves(True, o) for o in orders)
    assert not all(_leaves(False, o) for o in orders)

"""Host model of the relaxation's request protocol (own_tiles in
csrc/relax_tiles.cuh) under random interleavings.

Owners look at the request counts of their tiles, solve those that are not
zero, and add requests for the neighbours that a solve can improve.  `open`
counts the requests that are not answered: a solve adds its requests to it
before it makes them and takes off what it answered after.  Every schedule
must end, with every value at its fixed point, and no owner may leave before."""

import random

import pytest


def _fixed_point(val, w):
    n = len(val)
    v = list(val)
    for _ in range(n):
        for i in range(n):
            for j in (i - 1, i + 1):
                if 0 <= j < n:
                    v[i] = min(v[i], v[j] + w[min(i, j)])
    return v


def _owner(me, tiles, val, w, req, shared, answered):
    n = len(val)
    while True:
        seen = [(t, req[t]) for t in tiles]
        yield
        if all(v == 0 for _, v in seen):
            if shared["open"] == 0:
                return
            continue
        for t, v in seen:
            if v == 0:
                continue
            req[t] -= v
            yield
            ring = {j: val[j] for j in (t - 1, t + 1) if 0 <= j < n}   # staged
            yield
            new = min([val[t]] + [x + w[min(t, j)] for j, x in ring.items()])
            asks = []
            if new < val[t]:
                val[t] = new
                asks = [j for j, x in ring.items() if new + w[min(t, j)] < x]
                yield
                shared["open"] += len(asks)
                yield
                for j in asks:
                    req[j] += 1
                    yield
            shared["open"] -= v
            answered[0] += v
            yield


@pytest.mark.parametrize("seed", range(40))
def test_ends_at_the_fixed_point(seed):
    rng = random.Random(seed)
    n, owners = rng.randint(1, 14), rng.randint(1, 5)
    val = [rng.randint(0, 60) for _ in range(n)]
    w = [rng.randint(0, 5) for _ in range(n)]
    want = _fixed_point(val, w)
    req = [1] * n
    shared, answered = {"open": n}, [0]
    live = [_owner(o, range(o, n, owners), val, w, req, shared, answered) for o in range(owners)]
    for _ in range(200000):
        if not live:
            break
        g = rng.choice(live)
        try:
            next(g)
        except StopIteration:
            live.remove(g)
            assert shared["open"] == 0 and not any(req)
    assert not live
    assert val == want

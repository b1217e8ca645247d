"""The order of waits in the persistent key-side gradient kernel, as a model: its roles (two producers, the
log-sum-exp warp, the product issuer, the warps of the epilogue) as coroutines over counted barriers, on lists of
work items most of which are empty.  No order of items may leave the roles waiting for one another, and no product
may overwrite what one still in flight reads: products on different accumulators finish in any order."""
import itertools
import random

import pytest

RING, QS, OS = 16, 3, 2                  # slots of the item ring, Q pairs, dO pairs


class Stuck(Exception):
    pass


class Overwritten(Exception):
    pass


def run(tiles, due_across_empty=False, overwrite_waits=True):
    """Runs the roles of one CTA over items of tiles[i] tiles (0: a key block no query block kept).  What must not
    be: with `due_across_empty` the issuer holds an item's last dK over the empty items after it, without
    `overwrite_waits` it trusts products to finish in the order they are issued in."""
    n, done = len(tiles), {}
    flight, order = [], random.Random(sum(tiles))       # products issued and not finished: the barriers they arrive on
    done_of = lambda name, i: done.get((name, i), 0)  # noqa: E731

    def arrive(name, i=0):
        done[name, i] = done_of(name, i) + 1

    def product(*arrivals, over=None):     # `over`: what the product that reads its output's columns arrives on
        if any(over in p for p in flight):
            raise Overwritten(over)
        flight.append(arrivals)

    def wait(name, i=0, count=1):          # a condition: `count` arrivals on barrier instance i
        return lambda: done_of(name, i) >= count

    def get(reader, i):                    # item i, or None past the last; frees its slot for this reader
        yield wait("posted", i)
        arrive("read", i)
        return tiles[i] if i < n else None

    def post(i):
        if i >= RING:
            yield wait("read", i - RING, 4)
        arrive("posted", i)

    def producer_q():
        yield from post(0)
        k = g = 0
        for i in range(n):
            yield from post(i + 1)
            if not tiles[i]:
                continue
            if k >= 2:
                yield wait("kv_empty", k - 2)
            arrive("kv_full", k)
            for _ in range(tiles[i]):
                if g >= QS:
                    yield wait("q_empty", g - QS)
                arrive("q_full", g)
                g += 1
            k += 1

    def producer_o():
        g = 0
        for i in itertools.count():
            T = yield from get("o", i)
            if T is None:
                return
            for _ in range(T):
                if g >= OS:
                    yield wait("o_empty", g - OS)
                arrive("o_full", g)
                g += 1

    def stats():
        g = 0
        for i in itertools.count():
            T = yield from get("stats", i)
            if T is None:
                return
            for _ in range(T):
                if g >= 2:
                    yield wait("q_empty", g - 2)
                arrive("q_full", g)
                g += 1

    def issuer():
        k = g = 0
        due = last = False

        def grad_k():
            nonlocal due
            if due:
                yield wait("ds_full", g - 1)
                product(("q_empty", g - 1), *([("acc_full", k - 1)] if last else []))
                due = False

        for i in itertools.count():
            T = yield from get("issuer", i)
            if T is None:
                break
            if T == 0:
                if not due_across_empty:
                    yield from grad_k()
                continue
            yield wait("kv_full", k)
            k += 1
            for t in range(T):
                yield wait("q_full", g, 2)
                if g and overwrite_waits:               # S goes where the last P was: dV has read it
                    yield wait("o_empty", g - 1)
                product(("s_full", g), over=("o_empty", g - 1))
                k -= t == 0                             # (the tile before belongs to the item before)
                yield from grad_k()
                k += t == 0
                if g and overwrite_waits:               # dP goes where the last dS was: dK has read it
                    yield wait("q_empty", g - 1)
                yield wait("o_full", g)
                product(("dp_full", g), *([("kv_empty", k - 1)] if t == T - 1 else []), over=("q_empty", g - 1))
                if t == 0 and k >= 2:
                    yield wait("acc_empty", k - 2)
                yield wait("p_full", g)
                product(("o_empty", g))
                due, last = True, t == T - 1
                g += 1
        yield from grad_k()

    def epilogue():
        k = g = 0
        for i in itertools.count():
            T = yield from get("epilogue", i)
            if T is None:
                return
            for _ in range(T):
                yield wait("q_full", g, 2)
                yield wait("s_full", g)
                arrive("p_full", g)
                yield wait("dp_full", g)
                arrive("ds_full", g)
                g += 1
            if T:
                yield wait("acc_full", k)
                arrive("acc_empty", k)
                k += 1

    roles = {f: f() for f in (producer_q, producer_o, stats, issuer, epilogue)}
    waits = {f: next(r, None) for f, r in roles.items()}
    while any(w is not None for w in waits.values()):
        moved = False
        for f, w in waits.items():
            while w is not None and w():
                w = waits[f] = next(roles[f], None)
                moved = True
        if not moved and flight:
            for barrier in flight.pop(order.randrange(len(flight))):
                arrive(*barrier)
        elif not moved:
            raise Stuck([f.__name__ for f, w in waits.items() if w is not None])


def lists():
    for t in (1, 2, 3):
        for gap in (0, 1, 14, 15, 16, 17, 18, 40):
            yield [t] + [0] * gap
            yield [t] + [0] * gap + [t]
            yield [0] * gap + [t] + [0] * gap + [t, t] + [0] * gap
    rng = random.Random(0)
    for _ in range(200):
        p = rng.choice([0.02, 0.1, 0.5, 0.95])
        yield [rng.randint(1, 6) if rng.random() < p else 0 for _ in range(rng.randint(1, 120))]


def test_roles_finish_on_every_list():
    for tiles in lists():
        run(tiles)


@pytest.mark.parametrize("gap", [16, 17, 40])
def test_model_sees_a_product_held_over_empty_items(gap):
    with pytest.raises(Stuck):
        run([1] + [0] * gap + [1], due_across_empty=True)


def test_model_sees_a_product_that_overwrites_an_operand():
    with pytest.raises(Overwritten):
        run([3], overwrite_waits=False)

"""The attention kernels' warps hand over to one another at mbarriers, whose waits give up after a limit, and at named barriers, where a
wait has none.  A model of the roles (walk.cuh and forward_bf16.cu, statement for statement what waits, arrives or looks at the
abort flag) in simulated time: each run finishes, or a role is left at a barrier.  In sound runs every wait must meet the phase that it
means and every named barrier the arrivals of one tile; in the others one asynchronous completion (a copy, a product's commit, the
answer to a request for an item) never comes, one wait runs out although nothing is lost, or the flag goes up at any moment, and every
role must still come to its end.
Two of the four row quarters are modelled, with the counts that go with them."""
import heapq
import random

import pytest

POLL, LIMIT, PAUSE = 8000, 3_000_000, 40_000      # a try_wait's suspension, a wait's limit (the kernels' is larger), leave()'s pause
QUARTERS = (0, 1)


class Stuck(Exception):
    pass


class MBar:
    def __init__(self, count=1):
        self.count = self.left = count
        self.done, self.waiting = 0, []           # completed phases


class Cta:
    """Processes are generators that yield: a number (cycles of work), ("mbar", bar, phase, soft) -> whether it completed, ("sync", id, n, tag)."""

    def __init__(self, seed, lost=None, expire=None, raised=None):
        self.rng, self.now, self.heap, self.order = random.Random(seed), 0, [], 0
        self.flag, self.lost, self.expire = False, lost, expire
        self.asyncs = self.waits = 0              # completions scheduled, waits begun
        self.named, self.alive, self.pipes = {}, {}, {}
        self.sound = lost is None and expire is None and raised is None
        self.slow = {}
        if raised is not None:
            self.at(raised, self.give_up)

    def at(self, delay, fn, *args):
        self.order += 1
        heapq.heappush(self.heap, (self.now + delay, self.order, fn, args))

    def stall(self):                              # any warp may be held up, by less than a suspension
        return self.rng.randrange(POLL // 2) if self.rng.random() < 0.01 else 0

    def jitter(self, cycles):
        return self.rng.choice((cycles // 4, cycles, cycles, cycles * 3)) + self.rng.randrange(20)

    def spawn(self, name, gen):
        self.slow[name] = self.rng.choice((1, 1, 1, 4))
        self.alive[name] = "start"
        self.at(self.rng.randrange(500), self.step, name, gen, None)

    def step(self, name, gen, value):
        try:
            op = gen.send(value)
        except StopIteration:
            del self.alive[name]
            return
        self.alive[name] = op if isinstance(op, (int, float)) else op[:2] if op[0] == "sync" else (op[0], op[2], op[3])
        if isinstance(op, (int, float)):
            self.at(op * (self.slow[name] if op < PAUSE else 1) + self.stall(), self.step, name, gen, None)
        elif op[0] == "mbar":
            self.waits += 1
            _, bar, phase, soft = op
            if self.waits - 1 == self.expire:     # runs out, whatever its barrier does
                self.at(LIMIT, self.run_out, name, gen)
            elif self.complete(bar, phase):
                self.at(20 + self.stall(), self.step, name, gen, True)
            else:
                w = [name, gen, phase, soft, True, self.now]
                bar.waiting.append(w)
                self.at(POLL, self.poll, bar, w)
        else:                                     # ("sync", id, threads, tag): waits;
            self.arrive(op[1], op[2], op[3], (name, gen))

    def complete(self, bar, phase):
        if self.sound:
            assert bar.done <= phase + 1, "the barrier has come round: the wait's phase is over"
        return (bar.done & 1) != (phase & 1)

    def give_up(self):
        self.flag = True

    def run_out(self, name, gen):
        self.give_up()
        self.step(name, gen, False)

    def poll(self, bar, w):
        if not w[4]:
            return
        name, gen, _, soft, _, since = w
        if self.now - since > LIMIT or (self.flag and (soft or (self.now - since) // POLL % 16 == 15)):
            w[4] = False
            bar.waiting.remove(w)
            if self.now - since > LIMIT:
                self.flag = True
            self.step(name, gen, False)
        else:
            self.at(POLL, self.poll, bar, w)

    def mbar_arrive(self, bar):
        bar.left -= 1
        if bar.left == 0:
            bar.left, bar.done = bar.count, bar.done + 1
            for w in list(bar.waiting):
                if self.complete(bar, w[2]):
                    w[4] = False
                    bar.waiting.remove(w)
                    self.at(self.jitter(40), self.step, w[0], w[1], True)

    def later(self, delay, bar):                  # an asynchronous completion: copy, answer
        self.asyncs += 1
        if self.asyncs - 1 != self.lost:
            self.at(delay, self.mbar_arrive, bar)

    def product(self, pipe, cycles, bars):        # products of one issuer complete in order, its commits behind them
        t = max(self.pipes.get(pipe, 0), self.now) + self.jitter(cycles)
        self.pipes[pipe] = t
        for b in bars:
            self.later(t - self.now, b)

    def arrive(self, ident, n, tag, waiter=None):
        b = self.named.setdefault(ident, [0, [], []])
        b[0] += 1
        b[2].append(tag)
        if waiter:
            b[1].append(waiter)
        if b[0] == n:
            assert not self.sound or len(set(b[2])) == 1, f"{ident}: arrivals of different tiles"
            del self.named[ident]
            for name, gen in b[1]:
                self.at(self.jitter(30), self.step, name, gen, True)

    def run(self):
        while self.heap:
            self.now, _, fn, args = heapq.heappop(self.heap)
            fn(*args)
        if self.alive:
            raise Stuck(self.alive)
        assert not (self.sound and self.flag)


def walk(T, N, take, broken=(), **how):
    """N items of T KV tiles; take: the items come one after another from the grid, as the producer asks for them."""
    c = Cta(**how)
    stages, threads_free, threads_p = 6, 2 * len(QUARTERS) + 1, 3 * len(QUARTERS) + 1
    Q, QEMPTY, SFULL = [MBar(), MBar()], [MBar(), MBar()], [MBar(), MBar()]
    KFULL, ODONE = [MBar() for _ in range(stages)], [MBar() for _ in range(stages)]
    X = {(q, i): MBar() for q in QUARTERS for i in range(4)}
    NEXT, ring = MBar(), 2 if "few items" in broken else 8
    ITEM, items = [MBar() for _ in range(8)], [None] * 8
    F, known = N * T, {"all": None}
    mbar = lambda bar, phase, soft: ("mbar", bar, phase, soft)
    odone = lambda f, soft: mbar(ODONE[f % stages], f // stages, soft)
    item_known = lambda n, soft: mbar(ITEM[n % ring], n // ring, soft)

    def producer():
        n = f = 0
        ok, item = True, 0
        while ok and (take or n < N):
            if n >= 2 and not (yield mbar(QEMPTY[n & 1], (n - 2) >> 1, False)):
                break
            if take:
                items[n & 7] = item
                if item < 0:
                    known["all"] = n * T
                    c.mbar_arrive(Q[n & 1])
                    c.mbar_arrive(ITEM[n % ring])
                    if T == 1 and "one announcement" not in broken:
                        c.mbar_arrive(ITEM[(n + 1) % ring])
                    break
                c.mbar_arrive(ITEM[n % ring])
            c.later(c.jitter(900), Q[n & 1])
            for _ in range(T):
                if f >= stages and not (yield odone(f - stages, False)):
                    ok = False
                    break
                c.later(c.jitter(900), KFULL[f % stages])
                f += 1
                yield c.jitter(60)
            if take and ok:
                c.later(c.jitter(1000), NEXT)
                ok = yield mbar(NEXT, n, False)
                item = n + 1 if n + 1 < N else -1
            n += 1
        if take and known["all"] is None:
            known["all"] = n * T

    def issuer1():
        n = j = f = 0
        while take or f < F:
            if j == 0 and (not (yield mbar(Q[n & 1], n >> 1, False)) or (take and items[n & 7] < 0)):
                return
            if not (yield mbar(KFULL[f % stages], f // stages, False)):
                return
            if f >= 4 and not (yield odone(f - 4, False)):
                return
            if f >= 2:
                if c.flag:
                    return
                yield 10
                yield ("sync", ("free", f & 1), threads_free, f - 2)
            j += 1
            c.product("s", 130, [SFULL[f & 1]] + ([QEMPTY[n & 1]] if j == T else []))
            if j == T:
                j, n = 0, n + 1
            f += 1
            yield c.jitter(40)

    def issuer2():
        n = j = f = 0
        while take or f < F:
            if take and j == 0:
                if not (yield item_known(n, False)) or items[n & 7] < 0:
                    return
                n += 1
            if not (yield mbar(KFULL[f % stages], f // stages, False)):
                return
            if c.flag:
                return
            yield 10
            yield ("sync", ("p", f & 3), threads_p, f)
            c.product("o", 150, [ODONE[f % stages]])
            f, j = f + 1, (j + 1) % T
            yield c.jitter(40)

    def scaling(q):
        f = 0

        def tile(first):
            nonlocal f
            yield mbar(X[q, f & 3], f >> 2, True)
            yield c.jitter(60)
            if not first and c.rng.random() < 0.7:               # the accumulator is scaled
                yield odone(f - 1, True)
                yield c.jitter(300)
            c.arrive(("p", f & 3), threads_p, f)
            f += 1

        def next_item(n):
            if take:
                yield item_known(n, True)
                more = items[n & 7] is not None and items[n & 7] >= 0
            else:
                more = n < N
            if more:
                yield from tile(True)
            return more

        n, more = 0, (yield from next_item(0))
        while more:
            for _ in range(1, T):
                yield from tile(False)
            yield odone(f - 1, True)
            if c.flag:
                if "no last arrival" not in broken:
                    c.arrive(("p", f & 3), threads_p, f)
                return
            yield c.jitter(300)
            n += 1
            more = yield from next_item(n)

    def softmax(t, h, q):
        own, other = ("max", q, t), ("max", q, t ^ 1)
        quarter = 4                                              # warps of a row quarter: two wait, two arrive
        if t == 1:
            c.arrive(other, quarter, 0)

        def tile(f):
            yield mbar(SFULL[t], f >> 1, True)
            yield c.jitter(250)
            yield ("sync", own, quarter, f)
            if h == 0:
                c.mbar_arrive(X[q, f & 3])
            yield c.jitter(300)
            c.arrive(("free", t), threads_free, f)
            yield c.jitter(200)
            c.arrive(other, quarter, f + 1)
            yield c.jitter(100)
            c.arrive(("p", f & 3), threads_p, f)

        def leave(f):
            yield PAUSE
            if "no leave" not in broken:
                c.arrive(("free", t), threads_free, f)
                c.arrive(("p", f & 3), threads_p, f)

        def meetings(f, to):
            while f < to:
                yield ("sync", own, quarter, f)
                c.arrive(other, quarter, f + 1)
                f += 2

        f = t
        if not take:
            while f < F:
                if f & 60 == 0 and c.flag:
                    yield from leave(f)
                    yield from meetings(f, F)
                    return
                for _ in range(2):
                    if f < F:
                        yield from tile(f)
                    f += 2
            return
        while True:
            if f % T < 2 and (f % T == t or f < 2 or f // T != (f - 2) // T):       # the team's first tile of an item
                n = f // T
                yield item_known(n, True)
                if (known["all"] is not None and f >= known["all"]) or c.flag:
                    break
            yield from tile(f)
            f += 2
        if c.flag:
            yield from leave(f)
            while known["all"] is None:
                yield 1000
            yield from meetings(f, known["all"])

    c.spawn("producer", producer())
    c.spawn("score products", issuer1())
    c.spawn("output products", issuer2())
    for q in QUARTERS:
        c.spawn(f"scaling {q}", scaling(q))
        for t in (0, 1):
            for h in (0, 1):
                c.spawn(f"softmax {t}{h}{q}", softmax(t, h, q))
    c.run()
    return c


def bf16(T, two, broken=(), **how):
    c = Cta(**how)
    stages, groups = 4, (0, 1) if two else (0,)
    threads = 2 * len(QUARTERS) + 1
    Q, FULL, EMPTY = MBar(), [MBar() for _ in range(stages)], [MBar() for _ in range(stages)]
    SFULL, ODONE = [MBar(), MBar()], [MBar(), MBar()]
    mbar = lambda bar, phase, soft=False: ("mbar", bar, phase, soft)

    def producer():
        c.later(c.jitter(900), Q)
        for n in range(2 * T):
            if n >= stages and not (yield mbar(EMPTY[n % stages], n // stages - 1)):
                return
            c.later(c.jitter(1500), FULL[n % stages])
            yield c.jitter(40)

    def issuer():
        def landed(n):
            return (yield mbar(FULL[n % stages], n // stages))

        def join(ident, j):
            if c.flag:
                return False
            yield 10
            yield ("sync", ident, threads, j)
            return True

        def gemm1(t, j):
            c.product("m", 500, [SFULL[t]] + ([EMPTY[2 * j % stages]] if t == 1 or not two else []))
            yield c.jitter(60)

        def gemm2(t, j):
            c.product("m", 500, [ODONE[t]] + ([EMPTY[(2 * j + 1) % stages]] if t == 1 or not two else []))
            yield c.jitter(60)

        if not (yield mbar(Q, 0)) or not (yield from landed(0)):
            return
        yield from gemm1(0, 0)
        if not two:
            for j in range(T):
                if j + 1 < T:
                    if not (yield from landed(2 * j + 2)) or not (yield from join(("free", 0), j)):
                        return
                    yield from gemm1(0, j + 1)
                if not (yield from landed(2 * j + 1)) or not (yield from join(("p", 0), j)):
                    return
                yield from gemm2(0, j)
            return
        if not (yield from join(("free", 0), 0)):
            return
        yield from gemm1(1, 0)
        if T > 1:
            if not (yield from landed(2)) or not (yield from join(("free", 1), 0)):
                return
            yield from gemm1(0, 1)
        for j in range(T):
            if not (yield from landed(2 * j + 1)) or not (yield from join(("p", 0), j)):
                return
            yield from gemm2(0, j)
            if j + 1 < T:
                if not (yield from join(("free", 0), j + 1)):
                    return
                yield from gemm1(1, j + 1)
            if j + 2 < T and not (yield from landed(2 * j + 4)):
                return
            if not (yield from join(("p", 1), j)):
                return
            yield from gemm2(1, j)
            if j + 2 < T:
                if not (yield from join(("free", 1), j + 1)):
                    return
                yield from gemm1(0, j + 2)

    def softmax(t, h, q):
        for j in range(T):
            done = yield mbar(SFULL[t], j, True)
            if not done and "leaves" in broken:
                return
            yield c.jitter(100)
            c.arrive(("free", t), threads, j)
            yield c.jitter(150)
            yield ("sync", ("pair", t, q), 2, j)
            if j > 0:
                yield mbar(ODONE[t], j - 1, True)
            yield c.jitter(600)
            c.arrive(("p", t), threads, j)
        yield ("sync", ("pair", t, q), 2, T)
        yield mbar(ODONE[t], T - 1, True)

    c.spawn("producer", producer())
    c.spawn("issuer", issuer())
    for t in groups:
        for q in QUARTERS:
            for h in (0, 1):
                c.spawn(f"softmax {t}{h}{q}", softmax(t, h, q))
    c.run()
    return c


# (KV tiles per item, items, whether they are taken); fixed shares look at the flag every 64 tiles
WALKS = [(1, 9, False), (2, 5, False), (3, 5, False), (5, 3, False), (70, 1, False),
         (1, 9, True), (2, 6, True), (3, 5, True), (4, 4, True), (5, 3, True), (7, 2, True), (9, 1, True)]


@pytest.mark.parametrize("T,N,take", WALKS)
def test_walking_kernel(T, N, take):
    for seed in range(12):
        c = walk(T, N, take, seed=seed)
    for k in range(0, c.asyncs, 1 if c.asyncs < 60 else 5):
        for seed in (2 * k, 2 * k + 1):
            walk(T, N, take, seed=seed, lost=k)
    for k in range(0, c.waits, 2 if c.waits < 300 else 11):
        walk(T, N, take, seed=k, expire=k)
    for seed in range(150):
        walk(T, N, take, seed=seed, raised=c.rng.randrange(c.now))


@pytest.mark.parametrize("T", [1, 2, 3, 6])
@pytest.mark.parametrize("two", [True, False])
def test_bf16_kernel(T, two):
    for seed in range(12):
        c = bf16(T, two, seed=seed)
    for k in range(c.asyncs):
        for seed in range(4):
            bf16(T, two, seed=seed, lost=k)
    for k in range(c.waits):
        bf16(T, two, seed=k, expire=k)
    for seed in range(60):
        bf16(T, two, seed=seed, raised=c.rng.randrange(c.now))


def fails(run):
    for seed in range(200):
        for how in [{}, {"lost": seed}] + [{"raised": 300 * i} for i in range(50)]:
            try:
                run(seed=seed, **how)
            except (Stuck, AssertionError):
                return True
    return False


@pytest.mark.parametrize("T,N,take,broken", [(2, 6, True, "no leave"), (3, 4, False, "no last arrival"), (1, 9, True, "one announcement"), (2, 6, True, "few items")])
def test_the_model_notices_what_is_left_out(T, N, take, broken):
    assert fails(lambda **how: walk(T, N, take, broken=(broken,), **how))


def test_the_bf16_model_notices_a_warp_that_leaves():
    assert fails(lambda **how: bf16(3, True, broken=("leaves",), **how))

"""Host-side model of the barrier protocol of the spare-buffer fused kernel (fused4s_kernel.cuh).

The kernel hands score buffers round between T query tiles through mbarriers whose waits are PARITY waits:
`wait(parity)` returns as soon as the barrier's current phase has the other parity, so it is only sound for a
waiter exactly one phase behind.  This model runs the same roles (TMA producer, one MMA issuer per tile, the
softmax warps, an in-order tensor pipe) as coroutines under a random scheduler, with barriers that have exactly
that semantics, and checks that nothing deadlocks and that every read sees the contents it expects (the right
score tile, the right weights, the right K/V stage).  A per-buffer barrier (instead of one per tile and buffer)
fails here within a few schedules -- on the GPU it showed as expired waits.
"""
import random

import pytest


class Bar:
    def __init__(self, count):
        self.count, self.pending, self.phase = count, count, 0

    def arrive(self):
        self.pending -= 1
        assert self.pending >= 0
        if self.pending == 0:
            self.phase += 1
            self.pending = self.count

    def done(self, parity):   # mbarrier.try_wait.parity
        return (self.phase & 1) != parity


def simulate(T, n_kv, stages, seed, warps=4, per_tile_barriers=True, limit=400000, products_per_buffer=False):
    """products_per_buffer: a products' barrier per tile AND buffer, waited for only where a row is re-anchored (at random); otherwise
    one per tile, every phase of which the softmax warps take."""
    rnd = random.Random(seed)
    NB = T + 1
    nt = 4 if per_tile_barriers else 1
    s_full = [[Bar(1) for _ in range(5)] for _ in range(nt)]
    p_full = [[Bar(warps) for _ in range(5)] for _ in range(nt)]
    sel = (lambda t: t) if per_tile_barriers else (lambda t: 0)
    q_full = [Bar(1) for _ in range(4)]
    pv_done = [Bar(1) for _ in range(4)]
    pv_of_buffer = [[Bar(1) for _ in range(5)] for _ in range(4)]
    products = set()   # (tile, key tile) whose product has completed
    o_final = [Bar(1) for _ in range(4)]
    kv_full = [Bar(1) for _ in range(stages)]
    kv_empty = [Bar(T) for _ in range(stages)]
    pipe, buf, stage, errors = [], {}, {}, []

    def check(cond, what):
        if not cond:
            errors.append(what)

    def producer():
        for t in range(T):
            q_full[t].arrive()
        yield
        for j in range(n_kv):
            s = j % stages
            if j >= stages:
                while not kv_empty[s].done(((j // stages) - 1) & 1):
                    yield
            stage[s] = j
            kv_full[s].arrive()
            yield

    def issuer(t):
        tn = 0 if t + 1 == T else t + 1
        while not (kv_full[0].done(0) and q_full[t].done(0) and q_full[tn].done(0)):
            yield

        def issue_s(tile, j, b):
            check(stage.get(j % stages) == j, ("S reads a stale stage", tile, j))
            pipe.append(("S", tile, j, b, [s_full[sel(tile)][b]]))
        issue_s(t, 0, t)
        if t == T - 1 and n_kv > 1:
            while not kv_full[1 % stages].done((1 // stages) & 1):
                yield
            issue_s(tn, 1, T)
        b, ph, jm = t, 0, 0
        for j in range(n_kv):
            jn = j + (2 if t + 1 == T else 1)
            more = jn < n_kv
            if more:
                while not kv_full[jn % stages].done((jn // stages) & 1):
                    yield
            while not p_full[sel(t)][b].done(ph):
                yield
            check(stage.get(j % stages) == j, ("P V reads a stale stage", t, j))
            check(buf.get(b) == ("P", t, j), ("P V reads the wrong weights", t, j, b, buf.get(b)))
            pipe.append(("PV", t, j, b, []))
            if more:
                issue_s(tn, jn, b)
            pipe.append(("C", t, j, b, [pv_of_buffer[t][b] if products_per_buffer else pv_done[t], kv_empty[j % stages]] + ([o_final[t]] if j == n_kv - 1 else [])))
            b = NB - 1 if b == 0 else b - 1
            jm += 1
            if jm == NB:
                jm, ph = 0, ph ^ 1
            yield

    def softmax(t):
        b, ph, jm = t % NB, 0, 0
        for j in range(n_kv):
            while not s_full[sel(t)][b].done(ph):
                yield
            check(buf.get(b) in (("S", t, j), ("P", t, j)), ("softmax reads the wrong scores", t, j, b, buf.get(b)))
            yield
            if products_per_buffer and j > 0 and rnd.random() < 0.3:
                while not pv_of_buffer[t][0 if b == NB - 1 else b + 1].done(ph if jm > 0 else ph ^ 1):
                    yield
                check((t, j - 1) in products, ("re-anchored before the last product", t, j))
            buf[b] = ("P", t, j)
            if j > 0 and not products_per_buffer:
                while not pv_done[t].done((j - 1) & 1):
                    yield
            p_full[sel(t)][b].arrive()
            b = NB - 1 if b == 0 else b - 1
            jm += 1
            if jm == NB:
                jm, ph = 0, ph ^ 1
            yield
        while not o_final[t].done(0):
            yield

    procs = [producer()] + [issuer(t) for t in range(T)] + [softmax(t) for t in range(T) for _ in range(warps)]
    steps = 0
    while procs and not errors:
        steps += 1
        if steps > limit:
            return "deadlock"
        if pipe and rnd.random() < 0.5:      # the tensor pipe retires its queue in order
            kind, tile, j, b, bars = pipe.pop(0)
            if kind == "S":
                buf[b] = ("S", tile, j)
            if kind == "C":
                products.add((tile, j))
            for x in bars:
                x.arrive()
        i = rnd.randrange(len(procs))
        try:
            next(procs[i])
        except StopIteration:
            procs.pop(i)
    return errors[0] if errors else "ok"


@pytest.mark.parametrize("T", [1, 2, 3, 4])
@pytest.mark.parametrize("n_kv", [1, 2, 3, 8, 9, 17])
def test_rotation_protocol_completes_with_the_right_contents(T, n_kv):
    for seed in range(3):
        assert simulate(T, n_kv, 8, seed) == "ok"


@pytest.mark.parametrize("T", [1, 2, 3, 4])
@pytest.mark.parametrize("n_kv", [1, 2, 5, 6, 11, 17])
def test_products_barriers_that_are_waited_for_now_and_then(T, n_kv):
    for seed in range(4):
        assert simulate(T, n_kv, 8, seed, products_per_buffer=True) == "ok"


def test_one_barrier_per_buffer_is_not_enough():
    """Different tiles consuming successive phases of ONE barrier per buffer can start waiting a phase early."""
    outcomes = {simulate(4, 17, 8, seed, per_tile_barriers=False) for seed in range(12)}
    assert outcomes != {"ok"}


# ---------------------------------------------------------------------------------------------------------------
# The variant for ONE query tile per CTA: the key tiles are dealt out among SPLIT warpgroups ("parts": part g takes
# key tiles g, g + SPLIT, ...), NB score buffers run ahead of the products, and the MMAs come from TWO threads -- the
# products O_g (+)= P(j) V(j) from one, the scores of key tile j + NB from the other -- whose instructions the tensor
# pipe does not order against each other.

def simulate_parts(SPLIT, NB, n_kv, stages, seed, warps=4, wait_buf_free=True, limit=400000, apart=False):
    """apart: K and V by producers of their own, K's stage free when its scores are computed.  The products' barriers are waited for
    where a row is re-anchored only (at random)."""
    rnd = random.Random(seed)
    s_full = [Bar(1) for _ in range(NB)]
    p_full = [Bar(warps) for _ in range(NB)]
    buf_free = [Bar(1) for _ in range(NB)]
    pv_done = [Bar(1) for _ in range(SPLIT)]
    o_final = Bar(1)
    q_full = Bar(1)
    kv_full = [Bar(1) for _ in range(stages)]
    kv_empty = [Bar(1) for _ in range(stages)]
    k_full, k_empty = [Bar(1) for _ in range(stages)], [Bar(1) for _ in range(stages)]   # (apart)
    k_stage, products = {}, set()
    pipe_a, pipe_b = [], []                      # per issuing thread, each retired in order
    buf = {b: {} for b in range(NB)}             # per buffer and warp: what it holds
    stage, errors = {}, []

    def check(cond, what):
        if not cond:
            errors.append(what)

    def producer(holds, full, empty, with_q):
        if with_q:
            q_full.arrive()
            yield
        for j in range(n_kv):
            s = j % stages
            if j >= stages:
                while not empty[s].done(((j // stages) - 1) & 1):
                    yield
            holds[s] = j
            full[s].arrive()
            yield

    def score_thread():
        while not q_full.done(0):
            yield
        holds, full = (k_stage, k_full) if apart else (stage, kv_full)
        for jn in range(n_kv):
            b = jn % NB
            while not full[jn % stages].done((jn // stages) & 1):
                yield
            if jn >= NB and wait_buf_free:
                while not buf_free[b].done(((jn // NB) - 1) & 1):
                    yield
            check(holds.get(jn % stages) == jn, ("S reads a stale stage", jn))
            pipe_b.append(("S", jn, b, [s_full[b]] + ([k_empty[jn % stages]] if apart else [])))
            yield

    def product_thread():
        for j in range(n_kv):
            b = j % NB
            while apart and not kv_full[j % stages].done((j // stages) & 1):
                yield
            while not p_full[b].done((j // NB) & 1):
                yield
            check(stage.get(j % stages) == j, ("P V reads a stale stage", j))
            pipe_a.append(("PV", j, b, [pv_done[j % SPLIT], buf_free[b], kv_empty[j % stages]] +
                           ([o_final] if j == n_kv - 1 else [])))
            yield

    def part_warp(g, w):
        for i, j in enumerate(range(g, n_kv, SPLIT)):
            b = j % NB
            while not s_full[b].done((j // NB) & 1):
                yield
            check(buf[b].get(w) == ("S", j), ("a part reads the wrong scores", g, w, j, b, buf[b].get(w)))
            yield
            buf[b][w] = ("P", j)
            if i > 0 and rnd.random() < 0.3:   # re-anchored behind the product of the part's previous key tile
                while not pv_done[g].done((i - 1) & 1):
                    yield
                check(j - SPLIT in products, ("re-anchored before the part's last product", g, j))
            p_full[b].arrive()
            yield
        while not o_final.done(0):
            yield

    procs = [producer(stage, kv_full, kv_empty, not apart), score_thread(), product_thread()]
    procs += [producer(k_stage, k_full, k_empty, True)] if apart else []
    procs += [part_warp(g, w) for g in range(SPLIT) for w in range(warps)]
    steps = 0
    while procs and not errors:
        steps += 1
        if steps > limit:
            return "deadlock"
        for pipe in (pipe_a, pipe_b):        # two in-order queues, retired independently of one another
            if pipe and rnd.random() < 0.4:
                kind, j, b, bars = pipe.pop(0)
                if kind == "S":
                    for w in range(warps):
                        buf[b][w] = ("S", j)
                else:
                    check(all(buf[b].get(w) == ("P", j) for w in range(warps)), ("P V reads the wrong weights", j, b))
                    products.add(j)
                for x in bars:
                    x.arrive()
        i = rnd.randrange(len(procs))
        try:
            next(procs[i])
        except StopIteration:
            procs.pop(i)
    return errors[0] if errors else "ok"


@pytest.mark.parametrize("SPLIT,NB", [(2, 2), (2, 4), (4, 4)])
@pytest.mark.parametrize("n_kv", [1, 2, 3, 4, 5, 8, 16, 17])
def test_lone_tile_in_parts_protocol(SPLIT, NB, n_kv):
    for seed in range(4):
        assert simulate_parts(SPLIT, NB, n_kv, 8, seed) == "ok"
        assert simulate_parts(SPLIT, NB, n_kv, NB + 1, seed) == "ok"


@pytest.mark.parametrize("n_kv", [1, 3, 4, 5, 8, 16, 17])
def test_lone_tile_in_parts_with_k_and_v_apart(n_kv):
    for seed in range(6):
        assert simulate_parts(2, 3, n_kv, 3, seed, apart=True) == "ok"


def test_scores_must_wait_for_the_completion_of_the_products_they_overwrite():
    """Without the per-buffer completion barrier the second thread's scores can land on weights not yet read."""
    outcomes = {simulate_parts(2, 4, 17, 8, seed, wait_buf_free=False) for seed in range(12)}
    assert outcomes != {"ok"}


# ---------------------------------------------------------------------------------------------------------------
# K and V apart, with an issuing thread per part: it issues the product of key tile j and, behind it, in order, the scores of key tile j + NB
# into the buffer the product frees.  The threads are not ordered among one another, so every barrier has one consumer:
# scores and weights one per part and buffer, "K(n) has landed" one of eight, a multiple of the parts and no less than the stages.

def simulate_parts_by_threads(SPLIT, NB, n_kv, stages, seed, warps=4, limit=400000, landed=8, per_part=True, products=5, landing=0.3,
                              anchors=0.3):
    """per_part: barriers of scores and weights per part and buffer, not per buffer alone.  landing, anchors: how soon a copy lands, how often
    a row is re-anchored."""
    rnd = random.Random(seed)
    parts = SPLIT if per_part else 1
    s_full = [[Bar(1) for _ in range(NB)] for _ in range(parts)]
    p_full = [[Bar(warps) for _ in range(NB)] for _ in range(parts)]
    meets = NB   # (as the kernel counts: a part comes back to a buffer after so many of its key tiles, if SPLIT and NB have no common factor)
    pv_done = [[Bar(1) for _ in range(products)] for _ in range(SPLIT)]
    o_final, q_full = Bar(min(SPLIT, n_kv)), Bar(1)
    kv_full, k_full = ([Bar(1) for _ in range(landed)] for _ in range(2))
    kv_empty, k_empty = ([Bar(1) for _ in range(stages)] for _ in range(2))
    pipes = [[] for _ in range(SPLIT)]           # per issuing thread, each retired in order
    buf = {b: {} for b in range(NB)}
    k_stage, v_stage, done, errors, in_flight = {}, {}, set(), [], []

    def check(cond, what):
        if not cond:
            errors.append(what)

    def phase_of(i, j):   # of a part's i-th key tile in its barrier
        return (i // meets if per_part else j // NB) & 1

    def loader(holds, full, empty, with_q):
        if with_q:
            in_flight.append(([], None, q_full))
        for j in range(n_kv):
            s = j % stages
            if j >= stages:
                while not empty[s].done(((j // stages) - 1) & 1):
                    yield
            in_flight.append(([(h, s) for h in holds], j, full[j % landed]))
            yield

    def issuer(g):
        part_n = (g + NB) % SPLIT

        def issue_s(n):
            check(k_stage.get(n % stages) == n, ("S reads a stale stage", n))
            check(n % SPLIT == part_n, ("another part's scores", n))
            pipes[g].append(("S", n, n % NB, [s_full[part_n if per_part else 0][n % NB]] + [k_empty[n % stages]]))

        while not q_full.done(0):
            yield
        for n in range(part_n, min(NB, n_kv), SPLIT):
            while not k_full[n % landed].done(0):
                yield
            issue_s(n)
        for i, j in enumerate(range(g, n_kv, SPLIT)):
            b, n = j % NB, j + NB
            while n < n_kv and not k_full[n % landed].done((n // landed) & 1):
                yield
            while not kv_full[j % landed].done((j // landed) & 1):
                yield
            while not p_full[g if per_part else 0][b].done(phase_of(i, j)):
                yield
            check(v_stage.get(j % stages) == j, ("P V reads a stale stage", j))
            pipes[g].append(("PV", j, b, []))
            if n < n_kv:
                issue_s(n)
            pipes[g].append(("C", j, b, [kv_empty[j % stages], pv_done[g][i % products]] + ([o_final] if j + SPLIT >= n_kv else [])))
            yield

    def part_warp(g, w):
        for i, j in enumerate(range(g, n_kv, SPLIT)):
            b = j % NB
            while not s_full[g if per_part else 0][b].done(phase_of(i, j)):
                yield
            check(buf[b].get(w) == ("S", j), ("a part reads the wrong scores", g, w, j, b, buf[b].get(w)))
            yield
            buf[b][w] = ("P", j)
            if i > 0 and rnd.random() < anchors:   # re-anchored behind the product of the part's previous key tile
                while not pv_done[g][(i - 1) % products].done(((i - 1) // products) & 1):
                    yield
                check(j - SPLIT in done, ("re-anchored before the part's last product", g, j))
            p_full[g if per_part else 0][b].arrive()
            yield
        while not o_final.done(0):
            yield
        check(len(done) == n_kv, ("output before the last product", g))

    procs = [issuer(g) for g in range(SPLIT)]
    procs += [loader([k_stage], k_full, k_empty, True), loader([v_stage], kv_full, kv_empty, False)]
    procs += [part_warp(g, w) for g in range(SPLIT) for w in range(warps)]
    speed = [rnd.choice((0.02, 0.3, 1.0)) for _ in range(len(pipes))]   # a queue may lag far behind the others
    eager = {id(p): rnd.choice((0.05, 0.5, 1.0)) for p in procs}
    steps = 0
    while procs and not errors:
        steps += 1
        if steps > limit:
            return "deadlock"
        if in_flight and rnd.random() < landing:     # copies land in any order
            holds, j, bar = in_flight.pop(rnd.randrange(len(in_flight)))
            for h, s in holds:
                h[s] = j
            bar.arrive()
        for pipe, p in zip(pipes, speed):
            if pipe and rnd.random() < p:
                kind, j, b, bars = pipe.pop(0)
                if kind == "S":
                    for w in range(warps):
                        buf[b][w] = ("S", j)
                elif kind == "PV":
                    check(all(buf[b].get(w) == ("P", j) for w in range(warps)), ("P V reads the wrong weights", j, b))
                else:
                    done.add(j)
                for x in bars:
                    x.arrive()
        i = rnd.randrange(len(procs))
        if rnd.random() < eager[id(procs[i])]:
            try:
                next(procs[i])
            except StopIteration:
                procs.pop(i)
    return errors[0] if errors else "ok"


@pytest.mark.parametrize("stages", [3, 5, 8])
@pytest.mark.parametrize("n_kv", [1, 2, 3, 4, 5, 8, 17, 31])
def test_parts_with_issuing_threads_of_their_own(stages, n_kv):
    for seed in range(8):
        assert simulate_parts_by_threads(2, 3, n_kv, stages, seed) == "ok"


def test_issuing_threads_of_their_own_need_barriers_of_their_own():
    """Barriers of scores and weights that parts share fail."""
    outcomes = {simulate_parts_by_threads(2, 3, 31, 3, seed, per_part=False) for seed in range(80)}
    assert outcomes != {"ok"}


@pytest.mark.parametrize("NB", [2, 4])
def test_parts_and_score_buffers_with_a_common_factor_fail(NB):
    """A part comes back to a buffer after NB of its key tiles only where SPLIT and NB have no common factor."""
    outcomes = {simulate_parts_by_threads(2, NB, 17, 5, seed) for seed in range(8)}
    assert "ok" not in outcomes


def test_one_products_barrier_a_part_is_not_enough():
    """A softmax warp that looks now and then can be two phases of one barrier behind."""
    outcomes = {simulate_parts_by_threads(2, 3, 17, 3, seed, products=1) for seed in range(12)}
    assert outcomes != {"ok"}


def test_a_landed_barrier_has_one_issuer():
    """Barriers by stage, three of them: successive key tiles of a barrier belong to different issuers, and one that runs ahead takes an earlier
    copy's phase for its own while its copy is on its way."""
    outcomes = {simulate_parts_by_threads(2, 3, 17, 3, seed, landed=3, landing=0.005) for seed in range(12)}
    assert outcomes != {"ok"}
    assert {simulate_parts_by_threads(2, 3, 17, 3, seed, landing=0.005) for seed in range(12)} == {"ok"}

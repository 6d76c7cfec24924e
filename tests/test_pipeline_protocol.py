"""The barriers of the GEMM kernels (csrc/umma_gemm.cu) as models on the CPU: the order in which a group of unpacker warps
waits for its two barriers (expand_codes), and the CTAs of a tile, one or a pair, from their first step to their exit.

Weight codes travel through a ring of code stages into shared memory (TMA, whose copies may land in any order), two groups
of warps take alternate pipeline steps and expand them into a ring of operand stages, and the MMA consumes those in order.
A barrier is waited for by the parity of its phase, and a wait for the phase after next is passed at once: with three code
stages a stage's steps belong to the two groups in turn, so a group that asked for its codes first could be through before
the other group's codes had even landed in that stage."""
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_14435_b200", "csrc", "umma_gemm.cu")


class Barrier:
    """One arrival per phase; `landing`: the phase also waits for a copy in flight."""

    def __init__(self):
        self.phase, self.arrived, self.landing = 0, False, False

    def passed(self, parity):
        return (self.phase & 1) != parity

    def arrive(self, landing=False):
        assert not self.arrived, "a second arrival in one phase"
        self.arrived, self.landing = True, landing
        self._turn()

    def land(self):
        self.landing = False
        self._turn()

    def _turn(self):
        if self.arrived and not self.landing:
            self.phase, self.arrived = self.phase + 1, False


def walk(order, stages, code_stages, steps, rng):
    """One walk over `steps` pipeline steps under a random schedule; raises where a step meets the wrong data."""
    empty, full_u = [Barrier() for _ in range(stages)], [Barrier() for _ in range(stages)]
    empty_p, full_p = [Barrier() for _ in range(code_stages)], [Barrier() for _ in range(code_stages)]
    codes, operand = [None] * code_stages, [None] * stages

    def landing(n):
        codes[n % code_stages] = n
        full_p[n % code_stages].land()
        return
        yield

    def producer():
        for n in range(steps):
            s = n % code_stages
            yield lambda: empty_p[s].passed(((n // code_stages) & 1) ^ 1)
            full_p[s].arrive(landing=True)
            agents.append([landing(n), None])

    def group(g):
        for n in range(g, steps, 2):
            s, q = n % stages, n % code_stages
            waits = {"empty": lambda: empty[s].passed(((n // stages) & 1) ^ 1),
                     "full_p": lambda: full_p[q].passed((n // code_stages) & 1)}
            for name in order:
                yield waits[name]
            assert codes[q] == n, "expanded codes of another step"
            operand[s] = n
            full_u[s].arrive()
            empty_p[q].arrive()

    def mma():
        for n in range(steps):
            s = n % stages
            yield lambda: full_u[s].passed((n // stages) & 1)
            assert operand[s] == n
            empty[s].arrive()

    agents = [[a, None] for a in (producer(), group(0), group(1), mma())]
    while agents:
        ready = [a for a in agents if a[1] is None or a[1]()]
        assert ready, "deadlock"
        a = rng.choice(ready)
        try:
            a[1] = next(a[0])
        except StopIteration:
            agents.remove(a)


def source_order():
    text = open(SOURCE).read()
    body = text[text.index("expand_codes("):]
    wait = re.search(r"const bool ok = (.*?);", body, re.S).group(1)
    order = [m.group(1) for m in re.finditer(r"bars->(full_p|empty)\[", wait)]
    assert sorted(order) == ["empty", "full_p"], wait
    return order


@pytest.mark.parametrize("stages,code_stages", [(3, 3), (3, 4)])     # INT8 codes; 2-bit and 4-bit ones
def test_unpackers_meet_the_codes_of_their_own_step(stages, code_stages):
    for seed in range(400):
        walk(source_order(), stages, code_stages, 24, random.Random(seed))


def test_the_model_tells_the_orders_apart():
    with pytest.raises(AssertionError):
        for seed in range(400):
            walk(["full_p", "empty"], 3, 3, 24, random.Random(seed))


class CountingBarrier(Barrier):
    """`count` arrivals and all announced bytes per phase.  Bytes may land before they are announced."""

    def __init__(self, count):
        super().__init__()
        self.count, self.pending, self.bytes = count, count, 0

    def arrive(self, announced=0):
        assert self.pending > 0, "more arrivals than one phase has"
        self.pending, self.bytes = self.pending - 1, self.bytes + announced
        self._turn()

    def land(self):
        self.bytes -= 1
        self._turn()

    def _turn(self):
        if self.pending == 0 and self.bytes == 0:
            self.phase, self.pending = self.phase + 1, self.count


def walk_ctas(ctas, stages, code_stages, items, steps, rng, announced=None, waits=lambda r: True, commits=lambda r: True,
              tail=True):
    """The CTAs of one tile over `items` tiles of `steps` pipeline steps; code_stages = 0: the weights need no expansion.
    Every CTA has its own `empty`, `full_p`, `empty_p` and `tmem_full`; `full` and `tmem_empty` are the first one's.  Copies
    and commits land whenever they like, a commit in either CTA at a time of its own; only the commits of two steps, a step of MMAs
    apart, reach one CTA in their order (an accumulator's, issued right behind that of its last step, has none).  A CTA's shared
    memory goes when all warps have come to their end.  Wrong variants: announced (copies that the first producer announces
    per step), waits(r) (whether the producer of CTA r waits for a free stage), commits(r) (whether commits reach CTA r), tail
    (whether the producers stay for the last commits)."""
    unpack = code_stages > 0
    ranks, total = range(ctas), items * steps
    full = [CountingBarrier(1 + (ctas if unpack else 0)) for _ in range(stages)]
    tmem_empty = [CountingBarrier(ctas) for _ in range(2)]
    empty, tmem_full = [[CountingBarrier(1) for _ in range(stages)] for _ in ranks], [[CountingBarrier(1) for _ in range(2)] for _ in ranks]
    full_p, empty_p = [[[CountingBarrier(1) for _ in range(code_stages)] for _ in ranks] for _ in range(2)]
    tokens, weights, codes = [[None] * stages for _ in ranks], [[None] * stages for _ in ranks], [[None] * code_stages for _ in ranks]
    at_work, tensor_pipe, accumulator, committed = [0], [], [None, None], [0] * ctas

    def spawn(gen):
        agents.append([gen, None])

    def land(barrier, place=None, at=0, step=None):
        assert at_work[0], "something lands in shared memory that is given back"
        if place is not None:
            place[at] = step
        barrier.land() if place is not None else barrier.arrive()
        return
        yield

    def commit_step(r, n):
        yield lambda: committed[r] == n
        committed[r] += 1
        yield from land(empty[r][n % stages])

    def token_producer(r):
        own = 1 if unpack else 2                          # copies of one step: the token rows, and bf16 weight rows
        for n in range(total):
            s = n % stages
            yield lambda: not waits(r) or empty[r][s].passed(((n // stages) & 1) ^ 1)
            if r == 0:
                full[s].arrive(announced=ctas * own if announced is None else announced)
            spawn(land(full[s], tokens[r], s, n))
            if not unpack:
                spawn(land(full[s], weights[r], s, n))
        for n in range(total, total + stages if tail else total):
            yield lambda: empty[r][n % stages].passed(((n // stages) & 1) ^ 1)

    def code_producer(r):
        for n in range(total):
            s = n % code_stages
            yield lambda: empty_p[r][s].passed(((n // code_stages) & 1) ^ 1)
            full_p[r][s].arrive(announced=1)
            spawn(land(full_p[r][s], codes[r], s, n))

    def group(r, g):
        for n in range(g, total, 2):
            s, q = n % stages, n % code_stages
            yield lambda: empty[r][s].passed(((n // stages) & 1) ^ 1)
            yield lambda: full_p[r][q].passed((n // code_stages) & 1)
            assert codes[r][q] == n, "expanded codes of another step"
            weights[r][s] = n
            full[s].arrive()
            empty_p[r][q].arrive()

    def issuer():
        for i in range(items):
            yield lambda: tmem_empty[i & 1].passed(((i >> 1) & 1) ^ 1)
            for n in range(i * steps, (i + 1) * steps):
                yield lambda: full[n % stages].passed((n // stages) & 1)
                tensor_pipe.append((n, i))
            tensor_pipe.append((None, i))

    def mmas():
        for _ in range(total + items):
            yield lambda: tensor_pipe
            n, i = tensor_pipe.pop(0)
            for r in ranks:
                if n is not None:
                    assert tokens[r][n % stages] == n and weights[r][n % stages] == n, "operands of another step"
            accumulator[i & 1] = i
            for r in filter(commits, ranks):               # a commit: to the barrier at this offset in every CTA
                spawn(land(tmem_full[r][i & 1]) if n is None else commit_step(r, n))

    def epilogue(r):
        for i in range(items):
            yield lambda: tmem_full[r][i & 1].passed((i >> 1) & 1)
            assert accumulator[i & 1] == i
            tmem_empty[i & 1].arrive()

    def warp(gen):                                         # a warp of a CTA: the CTAs stay until all of theirs are done
        at_work[0] += 1
        yield from gen
        at_work[0] -= 1

    agents = [[mmas(), None], [warp(issuer()), None]]      # (the tensor pipe is not a warp: nobody waits for its end)
    for r in ranks:
        roles = [token_producer(r), epilogue(r)] + ([code_producer(r), group(r, 0), group(r, 1)] if unpack else [])
        agents += [[warp(w), None] for w in roles]
    for a in agents[1:]:
        a[1] = next(a[0], None)
    while agents:
        ready = [a for a in agents if a[1] is None or a[1]()]
        assert ready, "deadlock"
        a = rng.choice(ready)
        try:
            a[1] = next(a[0])
        except StopIteration:
            agents.remove(a)


def source_has_tail():
    """The token producer of umma_cta stays until the commits of its last stages have arrived."""
    text = open(SOURCE).read()
    body = text[text.index("void umma_cta("):]
    producer = body[body.index("token-operand producer"):body.index("packed-weight producer")]
    walks_on = re.search(r"bool await_last_commits\(.*?\n}\n", text, re.S)
    return ("await_last_commits<S>(bars, p)" in producer and walks_on is not None
            and "bars->empty[p.stage]), p.phase ^ 1" in walks_on.group(0))


RINGS = [(1, 3, 3), (1, 3, 4), (1, 4, 0), (2, 6, 6), (2, 6, 0)]     # CTAs per tile, stages, stages of codes (0: bf16 weights)


@pytest.mark.parametrize("ctas,stages,code_stages", RINGS)
def test_ctas_of_a_tile_from_first_step_to_exit(ctas, stages, code_stages):
    for seed in range(150):
        for items, steps in ((1, 2), (2, 7), (5, 4)):
            walk_ctas(ctas, stages, code_stages, items, steps, random.Random(seed), tail=source_has_tail())


WRONG = {"exit before the last commits": dict(tail=False), "bytes of one CTA": dict(announced=1),
         "no wait in the second CTA": dict(waits=lambda r: r == 0), "commits to the first CTA": dict(commits=lambda r: r == 0)}


@pytest.mark.parametrize("ctas,stages,code_stages,wrong",
                         [(*ring, w) for ring in RINGS for w in WRONG if ring[0] == 2 or w == "exit before the last commits"])
def test_the_model_of_the_ctas_tells_wrong_protocols(ctas, stages, code_stages, wrong):
    with pytest.raises(AssertionError):
        for seed in range(400):
            walk_ctas(ctas, stages, code_stages, 3, 7, random.Random(seed), **WRONG[wrong])

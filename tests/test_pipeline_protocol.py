"""The order in which a group of unpacker warps waits for its two barriers (csrc/umma_gemm.cu, expand_codes), as a model
on the CPU.

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


@pytest.mark.parametrize("stages,code_stages", [(3, 3), (3, 4), (6, 6)])     # INT8 codes; 2-bit and 4-bit ones; pairs of CTAs
def test_unpackers_meet_the_codes_of_their_own_step(stages, code_stages):
    for seed in range(400):
        walk(source_order(), stages, code_stages, 24, random.Random(seed))


def test_the_model_tells_the_orders_apart():
    with pytest.raises(AssertionError):
        for seed in range(400):
            walk(["full_p", "empty"], 3, 3, 24, random.Random(seed))

"""A model, on the CPU, of how a CTA with two producers leaves after a wait that ran out (decode_tc.cu,
prefill.cu, gemm_tc.cu).

Producer A arms a stage's barrier with all its bytes and copies the weights, producer B copies the other
operand into the same stage; each first waits (bounded) until the MMAs have read the stage's last
use. A closes by waiting for the last use of every stage that it armed. If A gives up and B does not, B's
copy completes no phase, so that A's closing wait does not cover it.

The safety property: no copy lands after the CTA has left. The kernels get it by a producer that gave up
staying 100 ms longer; the model checks random delays and limits, and that the closing wait alone
breaks it.
"""
import math
import random

import pytest

CLOSE = 100e6  # ns, the bound of the closing waits and the stay of a producer that gave up


def late_copies(rng, stages, total, limit, stay):
    """One random run of a CTA: the number of copies that land after it has left."""
    hold = lambda: rng.choice([0.0, rng.uniform(0, 50), rng.uniform(0, 20000)])  # a thread held up
    t = {"A": 0.0, "B": rng.uniform(0, 5000), "M": 0.0}  # B also waits for the kernel before
    dead = {"A": False, "B": False, "M": False}
    armed, landed_a, landed_b, consumed = ([math.inf] * total for _ in range(4))

    def wait(who, event):
        t[who] += hold()
        if event <= t[who] + limit:
            t[who] = max(t[who], event)
        else:
            t[who] += limit
            dead[who] = True
        return not dead[who]

    for it in range(total):
        free = consumed[it - stages] if it >= stages else 0.0
        for who, landed in (("A", landed_a), ("B", landed_b)):
            if not dead[who] and wait(who, free):
                if who == "A":
                    armed[it] = t["A"]
                landed[it] = t[who] + rng.uniform(500, 20000)
        if not dead["M"] and wait("M", max(armed[it], landed_a[it], landed_b[it])):
            consumed[it] = t["M"] + rng.uniform(100, 500)
    n = sum(a < math.inf for a in armed)
    for it in range(max(0, n - stages), n):  # A's closing waits
        t["A"] = max(t["A"], min(t["A"] + CLOSE, max(landed_a[it], landed_b[it])))
    if stay:
        for who in "AB":
            t[who] += CLOSE if dead[who] else 0.0
    return sum(x < math.inf and x > max(t.values()) for x in landed_a + landed_b)


@pytest.mark.parametrize("limit", [1.0, 3e3, 1e4, 1e6, 1e9])
def test_no_copy_lands_after_a_cta_whose_producers_gave_up_has_left(limit):
    rng = random.Random(int(limit))
    for _ in range(600):
        assert late_copies(rng, rng.randint(2, 8), rng.randint(1, 24), limit, stay=True) == 0


def test_the_closing_wait_alone_lets_copies_land_late():
    rng = random.Random(5)
    assert sum(late_copies(rng, rng.randint(2, 8), rng.randint(1, 24), 3e3, stay=False) for _ in range(600)) > 0

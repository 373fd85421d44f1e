"""Which phase of a barrier a wait can meet: the roles of the forward at d = 256, walked through in random order.

A parity wait tells two neighbouring phases apart and no more.  A wait for phase p is sound if, whenever it is polled, p - 1 has
completed and p + 1 has not; otherwise it passes too early or never.  The model holds the roles' waits, arrivals and commits:
loads complete in any order, the products of one issuing thread in issue order, every role as early or late as it likes.
"""
import random

import pytest

STAGES = 2     # of K and V, of S / P


class Barrier:
    def __init__(self, count=1):
        self.count, self.pending, self.phase = count, count, 0     # phase: completions so far

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending, self.phase = self.count, self.phase + 1


def poll(bar, phase):
    assert phase <= bar.phase <= phase + 1, f"a wait for phase {phase} meets a barrier at phase {bar.phase}"
    return bar.phase == phase + 1


def run(tiles, rng, o_barrier):
    """`o_barrier`: a barrier of its own that completes with every tile's product, committed behind the release of the stage."""
    full, empty, S = ([Barrier() for _ in range(STAGES)] for _ in range(3))
    P = [Barrier(2) for _ in range(STAGES)]
    met, O = Barrier(2), Barrier()
    loads, products = [], {"S": [], "PV": []}     # not complete yet
    sees_all = [rng.random() < 0.5 for _ in range(2)]

    def loader():
        for k in range(tiles):
            if k >= STAGES:
                yield empty[k % STAGES], k // STAGES - 1
            loads.append(full[k % STAGES])

    def scores():
        for k in range(tiles):
            yield full[k % STAGES], k // STAGES
            products["S"].append([S[k % STAGES]])

    def values():
        for k in range(tiles):
            yield P[k % STAGES], k // STAGES
            products["PV"].append([empty[k % STAGES]] + ([O] if o_barrier else []))

    def softmax(w):
        for k in range(tiles):
            yield S[k % STAGES], k // STAGES
            met.arrive()
            yield met, k
            if k > 0 and (sees_all[w] or rng.random() < 0.3):      # O is rescaled
                yield (O, k - 1) if o_barrier else (empty[(k - 1) % STAGES], (k - 1) // STAGES)
            P[k % STAGES].arrive()
        if not o_barrier:
            yield empty[(tiles - 1) % STAGES], (tiles - 1) // STAGES

    roles = {r: next(r, None) for r in (loader(), scores(), values(), softmax(0), softmax(1))}
    while any(roles.values()) or loads or any(products.values()):
        asleep = rng.randrange(9)      # one actor is held back for a while
        for _ in range(40):
            i = rng.randrange(8)
            if i == asleep:
                continue
            if i < 5:
                role = list(roles)[i]
                if roles[role] and poll(*roles[role]):
                    roles[role] = next(role, None)
            elif i == 5:
                if loads:
                    loads.pop(rng.randrange(len(loads))).arrive()
            else:
                queue = products["S" if i == 6 else "PV"]
                if queue:                                           # commits of one product complete one after the other
                    queue[0].pop(0).arrive()
                    if not queue[0]:
                        queue.pop(0)


@pytest.mark.parametrize("tiles", [1, 2, 3, 4, 7, 12])
def test_forward_of_256_waits_within_one_phase(tiles):
    for seed in range(300):
        run(tiles, random.Random(seed), o_barrier=False)


def test_a_barrier_committed_behind_the_release_is_met_two_phases_late():
    with pytest.raises(AssertionError, match="meets a barrier"):
        for seed in range(2000):
            run(12, random.Random(seed), o_barrier=True)


def give_up(rng, loader_stops, issuer_stops, tiles=12, stages=2):
    """A ring of stages in which some wait runs out although nothing is wrong (the CTA was not scheduled for a while): from then on
    every wait that is not fulfilled fails at once.  Asserts that no barrier is armed while a load for it is on its way."""
    full, empty = [0] * stages, [0] * stages      # completed phases
    on_their_way, late, steps = [], [False], 0

    def wait(bars, s, phase):
        while bars[s] <= phase and not late[0]:
            yield
        return bars[s] > phase

    def loader():
        for k in range(tiles):
            if k >= stages and not (yield from wait(empty, k % stages, k // stages - 1)) and loader_stops:
                return
            assert k % stages not in on_their_way, "armed twice in one phase"
            on_their_way.append(k % stages)
            yield

    def issuer():
        for k in range(tiles):
            if not (yield from wait(full, k % stages, k // stages)) and issuer_stops:
                return
            empty[k % stages] += 1
            yield

    roles = [loader(), issuer()]
    while roles:
        steps += 1
        late[0] = late[0] or rng.random() < 0.03
        if on_their_way and rng.random() < 0.2:
            full[on_their_way.pop(rng.randrange(len(on_their_way)))] += 1
        role = rng.choice(roles)
        try:
            next(role)
        except StopIteration:
            roles.remove(role)
    assert steps < 2000


def test_a_loading_and_an_issuing_thread_that_stop_arm_no_barrier_twice():
    for seed in range(2000):
        give_up(random.Random(seed), True, True)


@pytest.mark.parametrize("loader_stops,issuer_stops", [(False, False), (True, False), (False, True)])
def test_one_that_goes_on_arms_a_barrier_twice(loader_stops, issuer_stops):
    with pytest.raises(AssertionError, match="armed twice"):
        for seed in range(2000):
            give_up(random.Random(seed), loader_stops, issuer_stops)

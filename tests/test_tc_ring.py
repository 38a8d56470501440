"""The barrier protocol of the tcgen05 kernel's rings, as a model on the CPU under adversarial schedules.

A parity wait passes when the barrier's running phase has the other parity.  So it is wrong in both directions for a waiter
that has lost count: it passes early when the phase before the wanted one is still running, and not at all when the wanted one
was followed by another before the waiter looked.  Every role of the kernel is a process here, and each wait states the phase it means;
the model checks that it passes exactly on that phase and that no schedule ends in a standstill.
"""
import random

import pytest


class Barrier:
    def __init__(self, count):
        self.count, self.left, self.phase = count, count, 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.phase = self.count, self.phase + 1

    def passes(self, n):
        """try_wait.parity(n & 1); a pass must mean that phase n, and no later one, is complete."""
        if (self.phase & 1) == (n & 1):
            assert self.phase <= n, f"phase {n} was missed: the barrier is in phase {self.phase}"
            return False
        assert self.phase == n + 1, f"passed for phase {n} while the barrier is in phase {self.phase}"
        return True


# Restated from fq_tc_kernel.cuh (tc_stages, TcShape): tensor memory and shared memory of a launch
def shape(nr, gps, nmma):
    ndb = next(d for d in (4, 2, 1) if d == 1 or (4 if d == 4 else 2) * 64 + d * gps * nr + nr <= 512)
    nab = 4 if 4 * 64 + ndb * gps * nr + nr <= 512 else 2
    ug, sg = 3 if nr == 16 else 2, 3 if nr <= 32 else 2 if nr <= 64 else 1
    stage = -(-(256 * nmma + 8192 + 512 * gps) // 1024) * 1024
    s = min(12, (232448 - 2048 - (2 if sg == 1 else sg) * 32768) // stage)
    return dict(S=s - s % ug if s >= 2 * ug else s, UG=ug, NAB=nab, NDB=ndb, XB=nr <= 32)


def run(S, UG, NAB, NDB, XB, units, order, rng, drop=None):
    """XB: the activations' arrival in a stage has barriers of its own; else both producers arrive on the stage's one."""
    full, empty = [Barrier(1 if XB else 2) for _ in range(S)], [Barrier(4) for _ in range(S)]
    x_full = [Barrier(1) for _ in range(S)] if XB else full
    a_full, a_empty = [Barrier(1) for _ in range(NAB)], [Barrier(1) for _ in range(NAB)]
    d_full, d_free = [Barrier(1) for _ in range(NDB)], [Barrier(1) for _ in range(NDB)]
    mmas = []                                              # issued, not yet complete
    codes_here, x_here = set(), set()                      # units whose copies have landed

    def producer(loads):
        for it in range(units):
            while it >= S and not empty[it % S].passes(it // S - 1):
                yield
            loads.append(it)
            yield

    def landing(loads, barriers, here):                    # copies land in any order, those of the two producers independently
        done = 0
        while done < units:
            if loads:
                it = loads.pop(rng.randrange(len(loads)))
                here.add(it)
                barriers[it % S].arrive()
                done += 1
            yield

    def unpack(ug):
        for it in range(units):
            ab, mine = it % NAB, it % UG == ug
            if not mine and order != "visits others":
                continue
            if order == "operand first" and it >= NAB:
                while not a_empty[ab].passes(it // NAB - 1):
                    yield
            while not full[it % S].passes(it // S):
                yield
            if not mine:
                continue
            assert it in codes_here, "codes are not here"
            yield
            if order != "operand first" and it >= NAB:
                while not a_empty[ab].passes(it // NAB - 1):
                    yield
            yield
            a_full[ab].arrive()
            empty[it % S].arrive()

    def dense():
        ready = False
        for it in range(units):
            if not ready:
                while it >= NDB and not d_free[it % NDB].passes(it // NDB - 1):
                    yield
                while XB and drop != "dense warp's wait for X" and not x_full[it % S].passes(it // S):
                    yield
                while not a_full[it % NAB].passes(it // NAB):
                    yield
            assert it in x_here, "the dense MMAs' activations are not here"     # (without XB the unpack group has waited for them)
            nx = it + 1                                    # the next unit's barriers, looked at once
            ready = nx < units and a_full[nx % NAB].passes(nx // NAB) and (nx < NDB or d_free[nx % NDB].passes(nx // NDB - 1))
            yield
            mmas.append(it)
            if XB and drop != "dense warp's wait for X" and nx < units:
                ready = x_full[nx % S].passes(nx // S) and ready
            yield

    def tensor_pipe():                                     # MMAs retire in order
        for it in range(units):
            while not mmas:
                yield
            assert mmas.pop(0) == it
            for b in (d_full[it % NDB], a_empty[it % NAB], empty[it % S]):
                b.arrive()
            yield

    def drain():
        for it in range(units):
            while not full[it % S].passes(it // S):
                yield
            assert it in codes_here, "scales are not here"
            empty[it % S].arrive()
            while not d_full[it % NDB].passes(it // NDB):
                yield
            d_free[it % NDB].arrive()

    def outliers():
        for it in range(units):
            while drop != "outlier warp's wait for X" and not x_full[it % S].passes(it // S):
                yield
            assert it in x_here, "the outlier MMAs' activations are not here"
            yield
            empty[it % S].arrive()

    codes, xs = [], []                                     # copies under way
    procs = [producer(codes), producer(xs), landing(codes, full, codes_here), landing(xs, x_full, x_here), dense(), tensor_pipe(), drain(),
             outliers()] + [unpack(g) for g in range(UG)]
    weight = [10 ** rng.uniform(-2, 0) for _ in procs]     # some much slower than others
    live = list(range(len(procs)))
    for _ in range(4000 * units):
        if not live:
            return
        i = rng.choices(live, [weight[j] for j in live])[0]
        if next(procs[i], "end") == "end":
            live.remove(i)
        if rng.random() < 0.01:
            weight[rng.randrange(len(procs))] = 10 ** rng.uniform(-2, 0)
    raise AssertionError("standstill")


@pytest.mark.parametrize("nr", [16, 32, 64, 128])
@pytest.mark.parametrize("gps", [1, 2])
def test_every_wait_meets_its_phase(nr, gps):
    rng = random.Random(100 * nr + gps)
    for nmma in range(max(16, nr // 2 + 16), nr + 1, 16):
        sh = shape(nr, gps, nmma)
        assert sh["S"] >= sh["NAB"]
        order = "stage first" if sh["S"] >= sh["UG"] + sh["NAB"] else "operand first"
        assert order == "stage first" or nr == 128
        for _ in range(40):
            run(**sh, units=rng.randint(1, 30), order=order, rng=rng)


@pytest.mark.parametrize("order", ["visits others", "stage first"])
def test_the_ring_of_three_stages_needs_the_operand_first(order):
    """113 to 128 rows: three stages, two unpack groups.  Waiting for the other group's units too, without releasing them, can miss a
    phase; waiting for the stage first can pass on the phase before."""
    sh = shape(128, 1, 128)
    assert sh["S"] == 3 and sh["UG"] == 2 and sh["NAB"] == 2
    rng = random.Random(1)
    with pytest.raises(AssertionError, match="phase"):
        for _ in range(400):
            run(**sh, units=30, order=order, rng=rng)


@pytest.mark.parametrize("drop", ["dense warp's wait for X", "outlier warp's wait for X"])
@pytest.mark.parametrize("nr", [16, 32])
def test_neither_tensor_warp_may_drop_its_wait_for_the_activations(nr, drop):
    """Up to 32 rows the unpack warps do not wait for X, so that nobody else's wait covers it."""
    sh, rng = shape(nr, 1, nr), random.Random(2)
    with pytest.raises(AssertionError, match=f"the {drop.split()[0]} MMAs' activations"):
        for _ in range(400):
            run(**sh, units=30, order="stage first", rng=rng, drop=drop)

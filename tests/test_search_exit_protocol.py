"""A host-side model of how the epilogue warps of the tensor-core search
(csrc/knn_tc.cu) leave their loops when a bounded wait runs out or another role
raises the abort flag, run under random schedules on the CPU.

The loops hold operations that all 32 lanes must execute together: votes and
reductions over the full mask and tensor-memory loads.  What a lane observes is its
own: the abort flag is set by another warp at any time, so two lanes of one test may
read different values, and a wait near its limit may succeed in one lane and run out
in another.  The model runs the control flow of one warp, lane by lane in random
order, each lane up to its next collective, and fails when lanes wait in different
ones or some have left while others wait.  The kernel's form votes on every such
observation before acting on it; with the observations taken lane by lane (the
planted form) the mismatch is caught."""
import random

import pytest

LANES = 32


class _Mismatch(Exception):
    pass


def _lane(obs, items, tiles, voted, log):
    """The control flow of one lane.  Yields (site, value) at a collective and gets
    back the values of all lanes; obs(kind) is what this lane observes."""
    if voted:
        ok, item = True, 0
        while item < items and ok:
            if any((yield ("abort at item", obs("abort")))):
                break
            for _ in range(tiles):
                if any((yield ("abort at tile", obs("abort")))):
                    ok = False
                    break
                if any((yield ("update vote", obs("update")))):
                    yield ("flush", None)
                ok = all((yield ("wait", obs("wait"))))
                if not ok:
                    break
                yield ("tensor memory load", None)
                yield ("admission vote", None)
            if ok:
                yield ("flush", None)
            item += 1
    else:
        item = 0
        while item < items and not obs("abort"):
            for _ in range(tiles):
                if obs("abort"):
                    break
                if any((yield ("update vote", obs("update")))):
                    yield ("flush", None)
                if not obs("wait"):
                    break
                yield ("tensor memory load", None)
                yield ("admission vote", None)
            yield ("flush", None)
            item += 1
    log.append("left")


def _run(seed, voted, abort_after=None, failing_wait=None):
    """abort_after: observations of the flag before it is set; failing_wait: the
    tile whose wait is at its limit (each lane's outcome is random there)."""
    rng = random.Random(seed)
    reads = [0]
    waits = [0] * LANES
    log = []

    def observer(lane):
        def obs(kind):
            if kind == "abort":
                reads[0] += 1
                return abort_after is not None and reads[0] > abort_after
            if kind == "wait":
                waits[lane] += 1
                return not (failing_wait is not None and waits[lane] - 1 == failing_wait and rng.random() < 0.5)
            return rng.random() < 0.1
        return obs

    lanes = {i: _lane(observer(i), 3, 4, voted, log) for i in range(LANES)}
    at = {}
    send = {i: None for i in lanes}
    steps = 0
    while lanes:
        order = list(lanes)
        rng.shuffle(order)
        for i in order:
            try:
                at[i] = lanes[i].send(send[i])
            except StopIteration:
                del lanes[i]
                at.pop(i, None)
        if not lanes:
            break
        if len(lanes) != LANES or len({site for site, _ in at.values()}) != 1:
            raise _Mismatch({site for site, _ in at.values()})
        values = [at[i][1] for i in range(LANES)]
        send = {i: values for i in lanes}
        steps += 1
        assert steps < 1000
    assert len(log) == LANES
    return steps


@pytest.mark.parametrize("seed", range(40))
def test_lanes_leave_together(seed):
    whole = _run(seed, True)
    assert _run(seed, True, abort_after=random.Random(seed).randrange(0, 32 * 15)) <= whole + 24
    _run(seed, True, failing_wait=seed % 12)


def test_observations_of_single_lanes_are_caught():
    def caught(**kw):
        n = 0
        for seed in range(40):
            try:
                _run(seed, False, **kw)
            except _Mismatch:
                n += 1
        return n
    assert caught() == 0  # without a timeout both forms agree
    assert caught(failing_wait=5) == 40
    assert caught(abort_after=5 * LANES + 7) == 40

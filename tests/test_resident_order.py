"""CPU model of the order of the ring exchange of lattices kept on the chip (csrc/lbm_resident.cuh).

Each tile's warps run as in the kernel: in a step they take pieces of the inbox until none is left, meet at a
barrier, meet again after the pulls, and then each sends its rows (and the ghosts of its edge tasks) by itself and goes
on to the next step's pieces.  A scheduler runs one warp's next action at a time, any warp of any tile, some of them
held back for long.  Whatever it does: no value is overwritten before its reader has read it, every reader gets
the value of the step that it waits for, and somebody can always go on."""
import random
from collections import defaultdict

import pytest

from test_resident_exchange import Tile, receives, sends


class Lost(AssertionError):
    pass


class Model:
    def __init__(self, rng, nx, nr, ns, nb, bc, W, TH, warps, halves=2):
        self.rng, self.halves, self.warps = rng, halves, warps
        tiles = [Tile(nx, nr, ns, nb, t) for t in range(ns * nb)]
        self.n = len(tiles)
        # what warp w of tile n sends: (tile, entry); rows belong to their warp, ghosts to an edge task's
        self.out = defaultdict(list)
        for n, a in enumerate(tiles):
            for t, e, _, (i, j) in sends(tiles, n, nx, nr, ns, nb, bc, W, TH):
                row = (j - a.j0) * warps // max(a.h, 1)
                who = row if a.has(i, j) else 6 * (i + j) % 7  # (any warp: the model leaves the tasks to chance)
                self.out[n, min(max(who, 0), warps - 1)].append((t, e))
        # the pieces of each tile's inbox
        self.pieces = []
        for a in tiles:
            entries = sorted(e for e, *_ in receives(a, nx, nr, bc, W, TH))
            size = max(1, len(entries) // 5)
            self.pieces.append([entries[k:k + size] for k in range(0, len(entries), size)])
        self.box = {}     # (tile, half, entry) -> (state number, read)
        self.base = 0

    def put(self, t, e, seq):
        slot = (t, seq % self.halves, e)
        if slot in self.box and not self.box[slot][1]:
            raise Lost(f"state {self.box[slot][0]} of {slot} overwritten by {seq} before it was read")
        self.box[slot] = (seq, False)

    def warp(self, n, w, steps, shared):
        """One warp of a tile, as a generator: yields None after an action, or a condition to wait for."""
        for k in range(steps):
            seq = self.base + k
            if k > 0:
                while shared["taken"] < len(self.pieces[n]):
                    piece = self.pieces[n][shared["taken"]]
                    shared["taken"] += 1
                    for e in piece:
                        slot = (n, seq % self.halves, e)
                        yield lambda slot=slot: self.box.get(slot, (None,))[0] == seq
                        self.box[slot] = (seq, True)
            for point in ("pulled", "moments"):
                shared[point, k] = shared.get((point, k), 0) + 1
                yield lambda key=(point, k): shared[key] == self.warps
                if point == "pulled":
                    shared["taken"] = 0
            if k + 1 < steps:
                mine = list(self.out[n, w])
                self.rng.shuffle(mine)
                for t, e in mine:
                    self.put(t, e, seq + 1)
                    yield None

    def launch(self, steps):
        runs = []
        for n in range(self.n):
            shared = {"taken": 0}
            runs += [[self.warp(n, w, steps, shared), None, self.rng.random() < 0.3] for w in range(self.warps)]
        while runs:
            ready = [r for r in runs if r[1] is None or r[1]()]
            assert ready, "every warp waits"
            quick = [r for r in ready if not r[2]]
            r = self.rng.choice(quick if quick and self.rng.random() < 0.98 else ready)
            for _ in range(self.rng.choice((1, 4, 40))):  # a run of its actions
                try:
                    r[1] = next(r[0])
                except StopIteration:
                    runs.remove(r)
                    break
                if r[1] is not None and not r[1]():
                    break
            if self.rng.random() < 0.01:
                r[2] = not r[2]
        self.base += steps


def model(seed, halves=2):
    rng = random.Random(seed)
    bc = dict(bottom=rng.choice(("axis", "wall")), top=rng.choice(("wall", "open")), out=rng.choice(("outflow", "wall")))
    W, TH, ns, nb = 4, 4, rng.randint(1, 3), rng.randint(1, 3)
    if ns * nb == 1:
        ns = 2
    nx = rng.randint(2 * ns if ns > 1 else 1, W * ns)
    nr = rng.randint(2 * nb if nb > 1 else 1, TH * nb)
    return Model(rng, nx, nr, ns, nb, bc, W, TH, rng.randint(1, 3), halves)


@pytest.mark.parametrize("seed", range(60))
def test_no_value_is_lost_in_any_order(seed):
    m = model(seed)
    for steps in (5, 2, 4):  # launches of odd and even counts carry the numbers on
        m.launch(steps)


def test_the_model_sees_a_lost_value():
    """With one half instead of two, a sender a step ahead of its reader overwrites what is still to be read."""
    lost = 0
    for seed in range(12):
        try:
            model(seed, halves=1).launch(6)
        except Lost:
            lost += 1
    assert lost > 0

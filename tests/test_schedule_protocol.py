"""Host-side checks of the scoring kernel's schedule and of the hand-over of the softmax
statistics between its blocks (Eq. 1 needs each window row's normaliser over ALL keys before
any probability can be summed, so blocks that share a unit exchange partial log-sum-exps).

The item lists come from the library itself (snapkv_schedule_items and its counterpart for ragged
batches run the kernel's own item walk on the host).  The hand-over is modelled with three CPU threads
per block, as the kernel has warps: one walks the items, leaves its statistics in two buffers and adds up
votes; the publisher takes them from there and writes the partials (a written slot is its own flag); the
fetcher provides, for every vote item, the unit's row, eight rows ahead at most: it looks until every slot
is written, with a time limit, and folds them in slot order.  Where the fold is shared the publisher folds
the upper half of each row of a wave once it has published the wave's partials, and a row is there when
both halves are.  In a ragged batch the block with slot 0 folds, one wave ahead of the votes, and the
others wait for its row.  The model shows that the schedule cannot deadlock, that every block gets the
same row whatever the thread timing, that a block which never arrives turns into time-outs, not into a
hang, and that a phase with more vote items than row buffers must not share the fold."""
import queue
import threading
import time

import pytest

from paper_2404_14469_b200 import binding as sk

SHAPES = [
    # B, Hq, Hkv, L, d, W, grid
    (4, 32, 8, 32768, 128, 32, 148),    # workload 2
    (1, 32, 32, 16384, 128, 32, 148),   # workload 1
    (1, 32, 8, 131072, 128, 64, 148),   # workload 3: two head sub-groups per KV head
    (1, 32, 32, 380000, 128, 32, 148),  # workload 4: one unit per wave
    (1, 4, 4, 1024, 64, 32, 148),       # fewer tiles than blocks
    (2, 4, 2, 1000, 128, 32, 7),        # ragged, small grid
    (3, 2, 2, 257, 64, 32, 192),
    (1, 8, 1, 900, 64, 32, 33),
]


def _all_items(B, Hq, Hkv, L, d, W, grid, votes_only=False):
    per_cta, plan = [], None
    for c in range(grid):
        items, plan = sk.snapkv_schedule_items(B, Hq, Hkv, L, d, W, grid, c, votes_only)
        per_cta.append(items)
    return per_cta, plan


@pytest.mark.parametrize("B,Hq,Hkv,L,d,W,grid", SHAPES)
def test_every_tile_is_covered_once_and_slots_are_dense(B, Hq, Hkv, L, d, W, grid):
    per_cta, plan = _all_items(B, Hq, Hkv, L, d, W, grid)
    for vote, T in ((0, plan["tiles_stats"]), (1, plan["tiles_vote"])):
        seen = {}
        for c, items in enumerate(per_cta):
            for unit, t0, t1, v, slot, nseg in items:
                if v != vote:
                    continue
                assert 0 <= t0 < t1 <= T and 0 <= unit < plan["units"]
                for t in range(t0, t1):
                    assert (unit, t) not in seen, "a tile is handed out twice"
                    seen[(unit, t)] = c
        assert len(seen) == plan["units"] * T
    # statistics sweep: the blocks that share a unit hold slots 0 .. nseg-1, once each, and
    # all of them agree on nseg, which fits the workspace's partial slots
    slots = {}
    for items in per_cta:
        for unit, t0, t1, v, slot, nseg in items:
            if v == 0:
                slots.setdefault(unit, []).append((slot, nseg))
    for unit, lst in slots.items():
        nsegs = {n for _, n in lst}
        assert len(nsegs) == 1
        nseg = nsegs.pop()
        assert sorted(s for s, _ in lst) == list(range(nseg))
        assert nseg <= plan["maxseg"]
    # vote items carry the nseg of their unit's statistics sweep
    for items in per_cta:
        for unit, t0, t1, v, slot, nseg in items:
            if v == 1:
                assert nseg == len(slots[unit])


@pytest.mark.parametrize("B,Hq,Hkv,L,d,W,grid", SHAPES)
def test_a_block_reaches_a_units_votes_only_after_its_own_statistics(B, Hq, Hkv, L, d, W, grid):
    per_cta, plan = _all_items(B, Hq, Hkv, L, d, W, grid)
    # where each block has its statistics items of a unit
    own = [{} for _ in per_cta]
    for c, items in enumerate(per_cta):
        for i, (unit, t0, t1, v, slot, nseg) in enumerate(items):
            if v == 0:
                own[c][unit] = max(own[c].get(unit, -1), i)
    for c, items in enumerate(per_cta):
        for i, (unit, t0, t1, v, slot, nseg) in enumerate(items):
            if v == 1 and unit in own[c]:
                assert own[c][unit] < i   # else the block would wait for itself


def test_votes_only_schedule_is_one_phase_without_statistics():
    per_cta, plan = _all_items(2, 8, 2, 5000, 128, 32, 148, votes_only=True)
    assert plan["waves"] == 1
    assert all(v == 1 for items in per_cta for (_, _, _, v, _, _) in items)
    tiles = sum(t1 - t0 for items in per_cta for (_, t0, t1, _, _, _) in items)
    assert tiles == plan["units"] * plan["tiles_vote"]


RAGGED = [
    # lens, Hq, Hkv, d, W, grid
    ([24000, 5012, 1353, 9000, 600, 2047], 32, 8, 128, 32, 148),
    ([300, 129, 700, 17], 8, 2, 128, 16, 148),          # fewer tiles than blocks in every sequence
    ([60000, 1000, 70000, 50000], 16, 8, 128, 32, 148),  # several waves in a sequence
    ([900, 5000, 33], 8, 1, 64, 32, 7),                  # two head sub-groups, small grid
]


@pytest.mark.parametrize("lens,Hq,Hkv,d,W,grid", RAGGED)
def test_a_ragged_batch_is_cut_as_the_calls_one_by_one(lens, Hq, Hkv, d, W, grid):
    # block c has, of sequence i, what block (c + 53 i) % grid has in a call on that sequence alone: the
    # same tiles, slots and counts of slots, so that results do not depend on the batch
    ragged = [sk.ragged_schedule_items(lens, Hq, Hkv, d, W, grid, c) for c in range(grid)]
    for i, L in enumerate(lens):
        alone, _ = _all_items(1, Hq, Hkv, L, d, W, grid)
        for c in range(grid):
            assert [x[:6] for x in ragged[c] if x[6] == i and x[3] == 0] == \
                [x for x in alone[(c + 53 * i) % grid] if x[3] == 0]
            assert [x[:6] for x in ragged[c] if x[6] == i and x[3] == 1] == \
                [x for x in alone[(c + 53 * i) % grid] if x[3] == 1]


@pytest.mark.parametrize("lens,Hq,Hkv,d,W,grid", RAGGED)
def test_statistics_of_the_next_wave_come_before_a_waves_votes(lens, Hq, Hkv, d, W, grid):
    # what the folding blocks of a ragged batch rely on; waves are numbered through the launch
    waves = {}
    for c in range(grid):
        items = sk.ragged_schedule_items(lens, Hq, Hkv, d, W, grid, c)
        done = [-1, -1]
        for unit, t0, t1, vote, slot, nseg, seq, wave in items:
            assert wave >= done[vote]                       # each sweep in the order of the waves
            done[vote] = wave
            if vote == 0:
                waves.setdefault(wave, seq)
                assert waves[wave] == seq
        order = [(x[7], x[3]) for x in items]
        for at, (wave, vote) in enumerate(order):
            if vote:                                        # none of waves 0 .. wave + 1 is still to come
                assert not any(v == 0 and w <= wave + 1 for w, v in order[at:])


PARTIAL_BUFFERS, ROW_BUFFERS = 2, 8


class _Model:
    """Three threads per block; `absent` blocks never run.  Items are (unit key, vote, slot, nseg, wave).
    `shared`: the publisher folds the upper halves."""

    def __init__(self, per_cta, limit_s, ragged, shared):
        self.per_cta, self.limit, self.ragged, self.shared = per_cta, limit_s, ragged, shared
        self.slots, self.rows = {}, {}                    # (key, slot) -> partial; key -> row
        self.abort = [0] * len(per_cta)
        self.got = [[] for _ in per_cta]
        self.waves = 1 + max(x[4] for items in per_cta for x in items)

    def _wait(self, c, ready, limit, code):
        t_end = time.monotonic() + limit
        while not ready():
            if self.abort[c]:
                return False
            if time.monotonic() > t_end:
                self.abort[c] = self.abort[c] or code
                return False
            time.sleep(1e-4)
        return True

    # waits inside a block; the codes are the kernel's
    def _put(self, c, q, x, code):
        return self._wait(c, lambda: not q.full(), self.limit, code) and (q.put(x) or True)

    def _get(self, c, q, code):
        return q.get() if self._wait(c, lambda: not q.empty(), self.limit, code) else None

    # waits for other blocks: half the limit, and the code of the wait for a unit's statistics
    def _fold(self, c, key, nseg, half):
        if not self._wait(c, lambda: all((key, s) in self.slots for s in range(nseg)), self.limit / 2, 7):
            return None
        acc = half
        for s in range(nseg):                             # slot order: the same in every block
            acc = acc * 31 + self.slots[key, s]
        return acc

    def _items(self, c, vote, wave):
        return [x for x in self.per_cta[c] if x[1] == vote and x[4] == wave]

    def publisher(self, c, partials, upper):
        for w in range(self.waves):
            for key, _, slot, _, _ in self._items(c, 0, w):
                got = self._get(c, partials, 9)
                if got is None:
                    return
                assert got[0] == (key, slot), "partials come in the order of the items"
                self.slots[got[0]] = got[1]
            for key, _, _, nseg, _ in self._items(c, 1, w) if self.shared else ():
                row = self._fold(c, key, nseg, 1)
                if row is None or not self._put(c, upper, (key, row), 11):
                    return

    def fetcher(self, c, lower):
        for w in range(-1 if self.ragged else 0, self.waves):
            if self.ragged:
                for key, _, slot, nseg, _ in self._items(c, 0, w + 1):
                    if slot == 0:
                        row = self._fold(c, key, nseg, 0)
                        if row is None:
                            return
                        self.rows[key] = row
            for key, _, _, nseg, _ in self._items(c, 1, w):
                if self.ragged:
                    row = self.rows[key] if self._wait(c, lambda: key in self.rows, self.limit / 2, 7) else None
                else:
                    row = self._fold(c, key, nseg, 0)
                if row is None or not self._put(c, lower, (key, row), 11):
                    return

    def softmax(self, c, partials, halves, jitter):
        for k, (key, vote, slot, nseg, wave) in enumerate(self.per_cta[c]):
            if jitter:
                time.sleep(((c * 7 + k * 3) % 5) * 1e-4)
            if not vote:                                  # (the number stands for the block's partial)
                if not self._put(c, partials, ((key, slot), (hash(key) % 1009 + 1) * 1000 + slot), 8):
                    return
                continue
            row = ()
            for half in halves:                           # a row is there when all its parts are
                got = self._get(c, half, 10)
                if got is None:
                    return
                assert got[0] == key, "rows come in the order of the items"
                row += (got[1],)
            self.got[c].append((key, row))

    def run(self, absent=(), jitter=True):
        threads = []
        for c in range(len(self.per_cta)):
            if c not in absent:
                partials = queue.Queue(maxsize=PARTIAL_BUFFERS)
                halves = [queue.Queue(maxsize=ROW_BUFFERS) for _ in range(2 if self.shared else 1)]
                threads += [threading.Thread(target=self.fetcher, args=(c, halves[0])),
                            threading.Thread(target=self.publisher, args=(c, partials, halves[-1])),
                            threading.Thread(target=self.softmax, args=(c, partials, halves, jitter))]
        t0 = time.monotonic()
        for t in threads:
            t.start()
        for t in threads:
            t.join(timeout=30)
        assert not any(t.is_alive() for t in threads), "the model hangs"
        return time.monotonic() - t0


def _model(shape, limit_s, shared=False):
    """Of one length (B, Hq, Hkv, L, d, W, grid) or of a ragged batch ([lengths], Hq, Hkv, d, W, grid)."""
    if isinstance(shape[0], list):
        items = [[((x[6], x[0]), x[3], x[4], x[5], x[7]) for x in sk.ragged_schedule_items(*shape, c)]
                 for c in range(shape[-1])]
        return _Model(items, limit_s, True, shared)
    per_cta, plan = _all_items(*shape)
    return _Model([[(x[0], x[3], x[4], x[5], x[0] // plan["units_per_wave"]) for x in items] for items in per_cta],
                  limit_s, False, shared)


# (shape, whether the fold is shared)
HAND_OVER = [
    ((2, 8, 2, 3000, 128, 32, 24), False), ((1, 4, 4, 1024, 64, 32, 40), False),
    (([3000, 700, 150, 1200, 90], 8, 2, 128, 32, 24), False), (([60000, 50000], 16, 8, 128, 32, 16), False),
    ((2, 8, 2, 3000, 128, 32, 24), True),
    ((1, 8, 4, 250000, 128, 32, 24), True),   # four waves, 24 partials per unit
    ((48, 32, 8, 300, 128, 32, 19), True),    # three waves, phases with as many vote items as row buffers
]


@pytest.mark.parametrize("shape,shared", HAND_OVER)
def test_hand_over_completes_and_every_block_folds_the_same_value(shape, shared):
    m = _model(shape, limit_s=10.0, shared=shared)
    m.run()
    assert not any(m.abort)
    by_unit = {}
    for got in m.got:
        for key, row in got:
            by_unit.setdefault(key, set()).add(row)
    assert set(by_unit) == {x[0] for items in m.per_cta for x in items if x[1] == 1}
    assert all(len(v) == 1 for v in by_unit.values())
    assert [len(g) for g in m.got] == [sum(x[1] for x in items) for items in m.per_cta]


def test_the_shapes_of_the_shared_fold_have_what_they_are_for():
    many = _model(HAND_OVER[5][0], 1.0)
    assert many.waves == 4 and {x[3] for items in many.per_cta for x in items} == {24}
    full = _model(HAND_OVER[6][0], 1.0)
    assert full.waves == 3
    assert max(len(full._items(c, 1, w)) for c in range(19) for w in range(3)) == ROW_BUFFERS


def test_more_vote_items_in_a_phase_than_row_buffers_must_not_share_the_fold():
    # the publisher waits for a free row while the softmax warps wait for it to publish the next wave:
    # a cycle, which ends in time-outs.  With one warp that folds the same shape goes through.
    shape = (48, 32, 8, 300, 128, 32, 8)
    alone = _model(shape, limit_s=10.0)
    assert max(len(alone._items(c, 1, w)) for c in range(8) for w in range(alone.waves)) > ROW_BUFFERS
    alone.run(jitter=False)
    assert not any(alone.abort)
    shared = _model(shape, limit_s=0.5, shared=True)
    shared.run(jitter=False)
    assert any(shared.abort)


@pytest.mark.parametrize("shape,shared", HAND_OVER[::2])
def test_a_block_that_never_arrives_becomes_time_outs_not_a_hang(shape, shared):
    m = _model(shape, limit_s=0.4 if not shared else 2.0, shared=shared)
    took = m.run(absent={5})
    # blocks that need a unit which block 5 has a share of give up at half the limit with the code of
    # that wait; nobody waits longer than the limit
    units_of_5 = {x[0] for x in m.per_cta[5] if x[1] == 0}
    waiting = [c for c, items in enumerate(m.per_cta)
               if c != 5 and any(x[1] == 1 and x[0] in units_of_5 for x in items)]
    assert waiting and all(m.abort[c] == 7 for c in waiting)
    assert took < 5.0


def test_which_calls_share_the_fold():
    # one unit or many, where a unit has many partials; not where it has few, where a warpgroup's half of the
    # columns is not whole heads, or in a part of a call on host buffers that is one KV head, however many units
    # that has
    for shape in ((1, 4, 1, 8192, 128, 32), (1, 32, 8, 13013, 128, 32), (1, 32, 8, 131072, 128, 64)):
        assert sk.shared_fold(*shape)
    for shape in ((4, 32, 8, 5316, 128, 32), (1, 32, 32, 380000, 128, 32)):
        assert not sk.shared_fold(*shape)
    for part in ((1, 4, 1, 8192, 128, 32), (1, 4, 1, 8192, 128, 64), (1, 8, 2, 8192, 128, 32)):
        assert sk.shared_fold(*part) and sk.shared_fold(*part, host_part=True) == (part[2] > 1)


def test_wait_limit_setter_returns_the_previous_value_and_has_a_floor():
    prev = sk.snapkv_set_wait_limit_ns(5)            # raised to one millisecond
    try:
        assert sk.snapkv_set_wait_limit_ns(20_000_000) == 1_000_000
        assert sk.snapkv_set_wait_limit_ns(30_000_000) == 20_000_000
    finally:
        sk.snapkv_set_wait_limit_ns(prev)
    assert prev == 1_000_000_000

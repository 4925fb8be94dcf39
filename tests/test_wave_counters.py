"""Host-side check of the counters behind a wave's large transfers
(sg_kernels.cuh, next_wave): in every order in which two warps of a block can
run between the barriers, each reads for every wave the number that was added
in it.  One counter for all waves does not give that."""
import functools


def _warp(adds, counters, clears):
    """One warp's steps: adds of wave w, the barrier, its read of the count
    and (the clearing warp) the clear, wave after wave."""
    steps = []
    for w, n in enumerate(adds):
        steps += [("add", w % counters, n), ("barrier",), ("read", w % counters)]
        if clears and counters == 3:
            steps.append(("clear", (w + 2) % 3))
    return tuple(steps)


def _reads(warps, counters):
    """All sequences of counts that the warps read, over every interleaving."""
    @functools.lru_cache(None)
    def go(pc, count):
        out = set()
        if all(p == len(s) for p, s in zip(pc, warps)):
            return frozenset({()})
        at = [s[p] if p < len(s) else None for p, s in zip(pc, warps)]
        if all(a == ("barrier",) for a in at):
            return go(tuple(p + 1 for p in pc), count)
        for i, a in enumerate(at):
            if a is None or a == ("barrier",):
                continue
            c, head = list(count), ()
            if a[0] == "add":
                c[a[1]] += a[2]
            elif a[0] == "clear":
                c[a[1]] = 0
            else:
                head = ((i, c[a[1]]),)
            nxt = tuple(p + (j == i) for j, p in enumerate(pc))
            out |= {head + t for t in go(nxt, tuple(c))}
        return frozenset(out)
    return go((0,) * len(warps), (0,) * counters)


def _per_warp(seq, i):
    return tuple(n for j, n in seq if j == i)


def test_every_warp_reads_its_wave_s_count():
    for adds in ((0, 1, 0, 2, 0, 0, 3), (2, 0, 0, 1), (0, 0, 1, 1)):
        warps = (_warp(adds, 3, True), _warp((0,) * len(adds), 3, False))
        for seq in _reads(warps, 3):
            assert _per_warp(seq, 0) == adds and _per_warp(seq, 1) == adds


def test_one_counter_is_read_too_late():
    # a wave without large transfers, then one with: the second warp may see
    # the next wave's addition already and leave the block's common path
    warps = (_warp((0, 1), 1, True), _warp((0, 0), 1, False))
    assert any(_per_warp(seq, 1) != _per_warp(seq, 0) for seq in _reads(warps, 1))

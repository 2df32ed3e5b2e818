"""The x-panel kernel's stage buffers when a wait runs out, as a model on the CPU.

A stage buffer has a full mbarrier (one arrival, with the bytes of the copies)
and an empty one (an arrival per consumer warp).  Waits name a phase by its
parity only, so they are right as long as every stage that is issued is one
phase and nobody gets more than a phase ahead.  The model walks all orders of
events of a small CTA (2 buffers, 2 consumers, 5 stages; any wait may run out
at any time) under the kernel's rules: the first wait that runs out ends the
copy warp's or the consumer's loop, nothing is read or released after it, and
the CTA leaves after waiting for the last phase of every buffer that was issued
into.  Under the former rules (after a wait that ran out, or a stage that is
never issued, go on with the next stage) the same walk finds what they did.
"""
import pytest

B, C, S = 2, 2, 5     # buffers, consumers, stages


def walk(stop, skip=None):
    """Faults met in any order of events.  `stop`: a wait that ran out (or
    the skipped stage) ends its loop; else the loop goes on."""
    # a buffer: phases ended, arrival still due, copies in flight, stage described, empty phases, releases due,
    # stages issued; a copy warp: (next stage, 0 wait / 1 issue / 2 done); a consumer: (stage, 0 wait / 1 read / 2 done)
    buf0 = (0, 1, 0, None, 0, C, 0)
    start = ((buf0,) * B, tuple((b, 0) for b in range(B)), ((0, 0),) * C)
    seen, todo, faults, ended = {start}, [start], set(), 0

    def put(bufs, b, **kw):
        names = ("full", "due", "air", "desc", "empty", "rel", "issued")
        d = dict(zip(names, bufs[b]), **kw)
        if d["due"] == 0 and d["air"] == 0:       # arrival in, bytes landed: the phase ends
            d["full"], d["due"] = d["full"] + 1, 1
        if d["rel"] == 0:
            d["empty"], d["rel"] = d["empty"] + 1, C
        return bufs[:b] + (tuple(d[n] for n in names),) + bufs[b + 1:]

    while todo:
        bufs, copies, cons = state = todo.pop()
        nxt = []
        for b in range(B):
            if bufs[b][2]:                        # copies land
                nxt.append((put(bufs, b, air=bufs[b][2] - 1), copies, cons))
        for b, (s, at) in enumerate(copies):
            def to(ns, nat, nb=bufs):
                done = ns >= S or nat == 2
                nxt.append((nb, copies[:b] + ((ns, 2 if done else nat),) + copies[b + 1:], cons))
            full, due, air, desc, empty, rel, issued = bufs[b]
            if at == 2:
                continue
            if s == skip or (stop and skip is not None and s >= skip):
                to(s + B, 2 if stop else 0)
            elif at == 0:
                if s < B or empty % 2 != (s // B - 1) % 2:
                    to(s, 1)
                if s >= B:
                    to(s, 2 if stop else 1)       # the wait runs out
            else:
                if due == 0:
                    faults.add("second arrival in a phase")
                    continue
                if any(a == 1 and q % B == b for q, a in cons):
                    faults.add("buffer filled while it is read")
                to(s + B, 0, put(bufs, b, due=0, air=1, desc=s, issued=issued + 1))
        for i, (s, at) in enumerate(cons):
            def go(ns, nat, nb=bufs):
                done = ns >= S or nat == 2
                nxt.append((nb, copies, cons[:i] + ((ns, 2 if done else nat),) + cons[i + 1:]))
            if at == 2:
                continue
            b = s % B
            if at == 0:
                if bufs[b][0] % 2 != (s // B) % 2:
                    if bufs[b][3] != s:
                        faults.add("descriptor read before it was written")
                        continue
                    go(s, 1)
                if stop:
                    go(s, 2)
                else:                             # the wait runs out: released unread
                    go(s + 1, 0, put(bufs, b, rel=bufs[b][5] - 1))
            else:
                go(s + 1, 0, put(bufs, b, rel=bufs[b][5] - 1))
        if all(a == 2 for _, a in copies) and all(a == 2 for _, a in cons):
            ended += 1
            if stop:
                # the CTA leaves once the last phase that was issued has ended
                for full, due, air, desc, empty, rel, issued in bufs:
                    if issued and full % 2 != (issued - 1) % 2 and air:
                        faults.add("left with copies in flight")
        for t in nxt:
            if t not in seen:
                seen.add(t)
                todo.append(t)
    assert ended
    return faults


@pytest.mark.parametrize("skip", [None, 0, 1, 2, 3, 4])
def test_first_wait_that_runs_out_ends_the_cta(skip):
    assert walk(True, skip) == set()


def test_going_on_after_a_wait_reads_unwritten_descriptors_and_arrives_twice():
    got = walk(False)
    assert "descriptor read before it was written" in got and "second arrival in a phase" in got
    assert "descriptor read before it was written" in walk(False, 1)


@pytest.mark.parametrize("lanes", [1, 2, 3])
def test_lanes_of_a_warp_leave_a_wait_together(lanes):
    """The lanes of a consumer warp wait one by one; any of them may ask to
    give up at any time, and the phase may end at any time.  Whatever the
    order, no lane gets another answer than the others, and once the phase has
    ended or all have asked every lane gets one."""
    full = (1 << lanes) - 1
    # a lane: (step, mask read): 0 poll, 1 poll after asking, 2 read the mask (phase seen running), 3 the same (seen
    # ended), 4 compare and swap, then its answer
    start = (False, 0, ((0, 0),) * lanes)
    seen, todo = {start}, [start]
    while todo:
        ended, ask, ls = todo.pop()
        nxt = [] if ended else [(True, ask, ls)]
        for i, (at, m) in enumerate(ls):
            def to(step, mask=0, a=ask):
                nxt.append((ended, a, ls[:i] + ((step, mask),) + ls[i + 1:]))
            bit = 1 << i
            if at == 0:
                if ended:
                    to("went on")
                else:
                    to(0)
                    to(1, 0, ask | bit)
            elif at == 1:
                to(3 if ended else 2)
            elif at == 2:
                to("gave up" if ask == full else 1)
            elif at == 3:
                to(*(("gave up",) if ask == full else (4, ask)))
            elif at == 4:
                if ask == m:
                    to("went on", 0, ask & ~bit)
                else:
                    to(*(("gave up",) if ask == full else (4, ask)))
        answers = {at for at, _ in ls if isinstance(at, str)}
        assert len(answers) <= 1, ls
        if ended or ask == full:
            assert all(isinstance(at, str) for at, _ in ls) or any(t != (ended, ask, ls) for t in nxt)
        for t in nxt:
            if t not in seen:
                seen.add(t)
                todo.append(t)

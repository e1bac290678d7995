"""The stage ring of the persistent streamed-update kernel (csrc/gemm.cuh, UTMA && PERSIST) as a state machine.

Three roles share a ring of S stages: a producer that fills them in order (a tile's operand blocks, then its update
chunks), an MMA issuer and an epilogue.  They meet on mbarriers, and a parity wait only says "a phase of this parity was
the last to complete".  Every order in which loads, MMAs and roles can advance is walked: no waiter may pass before the
fill it waits for has landed, and no state may be stuck.  Which role waits on which barrier is read out of the kernel's
source, so the walk is that of the code as it stands."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_06629_b200", "csrc", "gemm.cuh")


def roles_of_the_source():
    text = open(SRC).read()
    text = text[text.index("gemm_tcgen05_kernel(const"):text.index("gemm_split_finish_kernel(const")]
    producer, rest = text.split("---- MMA issuer", 1)
    issuer, epilogue = rest.split("---- epilogue", 1)
    fills = re.findall(r"const uint32_t fb = (\w+)0 \+ 8u \* s;", producer)
    seen = re.findall(r"mbar_wait_addr\((\w+)0 \+ 8u \* s\b", issuer)
    chunk = re.findall(r"mbar_wait_addr\((\w+)0 \+ 8u \* us\b", epilogue)
    assert len(fills) == 2 and len(chunk) == 1 and seen, (fills, seen, chunk)
    return dict(op=fills[0], chunk=fills[1], issuer_sees_chunks=len(seen) > 1, epilogue=chunk[0])


ONE_BARRIER = dict(op="full", chunk="full", issuer_sees_chunks=True, epilogue="full")


def walk(protocol, S, num_kb, chunks, tiles, limit=400000):
    """All reachable states.  Returns None, or a description of the first fault."""
    n_fill = tiles * (num_kb + chunks)
    is_chunk = [i % (num_kb + chunks) >= num_kb for i in range(n_fill)]
    shared = protocol["op"] == protocol["chunk"]
    assert protocol["epilogue"] == protocol["chunk"], "the epilogue waits on the barrier that chunk fills complete"

    def turns(i):          # fills of fill i's barrier that came before it on that stage
        return sum(1 for j in range(i % S, i, S) if shared or is_chunk[j] == is_chunk[i])

    order = [turns(i) for i in range(n_fill)]
    # programs: a list of (wait condition, action) per role; fills are named by their number
    issuer, epi = [], []
    for t in range(tiles):
        first = t * (num_kb + chunks)
        issuer.append(("acce", t))
        issuer += [("fill", i, "mma") for i in range(first, first + num_kb)]
        issuer.append(("commit", t))
        if protocol["issuer_sees_chunks"]:
            issuer += [("fill", i, None) for i in range(first + num_kb, first + num_kb + chunks)]
        epi.append(("accf", t))
        for c in range(chunks):
            i = first + num_kb + c
            epi.append(("fill", i, "use"))
            if c > 0:
                epi.append(("release", i - 1))
            if c == chunks - 1:
                epi.append(("drained", t))
                epi.append(("release", i))

    # state: producer position, landed fills, released fills, issuer position, epilogue position, accf / acce counts
    start = (0, frozenset(), frozenset(), 0, 0, 0, 0)
    todo, known = [start], {start}
    while todo:
        prod, landed, released, ip, ep, accf, acce = todo.pop()
        nxt = []

        def passes(i):     # does a parity wait for fill i's phase return now?
            done = sum(1 for j in landed if j % S == i % S and (shared or is_chunk[j] == is_chunk[i]))
            return (done & 1) != (order[i] & 1)

        if prod < n_fill and (prod < S or (prod - S) in released):
            nxt.append((prod + 1, landed, released, ip, ep, accf, acce))
        for i in range(prod):                                     # a load in flight lands
            if i not in landed:
                nxt.append((prod, landed | {i}, released, ip, ep, accf, acce))
        if ip < len(issuer):
            op = issuer[ip]
            if op[0] == "acce" and acce >= op[1] - 1:             # (two accumulators)
                nxt.append((prod, landed, released, ip + 1, ep, accf, acce))
            elif op[0] == "commit":
                nxt.append((prod, landed, released, ip + 1, ep, accf + 1, acce))
            elif op[0] == "fill" and passes(op[1]):
                if op[1] not in landed:
                    return "the issuer passed fill %d before it landed" % op[1]
                nxt.append((prod, landed, released | {op[1]} if op[2] else released, ip + 1, ep, accf, acce))
        if ep < len(epi):
            op = epi[ep]
            if op[0] == "accf" and accf > op[1]:
                nxt.append((prod, landed, released, ip, ep + 1, accf, acce))
            elif op[0] == "drained":
                nxt.append((prod, landed, released, ip, ep + 1, accf, acce + 1))
            elif op[0] == "release":
                nxt.append((prod, landed, released | {op[1]}, ip, ep + 1, accf, acce))
            elif op[0] == "fill" and passes(op[1]):
                if op[1] not in landed:
                    return "the epilogue passed fill %d before it landed" % op[1]
                nxt.append((prod, landed, released, ip, ep + 1, accf, acce))
        if not nxt and (ip < len(issuer) or ep < len(epi) or prod < n_fill):
            return "stuck: producer at fill %d, issuer at %s, epilogue at %s" % (prod, issuer[ip:ip + 1], epi[ep:ep + 1])
        for s in nxt:
            if s not in known:
                known.add(s)
                todo.append(s)
        assert len(known) < limit
    return None


# ring depths the launch picks or can be told to take, one and several operand blocks a tile, four chunks of a
# 128-column tile and eight of a 256-column one
@pytest.mark.parametrize("S, num_kb, chunks, tiles", [(3, 1, 4, 4), (2, 1, 4, 4), (3, 2, 4, 3), (4, 1, 8, 2), (3, 5, 4, 2), (4, 3, 4, 3)])
def test_every_order_of_events_completes(S, num_kb, chunks, tiles):
    assert walk(roles_of_the_source(), S, num_kb, chunks, tiles) is None


def test_the_walk_finds_the_late_issuer_of_a_shared_barrier():
    """One barrier per stage for both kinds of fill, as the kernel once had it: an issuer that is late by one phase
    waits for ever."""
    assert "stuck" in walk(ONE_BARRIER, 3, 1, 4, 4)

"""The named barriers of the bf16 one-launch sampler (k_sample.cu) when a wait on the
other CTAs gives up.  The roles of a CTA -- compute warps, and a control and an I/O warp
for each request group -- are walked through every interleaving of a small model, with
each control warp giving up at any step or not at all: every role has to reach its end.
Runs on the CPU; the source is read for the barrier calls that the model makes."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2609_37029_gb300", "csrc", "k_sample.cu")
WARPS = 2                                   # compute warps of the model (16 in the kernel)


def role_sources():
    txt = open(SRC).read()
    body = txt[txt.index("sample_persistent_kernel("):txt.index("persistent kernel, fp32 storage")]
    parts = re.split(r"// =+ (?=compute warps|I/O warp|control warp)", body)[1:]
    assert [p.split()[0] for p in parts] == ["compute", "I/O", "control"]
    return [re.sub(r"//[^\n]*", "", p[p.index("for (int s = 0"):]) for p in parts]


def test_every_role_passes_the_same_barriers_in_every_step():
    compute, io, control = role_sources()
    calls = [re.findall(r"named_(bar|arrive)\((\d) \+ (?:h|grp)", t) for t in (compute, io, control)]
    assert calls[0] == [("bar", "3"), ("arrive", "1"), ("arrive", "5")]
    assert calls[1] == [("bar", "5")]
    # the second arrival is the one of a control warp that has given up
    assert calls[2] == [("bar", "1"), ("arrive", "3"), ("arrive", "3")]
    for t in (compute, io):                 # one return, behind the loop over the steps
        assert len(re.findall(r"\breturn;", t)) == 1 and re.search(r"\n    }\s*return;\s*}\s*(if|$)", t)
    assert not re.search(r"\breturn;", control)


def compute(w, groups, steps, flag_rule):
    """Operations of a compute warp; 'flag' is the former rule: read a shared flag, leave if it is set."""
    ops = []
    for s in range(steps):
        for h in range(groups):
            if s > 0:
                ops.append(("sync", ("key", h)))
                if flag_rule:
                    ops.append(("flag", None))
            ops += [("rows", (h, s)), ("arrive", ("red", h)), ("arrive", ("io", h))]
    return ops


def control(h, steps):
    ops = []
    for s in range(steps):
        ops += [("sync", ("red", h)), ("exchange", s)]
        if s + 1 < steps:
            ops.append(("arrive", ("key", h)))
    return ops


def io(h, steps):
    ops = []
    for s in range(steps):
        ops.append(("sync", ("io", h)))
        if s + 1 < steps:
            ops.append(("load", h))
    return ops


def stuck_state(groups, steps, flag_rule):
    """A reachable state in which a role waits and nothing can move, or None."""
    progs = [compute(w, groups, steps, flag_rule) for w in range(WARPS)]
    progs += [control(h, steps) for h in range(groups)] + [io(h, steps) for h in range(groups)]
    ctl0, bars = WARPS, [(k, h) for k in ("red", "io", "key") for h in range(groups)]
    bid = {b: i for i, b in enumerate(bars)}
    # pc of each role, (arrivals, bit set of waiting roles) of each barrier, rows loaded, given up, flag
    start = (tuple(0 for _ in progs), tuple((0, 0) for _ in bars), tuple(1 for _ in range(groups)),
             tuple(False for _ in range(groups)), False)
    seen, todo = {start}, [start]
    while todo:
        pcs, bar, rows, gone, flag = todo.pop()
        nxt = []

        def put(r, pc=None, **k):
            p = list(k.get("pcs", pcs))
            p[r] = p[r] + 1 if pc is None else pc
            nxt.append((tuple(p), k.get("bar", bar), k.get("rows", rows), k.get("gone", gone), k.get("flag", flag)))

        def arrive(r, b, wait):
            n, who = bar[b]
            n, who, p, nb = n + 1, who | (1 << r if wait else 0), list(pcs), list(bar)
            if n == WARPS + 1:              # complete: the waiting roles go on
                p = [pc + (who >> i & 1) for i, pc in enumerate(p)]
                n = who = 0
            nb[b] = (n, who)
            put(r, pc=p[r] + (0 if wait else 1), pcs=tuple(p), bar=tuple(nb))

        for r, prog in enumerate(progs):
            if pcs[r] >= len(prog) or any(who >> r & 1 for _, who in bar):
                continue
            op, x = prog[pcs[r]]
            h = r - ctl0
            if op == "sync" or op == "arrive":
                arrive(r, bid[x], op == "sync")
            elif op == "rows":
                if rows[x[0]] > x[1]:
                    put(r)
            elif op == "load":
                put(r, rows=tuple(n + (g == x) for g, n in enumerate(rows)))
            elif op == "exchange":
                put(r)
                if not gone[h]:
                    g2 = tuple(v or i == h for i, v in enumerate(gone))
                    # the former rule: set the flag, release the compute warps and leave
                    if flag_rule:
                        put(r, gone=g2, flag=True)
                    else:
                        put(r, gone=g2)
            elif op == "flag":
                if flag:                    # leave, releasing the control and I/O warps
                    nb, p = list(bar), list(pcs)
                    for k in ("red", "io"):
                        for g in range(groups):
                            n, who = nb[bid[(k, g)]]
                            n += 1
                            if n == WARPS + 1:
                                p = [pc + (who >> i & 1) for i, pc in enumerate(p)]
                                n = who = 0
                            nb[bid[(k, g)]] = (n, who)
                    put(r, pc=len(prog), pcs=tuple(p), bar=tuple(nb))
                else:
                    put(r)
        if not nxt and any(pcs[r] < len(progs[r]) for r in range(WARPS)):
            return pcs, bar, gone
        for st in nxt:
            if st not in seen:
                seen.add(st)
                todo.append(st)
    return None


@pytest.mark.parametrize("groups,steps", [(1, 4), (2, 3)])
def test_no_warp_is_left_at_a_barrier(groups, steps):
    assert stuck_state(groups, steps, flag_rule=False) is None


def test_the_model_finds_warps_that_leave_on_a_flag_of_their_own():
    """Two groups whose compute warps each read one flag that either control warp may set at
    any time: one warp leaves, another goes on to a barrier that is never complete."""
    assert stuck_state(2, 3, flag_rule=True) is not None
    assert stuck_state(1, 4, flag_rule=True) is None

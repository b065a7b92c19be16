"""The hand-offs between the warp roles of the tensor-core kernels as a model on the CPU.

An mbarrier wait names a phase by its parity only.  A waiter that comes so late that the next phase has completed as well
sees the parity of the phase after that, and if this one needs the waiter's own work it waits until its budget runs out.  So
no phase may complete while some role has not yet passed its wait for the phase before.

The roles are written down as their sequences of waits and arrivals.  The system has no choices in it (a role only ever waits
for one thing), so letting every other role run as far as it can shows the most that can happen while one is held up."""
import pytest


def overruns(roles, counts):
    """roles: name -> list of ("wait", barrier, phase) and ("arrive", barrier); counts: arrivals that complete a phase.
    Returns the waits (role, barrier, phase) whose following phase can complete before they are passed; the whole must end."""

    def run(held=None, stop=None):
        at = {r: 0 for r in roles}
        arrived = {b: 0 for b in counts}
        moved = True
        while moved:
            moved = False
            for r, ops in roles.items():
                while at[r] < len(ops) and not (r == held and at[r] == stop):
                    op = ops[at[r]]
                    if op[0] == "arrive":
                        arrived[op[1]] += 1
                    elif arrived[op[1]] // counts[op[1]] <= op[2]:
                        break
                    at[r] += 1
                    moved = True
        return at, {b: n // counts[b] for b, n in arrived.items()}

    at, _ = run()
    assert all(at[r] == len(ops) for r, ops in roles.items()), "the protocol does not end"
    found = []
    for r, ops in roles.items():
        for i, op in enumerate(ops):
            if op[0] == "wait" and run(r, i)[1][op[1]] > op[2] + 1:
                found.append((r, op[1], op[2]))
    return found


STAGES = 3


def state_kernel(pieces, fc_buffers, full_barriers, stages=STAGES):
    """tc_state_kernel: loads in `stages` stages, two groups of workers that take turns (one warp of each here), products.
    full_barriers: how many barriers the loads' arrivals go round; with one per stage a group must follow every phase."""
    full = lambda p: "full%d" % (p % full_barriers)
    n = stages
    producer, mma = [], []
    groups = {0: [], 1: []}
    for p in range(pieces):
        if p >= n:
            producer.append(("wait", "free%d" % (p % n), p // n - 1))
        producer.append(("arrive", full(p)))
        mma += [("wait", full(p), p // full_barriers), ("wait", "fc_ready%d" % (p % fc_buffers), p // fc_buffers),
                ("arrive", "free%d" % (p % n)), ("arrive", "fc_free%d" % (p % fc_buffers))]
        for g, ops in groups.items():
            own = p % 2 == g
            if own or full_barriers == n:
                ops.append(("wait", full(p), p // full_barriers))
            if own:
                if p >= fc_buffers:
                    ops.append(("wait", "fc_free%d" % (p % fc_buffers), p // fc_buffers - 1))
                ops.append(("arrive", "fc_ready%d" % (p % fc_buffers)))
    roles = {"producer": producer, "mma": mma, "even": groups[0], "odd": groups[1]}
    return roles, {op[1]: 1 for ops in roles.values() for op in ops}


@pytest.mark.parametrize("fc_buffers", [2, 4])
@pytest.mark.parametrize("pieces", [1, 2, 3, 7, 13, 30])
def test_state_kernel_phases_are_never_overrun(pieces, fc_buffers):
    assert overruns(*state_kernel(pieces, fc_buffers, 2 * STAGES)) == []


@pytest.mark.parametrize("pieces", [1, 5, 6, 7, 13, 30])
def test_state_kernel_of_64_features_phases_are_never_overrun(pieces):
    # (an even number of stages: all pieces of a stage are the same group's, so that a barrier a stage is enough)
    roles, counts = state_kernel(pieces, 4, 6, 6)
    for g, parity in (("even", 0), ("odd", 1)):
        roles[g] = [op for op in roles[g] if op[1][:4] != "full" or int(op[1][4:]) % 2 == parity]
    assert overruns(roles, counts) == []


@pytest.mark.parametrize("fc_buffers", [2, 4])
def test_state_kernel_with_one_barrier_a_stage_would_be_overrun(fc_buffers):
    # (the group that does not own a piece is held back by nothing)
    found = overruns(*state_kernel(7, fc_buffers, STAGES))
    assert ("odd", "full0", 0) in found and ("even", "full1", 0) in found


def walk_kernel(blocks, want_final, ready_barriers):
    """tc_walk_kernel (one warp of workers, one of the output group).  ready_barriers: how many barriers the completions of M3
    and of M4 go round."""
    two, k = lambda name, n: name + str(n % 2), ready_barriers
    dz, o = (lambda n: ("dz%d" % (n % k))), (lambda n: ("o%d" % (n % k)))
    producer = [("arrive", "m1_0"), ("arrive", "m1_0"), ("arrive", "c0")]
    if blocks > 1:
        producer += [("arrive", "m1_1"), ("arrive", "c1")]
    for n in range(blocks - 1):
        producer += [("wait", "m2_done", n), ("arrive", two("m1_", n + 1))]
        if n + 2 < blocks:
            producer += [("wait", dz(n), n // k), ("arrive", two("m1_", n)), ("wait", o(n), n // k), ("arrive", two("c", n))]
    mma = [("wait", "m1_0", 0), ("arrive", "s")]
    workers = [("arrive", "m1_0"), ("arrive", "m2_ok")]
    if blocks > 1 or want_final:
        workers.append(("wait", "c0", 0))
    output = [("arrive", "m2_ok")]
    for n in range(blocks):
        more = n + 1 < blocks
        mma += [("wait", "m2_ok", n), ("arrive", "m2_done")]
        if more or want_final:
            mma.append(("wait", "m3_ok", n))
        mma += [("arrive", dz(n)), ("wait", two("c", n), n // 2), ("wait", "m4_ok", n), ("arrive", o(n))]
        if more:
            mma += [("wait", two("m1_", n + 1), (n + 1) // 2), ("arrive", "s")]
        workers += [("wait", "s", n), ("arrive", "m3_ok"), ("arrive", "m4_ok")]
        if more:
            workers.append(("wait", two("c", n + 1), (n + 1) // 2))
        if more or want_final:
            workers.append(("wait", dz(n), n // k))
        if more:
            workers += [("arrive", two("m1_", n + 1)), ("arrive", "m2_ok")]
        output += [("wait", "m2_done", n), ("arrive", "m4_ok"), ("wait", o(n), n // k), ("arrive", "m2_ok")]
    roles = {"producer": producer, "mma": mma, "workers": workers, "output": output}
    counts = {op[1]: 1 for ops in roles.values() for op in ops}
    counts.update({"m1_0": 3, "m1_1": 3, "m2_ok": 2, "m4_ok": 2})
    return roles, counts


@pytest.mark.parametrize("want_final", [False, True])
@pytest.mark.parametrize("blocks", [1, 2, 3, 4, 9])
def test_walk_kernel_phases_are_never_overrun(blocks, want_final):
    assert overruns(*walk_kernel(blocks, want_final, 2)) == []


def test_walk_kernel_with_one_barrier_for_every_block_would_be_overrun():
    # (a producer that is a block late)
    found = overruns(*walk_kernel(6, True, 1))
    assert ("producer", "dz0", 0) in found and ("producer", "o0", 0) in found


def walk64_kernel(blocks, last_m3, ahead, tail=None, final=False):
    """tc_walk64_kernel (one warp of each group, of the state group one with the hi and one with the lo terms).  ahead: the state
    group fetches its value rows a block ahead.  tail: the block, if any, that a packed sequence ends in, whose rows past the end it
    clears and whose results leave row by row.  final: the state is handed out (last_m3)."""
    two, three = (lambda name, n: name + str(n % 2)), (lambda name, n: name + str(n % 3))
    m3 = lambda n: n + 1 < blocks or last_m3
    producer, p, output = [], [], []
    mma = [("wait", "ab0", 0), ("arrive", "s0")]
    state = []
    fc = lambda n: [("wait", three("ab", n), n // 3)] * (n == tail) + [("arrive", "fc")]
    if m3(0):
        mma += [("wait", "fc", 0), ("arrive", "dz")]
        state += [("wait", "c0", 0)] + fc(0)
    if ahead and m3(1) and blocks > 1:
        state.append(("wait", "c1", 0))
    state.append(("arrive", "z"))
    staged = 0
    for n in range(blocks):
        if n >= 3:
            producer.append(("wait", three("free", n), n // 3 - 1))
        producer += [("arrive", three("ab", n)), ("arrive", three("c", n))]
        more = n + 1 < blocks
        if more:
            mma += [("wait", three("ab", n + 1), (n + 1) // 3), ("arrive", two("s", n + 1))]
        mma.append(("wait", "z", n))
        if n > 0:
            mma.append(("wait", "o_free", n - 1))
        mma += [("arrive", "m2"), ("wait", three("c", n), n // 3), ("wait", two("p", n), n // 2), ("arrive", "o"), ("arrive", three("free", n))]
        if more and m3(n + 1):
            mma += [("wait", "fc", n + 1), ("arrive", "dz")]
        p += [("wait", two("s", n), n // 2), ("arrive", two("p", n))]
        if not ahead and more and m3(n + 1):
            state.append(("wait", three("c", n + 1), (n + 1) // 3))
        if more or last_m3:
            state.append(("wait", "dz", n))
        if more:
            if m3(n + 1):
                state += fc(n + 1)
            if ahead and n + 2 < blocks and m3(n + 2):
                state.append(("wait", three("c", n + 2), (n + 2) // 3))
            state += [("wait", "m2", n), ("arrive", "z")]
        output += [("wait", "o", n), ("arrive", "o_free")]
        if n != tail:
            output += [("wait", "stored", staged - 1)] * (staged > 0) + [("arrive", "staged"), ("wait", "staged", staged), ("arrive", "stored")]
            staged += 1
    # the lo terms' state leaves through the place of the state operand, once the last product has read that
    lo = [("wait", "m2", blocks - 1), ("arrive", "final")] if final else []
    hi = [("wait", "final", 0)] if final else []
    roles = {"producer": producer, "mma": mma, "p": p, "state_hi": state + hi, "state_lo": state + lo, "output": output}
    counts = {op[1]: 1 for ops in roles.values() for op in ops}
    counts.update({"fc": 2, "z": 2})
    return roles, counts


@pytest.mark.parametrize("ahead", [False, True])
@pytest.mark.parametrize("last_m3", [False, True])
@pytest.mark.parametrize("blocks", [1, 2, 3, 4, 5, 11])
def test_walk64_kernel_phases_are_never_overrun(blocks, last_m3, ahead):
    assert overruns(*walk64_kernel(blocks, last_m3, ahead)) == []


@pytest.mark.parametrize("ahead", [False, True])
@pytest.mark.parametrize("final", [False, True])
@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("blocks", [1, 2, 3, 4, 5, 11])
def test_walk64_kernel_phases_are_never_overrun_at_the_ends_of_sequences(blocks, reverse, final, ahead):
    """The state that is handed out, and a packed sequence that ends inside a block: the last one of a forward walk, which then has
    an M3 so that the rows past the end are cleared before M4, or the first one of a reverse walk."""
    last_m3 = final or not reverse or blocks == 1
    assert overruns(*walk64_kernel(blocks, last_m3, ahead, tail=0 if reverse else blocks - 1, final=final)) == []
    if final:
        assert overruns(*walk64_kernel(blocks, True, ahead, final=True)) == []

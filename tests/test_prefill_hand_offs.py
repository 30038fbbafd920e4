"""The hand-offs of the tcgen05 prompt encoder (encode_umma_kernel), played through on the CPU in every order.

Its roles (two issuing warps, the converting warps, the tensor pipe) only meet at mbarriers, and a wait by parity tells the
completed phase from the running one and nothing more: a warp that looks two completions late reads "not complete".  The model
below takes the roles' steps from the kernel and the barrier that group 1 starts on from its source, and visits every state
that any scheduling of the roles can reach."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_14468_b200", "csrc", "ha_encode_tc.cu")


def _start_gate() -> str:
    """The barrier in front of group 1's first tile, as the kernel has it."""
    with open(SRC) as f:
        gate = re.search(r"bool ok = g == 0 [^;]*wait\(smem_u32\(&s_(\w+(?:\[\d\])*)\), 0u\);", f.read())
    assert gate, "the start gate of group 1 is not where this test looks for it"
    return gate.group(1)


# Barriers: d{g} a hidden layer is summed, a{g}{half} half of it is converted, o{g} the outputs are summed (the names of the
# kernel's s_dbar, s_abar, s_obar), start: group 0 has converted its first layer.
ARRIVALS = {"d0": 1, "d1": 1, "o0": 1, "o1": 1, "a00": 2, "a10": 2, "a01": 1, "a11": 1, "start": 3}


def _issuer(g, n_tiles, gate):
    ops = [("wait", gate, 0)] if g == 1 and n_tiles else []
    for i in range(n_tiles):
        if i:
            ops.append(("wait", f"o{g}", (i - 1) & 1))
        ops.append(("commit", f"d{g}"))
        for parity, done in ((0, f"d{g}"), (1, f"o{g}")):
            ops += [("wait", f"a{g}0", parity), ("wait", f"a{g}1", parity), ("commit", done)]
    return tuple(ops)


def _converter(role, na, nb):
    """role 0 and 1: the quarters that also write the signatures of group 0 and 1 (first half of the columns); 2: the rest."""
    half, ops = role >> 1, []

    def convert(g, parity):
        ops.extend([("wait", f"d{g}", parity), ("arrive", f"a{g}{half}")])

    for i in range(na + 1):
        a, b = i < na, 0 < i <= nb
        if a:
            convert(0, 0)
            if i == 0:
                ops.append(("arrive", "start"))
        if b:
            convert(1, 1)
        if a:
            convert(0, 1)
        if b and role == 1:
            ops.append(("wait", "o1", (i - 1) & 1))
        if i < nb:
            convert(1, 0)
        if a and role == 0:
            ops.append(("wait", "o0", i & 1))
    return tuple(ops)


def _stuck_state(na, nb, gate):
    """A reachable state in which somebody still has work and nobody can go on, or None."""
    roles = [_issuer(0, na, gate), _issuer(1, nb, gate)] + [_converter(r, na, nb) for r in range(3)]
    names = sorted(ARRIVALS)

    def arrive(bars, name):
        done, pending = bars[names.index(name)]
        pending += 1
        new = (done + 1, 0) if pending == ARRIVALS[name] else (done, pending)
        return tuple(new if n == name else b for n, b in zip(names, bars))

    first = ((0,) * len(roles), ((0, 0),) * len(names), ())     # program counters, (completions, arrivals), tensor pipe
    seen, todo = {first}, [first]
    while todo:
        pcs, bars, pipe = state = todo.pop()
        after = []
        if pipe:                                                # the tensor pipe completes its commits in order
            after.append((pcs, arrive(bars, pipe[0]), pipe[1:]))
        for r, ops in enumerate(roles):
            if pcs[r] == len(ops):
                continue
            op, new_bars, new_pipe = ops[pcs[r]], bars, pipe
            if op[0] == "wait":
                if (bars[names.index(op[1])][0] & 1) == op[2]:   # the phase of that parity is not the completed one
                    continue
            elif op[0] == "commit":
                new_pipe = pipe + (op[1],)
            else:
                new_bars = arrive(bars, op[1])
            after.append((tuple(p + (i == r) for i, p in enumerate(pcs)), new_bars, new_pipe))
        if not after and any(pcs[r] < len(ops) for r, ops in enumerate(roles)):
            return state
        for s in after:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


TILES = [(1, 0), (1, 1), (2, 1), (2, 2), (3, 2), (3, 3)]        # group 0 has as many tiles as group 1 or one more


@pytest.mark.parametrize("na,nb", TILES)
def test_no_order_of_the_roles_leaves_a_wait_without_its_phase(na, nb):
    gate = {"abar[0][1]": "a01"}.get(_start_gate(), _start_gate())
    assert _stuck_state(na, nb, gate) is None


@pytest.mark.parametrize("na,nb", [(1, 1), (3, 3)])
def test_the_model_sees_a_gate_that_can_be_missed(na, nb):
    """A barrier that goes on to its next phase without group 1 is no gate: it is passed or missed by chance."""
    assert _stuck_state(na, nb, "a01") is not None

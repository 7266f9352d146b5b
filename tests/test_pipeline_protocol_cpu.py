"""Host model of the split-BF16 contraction's slot protocol (no device).

Producer teams take chunks i = t, t + T, t + 2T, ... (T teams); chunk i goes to A/B slot
s = i mod S (S slots).  Before writing a slot, a team waits for the MMAs of the slot's previous
use (chunk i - S) through a parity wait on the slot's barrier: the wait passes when the number c
of completed phases has the parity of u = i // S, so it is unambiguous only while c is u - 1 or u
when the wait starts.  If c could still be u - 2 (the MMAs of chunk i - 2S not complete), the
parity would match too early and the team would overwrite a slot the tensor core still reads.
The issuer consumes chunks in order and their MMAs complete in order.

The model explores random interleavings of the teams, the issuer and the MMA completions and
checks that every wait starts with c in {u - 1, u} when T <= S (the rule the kernel enforces by
capping its teams at its slots), and finds a schedule that breaks it when T > S.

A second model covers the drains.  The accumulators are handed over once per window of W chunks: the
issuer's MMAs complete phase w of `acc_ready` at the window's last chunk, the team of that chunk reads
the sums and completes phase w of `acc_free`, and the issuer starts window w + 1 only then.  Each warp
of a team runs by itself between its arrival on `produced` and its drain.
"""
import ctypes
import os
import random
import re

import numpy as np
import pytest

import fieldgen
import paper_1904_11055_gb300 as ps
from paper_1904_11055_gb300 import build as psbuild


def run(T, S, nch, rng):
    """One random schedule; returns the first aliasing wait (chunk, completed phases, use) or None."""
    team_next = list(range(T))               # next chunk of each team
    team_state = ["wait"] * T                # "wait": about to wait on the slot; "write": writing it
    produced = [False] * nch
    completed = [0] * S                      # completed phases of each slot's barrier
    issued = 0                               # chunks whose MMAs the issuer has started
    done = 0                                 # chunks whose MMAs have completed (in order)
    while done < nch:
        moves = []
        for t in range(T):
            i = team_next[t]
            if i >= nch:
                continue
            u = i // S
            if team_state[t] == "wait":
                if u == 0 or completed[i % S] % 2 == u % 2:  # the parity wait passes
                    moves.append(("pass", t))
            else:
                moves.append(("produce", t))
        if issued < nch and produced[issued]:
            moves.append(("issue", None))
        if done < issued:
            moves.append(("complete", None))
        assert moves, "no move: the protocol stalls"
        kind, t = rng.choice(moves)
        if kind == "pass":
            i = team_next[t]
            u, c = i // S, completed[i % S]
            if u > 0 and c != u:                 # passed without the MMAs of chunk i - S complete
                return i, c, u
            team_state[t] = "write"
        elif kind == "produce":
            produced[team_next[t]] = True
            team_next[t] += T
            team_state[t] = "wait"
        elif kind == "issue":
            issued += 1
        else:
            completed[done % S] += 1
            done += 1
    return None


@pytest.mark.parametrize("T,S", [(2, 2), (2, 3), (2, 4), (3, 3), (3, 4)])
def test_teams_up_to_the_slot_count_never_alias(T, S):
    rng = random.Random(1000 * T + S)
    for _ in range(400):
        assert run(T, S, 48, rng) is None


@pytest.mark.parametrize("T,S", [(3, 2), (4, 3)])
def test_more_teams_than_slots_can_alias(T, S):
    rng = random.Random(7 * T + S)
    assert any(run(T, S, 48, rng) is not None for _ in range(400))


def run_drains(T, S, W, nch, early, rng, warps=2):
    """One random schedule of the drains.  early: a warp waits for the window before its own arrival on `produced`
    for a window's last chunk, else after it.  Returns None, or what went wrong: "stall" (no warp can move) or
    the drain that read a window's sums before (or after) their time."""
    nt = min(T, S)
    last = lambda i: i == nch - 1 or i % W == W - 1
    prog = []  # per warp: its steps in program order
    for t in range(nt):
        steps = []
        for i in range(t, nch, nt):
            w = i // W
            before = [("ready", w - 1)] if last(i) and w > 0 else []
            steps += [("slot", i)] + (before if early else []) + [("arrive", i)]
            if last(i):
                steps += ([] if early else before) + [("ready", w), ("drain", w)]
        prog += [list(steps) for _ in range(warps)]
    pc = [0] * len(prog)
    arrived = [0] * nch
    slot_phases, ready, free, free_arrivals = [0] * S, 0, 0, 0
    issued = done = 0
    while True:
        moves = []
        for k, steps in enumerate(prog):
            if pc[k] == len(steps):
                continue
            op, v = steps[pc[k]]
            if op == "slot" and v >= S and slot_phases[v % S] % 2 != (v // S) % 2:
                continue  # a parity wait for phase u - 1 passes when the current phase has the parity of u
            if op == "ready" and ready % 2 == v % 2:
                continue
            moves.append(k)
        can_issue = issued < nch and arrived[issued] == warps
        if can_issue and issued % W == 0 and issued > 0 and free % 2 == (issued // W - 1) % 2:
            can_issue = False
        if can_issue:
            moves.append("issue")
        if done < issued:
            moves.append("complete")
        if not moves:
            return None if all(pc[k] == len(s) for k, s in enumerate(prog)) and done == nch else "stall"
        k = rng.choice(moves)
        if k == "issue":
            issued += 1
        elif k == "complete":
            slot_phases[done % S] += 1
            ready += last(done)
            done += 1
        else:
            op, v = prog[k][pc[k]]
            if op == "arrive":
                arrived[v] += 1
            elif op == "drain":
                if ready != v + 1 or free != v:
                    return f"drain of window {v} with {ready} complete and {free} read"
                free_arrivals += 1
                if free_arrivals == warps:
                    free_arrivals, free = 0, free + 1
            pc[k] += 1


def kernel_waits_before_arriving():
    """Whether the contraction's producers wait for the window before ahead of their arrival on `produced`."""
    path = os.path.join(os.path.dirname(__file__), "..", "paper_1904_11055_gb300", "csrc", "contract_tc.cu")
    src = open(path).read()
    body = src[src.index("// ------------------------------------------------------------- producers"):]
    wait = re.search(r"mbar_wait_warp\(acc_ready, \(uint32_t\)\(\(win\.index - 1\) & 1\), s_abort\)", body)
    return wait.start() < body.index("tc::mbar_arrive(&produced[slot]);")


DRAINS = [(2, 2, 5), (2, 3, 5), (2, 4, 4), (3, 3, 3), (3, 3, 7), (3, 4, 5), (3, 4, 4)]


@pytest.mark.parametrize("T,S,W", DRAINS)
def test_drains_neither_stall_nor_read_another_window(T, S, W):
    rng = random.Random(100 * T + 10 * S + W)
    early = kernel_waits_before_arriving()
    for k in range(600):
        assert run_drains(T, S, W, 3 * W + 1 + k % W, early, rng) is None


def test_waiting_after_the_arrival_can_stall():
    """Once every warp has arrived, the window may complete before a warp's wait for the one before starts: that wait
    then asks for a phase whose parity the barrier will not show again."""
    rng = random.Random(5)
    assert "stall" in {run_drains(3, 3, 5, 21, False, rng) for _ in range(600)}


@pytest.mark.parametrize("T,S,W", [(2, 4, 2), (3, 3, 1), (3, 4, 1)])
def test_windows_shorter_than_the_slots_can_go_wrong(T, S, W):
    """The slot's previous chunk may then lie two or more windows back, and the wait for the window before passes early."""
    rng = random.Random(10 * S + W)
    assert any(run_drains(T, S, W, 8 * W + k % W, True, rng) is not None for k in range(2000))


@pytest.mark.parametrize("order,nshell,default", [(3, 12, 128), (4, 10, 14), (2, 12, 128)])
@pytest.mark.parametrize("env,window", [(None, None), ("1", 4), ("2", 4), ("3", 4), ("4", 4), ("5", 5), ("0", None)])
def test_window_holds_at_least_as_many_chunks_as_slots(monkeypatch, order, nshell, default, env, window):
    psbuild.build()
    fn = ps.load_library().poly_diag_tc_window
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_uint, ctypes.c_int, ctypes.c_void_p]
    monkeypatch.delenv("POLY_TC_WINDOW", raising=False)
    if env is not None:
        monkeypatch.setenv("POLY_TC_WINDOW", env)
    e, got = fieldgen.unit_edges(nshell), np.zeros(1, np.int32)
    assert fn(64, order, e.ctypes.data, nshell, 0, 0, got.ctypes.data) == 0
    assert got[0] == (window or default)

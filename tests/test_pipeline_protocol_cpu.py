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

A second model covers the drains.  The accumulators are handed over once per window of chunks: the
issuer's MMAs complete phase w of `acc_ready` at the window's last chunk, the team of that chunk waits
for it, reads the sums and completes phase w of `acc_free`, and the issuer starts window w + 1 only then.
Each warp of a team runs by itself between its arrival on `produced` and its drain.  The wait is
unambiguous where the team knows window w - 1 to be over, which the slot of the window's last chunk
tells it when windows hold more chunks than there are slots; the kernel therefore gives the first
window, not the last, the remainder.
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


def run_drains(T, S, ends, rng, wait=None, warps=2):
    """One random schedule of the drains.  ends[i]: the last chunk of chunk i's window.  wait: None (each drain waits
    for its own window alone), or "after" (a wait for the window before too, after the arrival on `produced`).
    Returns None, or what went wrong: "stall" (no warp can move) or the drain that read a window's sums early."""
    nch, nt = len(ends), min(T, S)
    window = [0] * nch
    for i in range(1, nch):
        window[i] = window[i - 1] + (ends[i] != ends[i - 1])
    prog = []  # per warp: its steps in program order
    for t in range(nt):
        steps = []
        for i in range(t, nch, nt):
            w = window[i]
            steps += [("slot", i), ("arrive", i)]
            if i == ends[i]:
                steps += [("ready", w - 1)] if wait == "after" and w > 0 else []
                steps += [("ready", w), ("drain", w)]
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
        if can_issue and issued and ends[issued] != ends[issued - 1] and free % 2 == (window[issued] - 1) % 2:
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
            ready += done == ends[done]
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


def last_window_short(nch, W):
    return [min(nch - 1, i // W * W + W - 1) for i in range(nch)]


def kernel_windows(monkeypatch, order, nshell, nch, env):
    """The window of a plan, and the last chunk of each chunk's window, from the library."""
    psbuild.build()
    fn = ps.load_library().poly_diag_tc_window
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_uint] + [ctypes.c_int] * 2 + \
        [ctypes.c_void_p] * 2
    monkeypatch.delenv("POLY_TC_WINDOW", raising=False)
    if env is not None:
        monkeypatch.setenv("POLY_TC_WINDOW", env)
    e, got, ends = fieldgen.unit_edges(nshell), np.zeros(1, np.int32), np.zeros(nch, np.int32)
    assert fn(64, order, e.ctypes.data, nshell, 0, 0, nch, got.ctypes.data, ends.ctypes.data) == 0
    return int(got[0]), ends.tolist()


@pytest.mark.parametrize("T,S", [(2, 2), (2, 3), (2, 4), (3, 3), (3, 4)])
@pytest.mark.parametrize("env", ["1", "2", "3", "4", "5", "6", "7"])
def test_drains_neither_stall_nor_read_another_window(monkeypatch, T, S, env):
    rng = random.Random(100 * T + 10 * S + int(env))
    for nch in (1, 2, 3, 4, 5, 6, 13, 16, 17, 18, 19, 20):
        _, ends = kernel_windows(monkeypatch, 3, 12, nch, env)
        assert ends[-1] == nch - 1 and all(ends[i] >= i for i in range(nch))
        for _ in range(60):
            assert run_drains(T, S, ends, rng) is None


@pytest.mark.parametrize("T,S,W,nch", [(2, 3, 5, 16), (3, 3, 5, 21), (3, 4, 5, 16)])
def test_short_last_windows_go_wrong(T, S, W, nch):
    """With the remainder in the last window its drain can come early; with a wait for the window before after the
    arrival, that window may be over by two phases when the wait starts, whose parity then never shows again."""
    rng = random.Random(10 * T + S)
    ends = last_window_short(nch, W)
    assert any("drain" in (run_drains(T, S, ends, rng) or "") for _ in range(2000))
    assert any(run_drains(T, S, ends, rng, "after") == "stall" for _ in range(2000))


@pytest.mark.parametrize("order,nshell,default", [(3, 12, 128), (4, 10, 14), (2, 12, 128), (5, 8, 12)])
@pytest.mark.parametrize("env,window", [(None, None), ("1", 5), ("3", 5), ("4", 5), ("5", 5), ("6", 6), ("0", None)])
def test_window_holds_more_chunks_than_there_are_slots(monkeypatch, order, nshell, default, env, window):
    assert kernel_windows(monkeypatch, order, nshell, 8, env)[0] == (window or default)

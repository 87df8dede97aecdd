"""The planner that cuts a layer into phases (csrc/pp_phase.h), compiled on the
CPU: every gate in exactly one phase, in order, and the label that deals
strings to blocks is the same for a string and for every string a gate of the
phase mixes it with -- also after other gates of the phase have acted."""
import os
import subprocess

import numpy as np
import pytest

import pp_inputs as pi

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "plan")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fsanitize=address,undefined",
                    os.path.join(HERE, "phase_plan_main.cpp"), "-o", exe], check=True)
    return exe


def as_int(words):
    return sum(int(w) << (64 * j) for j, w in enumerate(words))


def plan(driver, gates, n, activity, max_active, max_bits, occ, damp=0, tri=0):
    """(touched flags, [(first, count, commuting, ux, uz)]), gates: [(x, z)] as
    integers, occ: the OR of the strings' x and z bits."""
    W = (n + 63) // 64
    words = lambda v: [str((v >> (64 * j)) & (2 ** 64 - 1)) for j in range(W)]  # noqa: E731
    text = "%d %d %g %d %d %d %s\n" % (W, len(gates), max_active, max_bits, damp, tri,
                                    " ".join(words(occ[0]) + words(occ[1])))
    for (x, z), a in zip(gates, activity):
        text += " ".join([repr(float(a)), *words(x), *words(z)]) + "\n"
    out = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout
    lines = out.split("\n")
    rows = []
    for line in lines[1:]:
        if line:
            v = [int(t) for t in line.split()]
            rows.append((v[0], v[1], v[2], as_int(v[3:3 + W]), as_int(v[3 + W:])))
    return [int(t) for t in lines[0].split()], rows


def anticommute(a, b):
    return bin((a[0] & b[1]) ^ (a[1] & b[0])).count("1") & 1


def sum_or(values):
    out = 0
    for v in values:
        out |= v
    return out


def label(q, gates, phase, touch):
    """The kernels' label; no string that is dealt anticommutes with a gate that
    touches nothing, so those do not enter it."""
    first, count, commuting, ux, uz = phase
    active = 0
    if commuting:
        ux = uz = 0
        for k in range(count):
            if touch[first + k] and anticommute(gates[first + k], q):
                active |= 1 << k
                ux |= gates[first + k][0]
                uz |= gates[first + k][1]
    return active, q[0] & ~ux, q[1] & ~uz


CIRCUITS = {
    "ring5": (5, pi.ring_layer(5, 1, 1, 1)), "ring40": (40, pi.ring_layer(40, 1, 1, 1)),
    "ring130": (130, pi.ring_layer(130, 1, 1, 1)), "torus": (30, pi.torus_layer(5, 6, 1, 1, 1)),
    "heisenberg": (9, pi.heisenberg_layer(9, 1, 1, 1)),
    "random": (70, pi.random_circuit(70, 1, 90, seed=3).layers[0]),
    "one": (1, [("X", 1.0), ("Z", 1.0), ("Y", 1.0)]),
}


@pytest.mark.parametrize("name", sorted(CIRCUITS))
@pytest.mark.parametrize("tri", [0, 1])
@pytest.mark.parametrize("activity,max_active,max_bits,low", [
    (0.09, 3.0, 10, 0), (0.5, 1.0, 4, 0), (0.0, 3.0, 0, 0), (0.09, 3.0, 10, 3), (0.3, 2.0, 8, 1)])
def test_phases_cover_the_layer_and_close_under_it(driver, name, activity, max_active, max_bits, low,
                                                          tri):
    """low > 0: the strings start on the lowest `low` qubits only, so many gates
    touch nothing; strings then follow the gates from there."""
    n, layer = CIRCUITS[name]
    gx, gz = pi.to_masks([g[0] for g in reversed(layer)], n)
    gates = [(as_int(a), as_int(b)) for a, b in zip(gx, gz)]
    rng = np.random.default_rng(len(gates))
    room = (1 << (min(low, n) or n)) - 1
    strings = [tuple(as_int(rng.integers(0, 2 ** 63, 3)) & room for _ in range(2)) for _ in range(40)]
    touch, phases = plan(driver, gates, n, [activity] * len(gates), max_active, max_bits, (room, room),
                         tri=tri)
    at = 0
    for p in phases:
        assert p[0] >= at and 1 <= p[1] <= 32 and touch[p[0]] and touch[p[0] + p[1] - 1]
        assert not any(touch[at:p[0]])  # left out: no string anticommutes there
        mine = [k for k in range(p[0], p[0] + p[1]) if touch[k]]
        if p[2] == 3:  # a bit of every generator that no later one has
            for a in mine:
                later = [gates[b] for b in mine if b > a]
                assert any(gates[a][w] & ~sum_or(g[w] for g in later) for w in (0, 1))
        if p[2]:
            assert not any(anticommute(gates[a], gates[b]) for a in mine for b in mine)
            assert len(mine) == 1 or activity * (len(mine) - 0.5) <= max_active + 1e-6
        else:
            assert bin(p[3]).count("1") + bin(p[4]).count("1") <= max_bits
        for i, q in enumerate(strings):
            want = label(q, gates, p, touch)
            for k in range(p[0], p[0] + p[1]):
                g = gates[k]
                if anticommute(g, q):
                    assert touch[k]
                    if rng.random() < 0.7:
                        q = (q[0] ^ g[0], q[1] ^ g[1])
                assert label(q, gates, p, touch) == want
            strings[i] = q
        at = p[0] + p[1]
    assert not any(touch[at:])


def test_touched_gates_follow_the_letters(driver):
    """A gate touches when its letters can anticommute with, or (damped) meet,
    a letter that is there or that an earlier gate of the layer brought."""
    gates = [(0b1, 0), (0, 0b1), (0, 0b10), (0b110, 0), (0b10, 0)]  # X0 Z0 Z1 X1X2 X1
    act = [0.1] * len(gates)
    assert plan(driver, gates, 3, act, 3.0, 10, (0, 0b1))[0] == [1, 1, 0, 0, 0]
    assert plan(driver, gates, 3, act, 3.0, 10, (0, 0b100))[0] == [0, 0, 0, 1, 0]
    assert plan(driver, gates, 3, act, 3.0, 10, (0b10, 0), damp=1)[0] == [0, 0, 1, 1, 1]
    assert plan(driver, gates, 3, act, 3.0, 10, (0, 0))[0] == [0] * 5

"""Phases cut so that no class can outgrow its room (csrc/pp_phase.h), on the CPU: 2^r
strings for r commuting gates or r key bits."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("bound") / "bound")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fsanitize=address,undefined",
                    os.path.join(HERE, "phase_bound_main.cpp"), "-o", exe], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True).stdout
        return out.strip()
    return run


@pytest.mark.parametrize("plain,bits", [(32, 10), (9, 9), (8, 8), (7, 7)])
@pytest.mark.parametrize("tri", [0, 1])
@pytest.mark.parametrize("n,gates,support", [(9, 60, 1), (20, 200, 2), (64, 300, 2), (150, 200, 1)])
def test_no_phase_passes_the_bound(driver, n, gates, support, tri, plain, bits):
    total = [0, 0, 0]
    for seed in range(5):
        got = driver(n, gates, support, seed, 10, plain, bits, tri)
        kinds = got.split()
        assert len(kinds) == 3 and all(k.isdigit() for k in kinds), got
        total = [a + int(b) for a, b in zip(total, kinds)]
    assert sum(total) > 5 and (tri or total[2] == 0)


@pytest.mark.parametrize("n", [3, 8, 20, 64])
@pytest.mark.parametrize("limit", [0, 1, 64, 10000])
def test_a_plan_of_too_many_phases_stops(tmp_path_factory, n, limit):
    exe = str(tmp_path_factory.mktemp("stop") / "stop")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fsanitize=address,undefined",
                    os.path.join(HERE, "phase_stop_main.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, str(n), str(limit)], capture_output=True, text=True, check=True).stdout
    whole, part, same = map(int, out.split())
    assert part == min(whole, limit + 1) and same

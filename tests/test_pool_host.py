"""What the memory pool may keep of the memory nothing uses (csrc/pp_pool_host.h), on
the CPU."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
G = 1 << 30


@pytest.fixture(scope="module")
def keep(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pool") / "pool")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Wextra", "-Werror", "-fsanitize=address,undefined",
                    os.path.join(HERE, "pool_main.cpp"), "-o", exe], check=True)

    def run(*args):
        return int(subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True).stdout)
    return run


@pytest.mark.parametrize("unused,free,total,ends,want", [
    (0, 0, 276 * G, 1, 0), (G, 0, 276 * G, 1, G), (G, 0, 276 * G, 0, G),  # little is kept always
    (5 * G, 200 * G, 276 * G, 1, 5 * G), (20 * G, 200 * G, 276 * G, 1, 8 * G),  # between contexts
    (20 * G, 200 * G, 276 * G, 0, 20 * G), (60 * G, 69 * G, 276 * G, 0, 60 * G),  # of a context that goes on
    (60 * G, 69 * G - 1, 276 * G, 0, G), (20 * G, 10 * G, 276 * G, 1, G), (2 * G, 0, 276 * G, 0, G)])
def test_rule(keep, unused, free, total, ends, want):
    assert keep(unused, free, total, ends) == want

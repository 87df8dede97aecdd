"""The server's rule for memory lent to a phased layer (csrc/pp_admission.h), on the
CPU: only what no running and no queued job could have meanwhile."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def may_lend(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("lend") / "lend")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Wextra", "-Werror", "-fsanitize=address,undefined",
                    os.path.join(HERE, "lending_main.cpp"), "-o", exe], check=True)

    def run(budget, reserved, extra, growing=0, running=1, slots=2, queued=()):
        args = [budget, reserved, extra, growing, running, slots, *queued]
        return subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True).stdout == "1\n"
    return run


@pytest.mark.parametrize("want,kw", [
    (True, dict()),
    (True, dict(extra=70)), (False, dict(extra=71)), (False, dict(extra=2 ** 63)),  # the budget
    (False, dict(growing=1)),  # a running job needs memory
    (True, dict(queued=[20])), (False, dict(queued=[21])),  # would just fit beside it, would not any more
    (True, dict(queued=[71])),  # would not fit either way
    (False, dict(queued=[71, 70, 1])),
    (True, dict(queued=[70], running=2)),  # no slot free
    (False, dict(extra=1, reserved=100))])
def test_rule(may_lend, want, kw):
    case = dict(budget=100, reserved=30, extra=50)
    case.update(kw)
    assert may_lend(**case) == want

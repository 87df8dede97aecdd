"""The sizes of the phases' buckets (csrc/pp_phase.h), compiled on the CPU."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rooms(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("rooms") / "rooms")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fsanitize=address,undefined",
                    os.path.join(HERE, "phase_rooms_main.cpp"), "-o", exe], check=True)

    def run(strings, kinds, factor=1.0, blocks=(700, 304), warps=(368, 1824)):
        text = " ".join(map(str, [strings, factor, *blocks, *warps, *kinds]))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.strip().split("\n")]
    return run


@pytest.mark.parametrize("strings", [1, 255, 10 ** 4, 3 * 10 ** 5, 10 ** 7])
def test_each_phase_by_what_takes_its_buckets(rooms, strings):
    """A phase of warps has a bucket for each warp also where other phases of the
    layer, or those that truncation allows, are of blocks; and the other way round."""
    alone = {k: rooms(strings, [k])[0] for k in (0, 1)}
    assert alone[0][0] >= 1824 and alone[1][0] >= 304
    assert rooms(strings, [1, 0, 0, 1]) == [alone[1], alone[0], alone[0], alone[1]]


@pytest.mark.parametrize("factor", [1.0, 2.0, 8.0])
@pytest.mark.parametrize("strings", [1, 3 * 10 ** 5, 123456789])
@pytest.mark.parametrize("kind,fill,least", [(0, 368, 1824), (1, 700, 304)])
def test_fill_and_room(rooms, strings, factor, kind, fill, least):
    (nb, cg), = rooms(strings, [kind], factor)
    assert nb >= least and nb * fill >= strings * factor
    assert nb == least or (nb - 1) * fill < strings * factor
    assert cg >= 248 + 4 * strings / nb - 8 and cg <= 256 + 4 * strings / nb

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

    def run(terms, kinds, growth=1.2, possible=1e18, factor=1.0, blocks=(700, 304), warps=(368, 1824)):
        """(strings expected, buckets and room of each phase); growth 1.2: half as many again"""
        text = " ".join(map(str, [terms, growth, possible, factor, *blocks, *warps, *kinds]))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        lines = out.strip().split("\n")
        return float(lines[0].split()[0]), [tuple(map(int, line.split())) for line in lines[1:]]
    return run


@pytest.mark.parametrize("terms", [1, 255, 10 ** 4, 3 * 10 ** 5, 10 ** 7])
def test_each_phase_by_what_takes_its_buckets(rooms, terms):
    """A phase of warps has a bucket for each warp also where other phases of the
    layer, or those that truncation allows, are of blocks; and the other way round."""
    alone = {k: rooms(terms, [k])[1][0] for k in (0, 1)}
    assert alone[0][0] >= 1824 and alone[1][0] >= 304
    assert rooms(terms, [1, 0, 0, 1])[1] == [alone[1], alone[0], alone[0], alone[1]]


@pytest.mark.parametrize("factor", [1.0, 2.0, 8.0])
@pytest.mark.parametrize("terms", [1, 2 * 10 ** 5, 82304526])
@pytest.mark.parametrize("kind,fill,least", [(0, 368, 1824), (1, 700, 304)])
def test_fill_and_room(rooms, terms, factor, kind, fill, least):
    strings, ((nb, cg),) = rooms(terms, [kind], factor=factor)
    assert strings == 1.5 * terms
    assert nb >= least and nb * fill >= strings * factor
    assert nb == least or (nb - 1) * fill < strings * factor
    assert cg % 8 == 0 and cg >= 248 + 4 * strings / nb - 8 and cg <= 256 + 4 * min(strings / least, fill / factor)


@pytest.mark.parametrize("terms,growth,possible,want", [
    (1000, 1.0, 1e18, 1500), (1000, 2.0, 1e18, 2500), (1000, 20.0, 1e18, 25000), (1000, 26.0, 1e18, 32000),
    (3280, 3280.0, 65536, 65536), (9841, 9841.0, 262144, 262144), (8836, 2800.0, 1e18, 32 * 8836),
    (100, 1e9, 1e18, 3200), (10 ** 9, 1e9, 1e18, 32e9), (100, 2.0, 120, 120)])
def test_a_growth_is_extrapolated_so_far(rooms, terms, growth, possible, want):
    """A first layer that multiplies one term by thousands says nothing of the kind
    about the next, and no layer ends with more strings than the tables hold (whose
    room stops at twice the 4^n strings there are)."""
    strings, sizes = rooms(terms, [0, 1], growth, possible)
    assert strings == pytest.approx(want, rel=1e-12)
    for (nb, cg), fill, least in zip(sizes, (368, 700), (1824, 304)):
        assert least <= nb <= max(least, -(-want // fill))
        assert cg <= 256 + 4 * fill  # and room for lumps of up to four buckets' fill

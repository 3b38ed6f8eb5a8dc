"""How the n-tiles of a narrow seq2seq roll-out come to blocks (csrc/s2s_split.h), compiled for the host."""
import ctypes as C
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_05008_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("s2s_split")
    src, lib = str(d / "split.cc"), str(d / "libsplit.so")
    with open(src, "w") as f:
        f.write('#include "s2s_split.h"\nextern "C" void split(uint32_t u, uint32_t m, uint32_t t, uint32_t d, uint32_t* o)'
                "{ const evo::S2sSplit s = evo::s2s_split(u, m, t, d, 148); o[0] = s.chunk; o[1] = s.chunks; o[2] = s.places; }\n"
                'extern "C" uint32_t pieces(uint32_t f, uint32_t e, uint32_t t, uint32_t m) { return evo::s2s_pieces(f, e, t, m); }\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
    return C.CDLL(lib)


def _split(lib, units, members, tiles, digits=2):
    out = (C.c_uint32 * 3)()
    lib.split(units, members, tiles, digits, out)
    return tuple(out)


def test_pieces_are_those_that_a_block_works_off(lib):
    rng = random.Random(1)
    for _ in range(2000):
        tiles, most, first = rng.randint(1, 60), rng.choice([8, 14]), rng.randint(0, 500)
        end = first + rng.randint(1, 200)
        at, n = first, 0
        while at < end:                                     # as the kernel does
            left = min(end - at, tiles - at % tiles)
            at += -(-left // -(-left // most))
            n += 1
        assert lib.pieces(first, end, tiles, most) == n


@pytest.mark.parametrize("units", [32, 64, 96])
def test_every_tile_has_its_block(lib, units):
    rng = random.Random(units)
    for _ in range(3000):
        members, tiles = rng.choice([2, 30, 148, 296, 300, 1000, 5000]), rng.randint(1, 70)
        chunk, chunks, places = _split(lib, units, members, tiles, rng.randint(1, 4))
        if chunk == 0:                                      # runs: none of them empty
            assert units != 32 and members * tiles >= places
        else:                                               # chunks: all tiles, the last chunk not empty, eight tiles at most
            assert chunk <= 8 and chunk * chunks >= tiles > chunk * (chunks - 1)


def test_runs_count_their_tiles_in_32_bits(lib):
    """One tile fewer than 2^32 and as many: the latter in chunks."""
    assert _split(lib, 64, 65537, 65535)[0] == 0
    assert _split(lib, 64, 65536, 65536)[0] == 8


# units, digits, queries, members, whether runs are faster
MEASURED = [(64, 1, 47, 52, True), (64, 2, 100, 300, True), (64, 2, 100, 600, True), (64, 2, 64, 298, True), (64, 2, 8, 400, False), (64, 2, 24, 1000, False),
            (64, 2, 40, 400, False), (64, 2, 56, 100, False), (64, 2, 56, 1000, False), (64, 2, 64, 1000, False), (64, 3, 15, 192, False),
            (64, 1, 66, 844, True), (64, 4, 64, 400, False), (64, 1, 37, 432, False), (64, 4, 151, 214, True),
            (96, 2, 16, 200, True), (96, 2, 24, 200, True), (96, 2, 100, 300, True), (96, 2, 64, 600, True), (96, 2, 24, 400, False),
            (96, 2, 16, 400, False), (96, 3, 18, 356, False), (96, 4, 16, 440, False), (96, 2, 400, 298, True)]


@pytest.mark.parametrize("units,digits,queries,members,runs", MEASURED)
def test_the_faster_form_is_taken(lib, units, digits, queries, members, runs):
    """Sizes at which one of the two was measured at least 5 % faster."""
    assert (_split(lib, units, members, (queries + 7) // 8, digits)[0] == 0) == runs


def test_items_of_128_units_cover_the_batch_and_fill_the_gpu(tmp_path):
    src, out = str(tmp_path / "items.cc"), str(tmp_path / "libitems.so")
    with open(src, "w") as f:
        f.write('#include "s2s_split.h"\nextern "C" void items(uint32_t m, uint32_t q, uint32_t d, uint32_t* o)'
                "{ const evo::S2sSplit s = evo::s2s_items(m, q, d, 148); o[0] = s.chunk; o[1] = s.chunks; }\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", out, src], check=True)
    fn, o = C.CDLL(out).items, (C.c_uint32 * 2)()
    rng = random.Random(3)
    for members, queries, digits in [(2, 1, 1), (2, 16, 4), (1 << 20, 128, 3)] + [(rng.randint(2, 3000), rng.randint(1, 700), rng.randint(1, 4)) for _ in range(3000)]:
        fn(members, queries, digits, o)
        chunk, chunks = o
        assert chunk % 8 == 0 and 0 < chunk <= 128 and (chunks - 1) * chunk < queries <= chunks * chunk
        assert chunks <= (queries + 7) // 8                      # the scratch memory has a sum for every 8 queries
        if members >= 148 * 20:
            assert chunks == -(-queries // 128)                  # nothing to fill
    for members, queries, chunk in [(1024, 128, 128), (37, 128, 32), (74, 128, 64), (148, 128, 128), (148, 130, 72), (82, 362, 128)]:
        fn(members, queries, 3, o)
        assert o[0] == chunk, (members, queries, o[0])

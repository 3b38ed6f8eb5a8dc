"""Which kernel a control policy of three or four hidden layers runs on (csrc/mlp_choice.h), compiled for the host."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_05008_b200", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("mlp_choice")
    src, lib = str(d / "choice.cc"), str(d / "libchoice.so")
    with open(src, "w") as f:
        f.write('#include "mlp_choice.h"\nextern "C" uint32_t resident(uint32_t r, size_t s, uint32_t t) { return evo::resident_blocks(r, s, t); }\n'
                'extern "C" double waves(uint64_t b, uint32_t r) { return evo::mlp_waves(b, 148, r); }\n'
                'extern "C" bool pays(uint32_t h, bool w, uint32_t e, uint64_t b, uint32_t rd, uint32_t rm)'
                "{ return evo::mlp_deep_pays(h, w, e, b, 148, rd, rm); }\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
    lib = C.CDLL(lib)
    lib.resident.argtypes, lib.resident.restype = [C.c_uint32, C.c_size_t, C.c_uint32], C.c_uint32
    lib.waves.argtypes, lib.waves.restype = [C.c_uint64, C.c_uint32], C.c_double
    lib.pays.argtypes, lib.pays.restype = [C.c_uint32, C.c_bool, C.c_uint32, C.c_uint64, C.c_uint32, C.c_uint32], C.c_bool
    return lib


# hidden layers, one above 64 units, episodes and number of blocks, blocks on an SM of the kernel with the weights in registers and of that
# with the weights in shared memory, whether the former is faster.  Roll-outs where one of them was measured at least 10 % faster
MEASURED = [
    (3, False, 4, 1300, 8, 12, True),   # 28-6-15-24-8: 2.02 / 2.55 us a step
    (3, False, 8, 900, 5, 8, True),     # 5-32-39-35-1: 2.62 / 3.33
    (3, True, 4, 1000, 2, 3, True),     # 5-48-90-112-1: 5.95 / 7.44
    (3, True, 4, 1000, 2, 4, False),    # 5-70-16-112-1: 5.15 / 4.61
    (3, True, 4, 304, 2, 5, False),     # 5-70-10-90-1: 2.47 / 2.11
    (3, True, 8, 2000, 2, 3, True),     # 5-55-91-70-1: 12.50 / 16.02
    (3, True, 8, 1000, 2, 5, False),    # 5-70-10-90-1: 6.80 / 5.12
    (3, True, 8, 304, 2, 5, False),     # 5-40-20-90-1: 3.15 / 2.45
    (4, False, 4, 2000, 4, 6, True),    # 28-52-22-6-34-8: 5.33 / 7.20
    (4, False, 4, 1300, 4, 9, False),   # 28-16-60-7-11-8: 3.72 / 3.16
    (4, False, 8, 2000, 4, 6, True),    # 5-13-50-34-40-1: 7.65 / 9.25
    (4, False, 8, 740, 4, 6, False),    # 28-53-8-16-43-8: 3.51 / 3.17
    (4, True, 4, 1000, 1, 2, True),     # 28-128-48-48-80-8: 7.75 / 10.37
    (4, True, 4, 400, 1, 4, False),     # 28-100-10-32-60-8: 3.06 / 2.41
    (4, True, 4, 592, 1, 6, False),     # 5-25-15-60-66-1: 4.37 / 2.87
    (4, True, 8, 152, 1, 2, True),      # 5-60-60-100-40-1: 2.59 / 3.19
    (4, True, 8, 740, 1, 5, False),     # 5-14-9-8-82-1: 6.13 / 3.29
    (4, True, 8, 400, 1, 4, False),     # 5-112-32-16-10-1: 3.44 / 2.76
]


@pytest.mark.parametrize("hidden,wide,eb,blocks,deep,mma,faster", MEASURED)
def test_the_faster_kernel_is_taken(lib, hidden, wide, eb, blocks, deep, mma, faster):
    assert lib.pays(hidden, wide, eb, blocks, deep, mma) == faster


def test_no_more_waves_than_the_other_kernel_is_always_faster(lib):
    for hidden in (3, 4):
        for wide in (False, True):
            for eb in (4, 8):
                for blocks in (1, 147, 148, 149, 295, 297, 1000, 4096, 5000):
                    for resident in range(1, 9):
                        assert lib.pays(hidden, wide, eb, blocks, resident, resident)


def test_kernels_that_do_not_fit(lib):
    assert lib.pays(4, True, 4, 5000, 1, 0)                 # the weights do not fit the shared memory
    assert not lib.pays(4, True, 4, 5000, 0, 1)
    assert lib.pays(1, True, 4, 5000, 1, 12)                # one hidden layer: never measured slower


def test_waves(lib):
    assert lib.waves(148, 1) == 1.0 and lib.waves(149, 1) == 2.0 and lib.waves(296, 2) == 1.0
    assert lib.waves(148, 2) == pytest.approx(0.8) and lib.waves(445, 2) == 2.0


@pytest.mark.parametrize("regs,smem,threads,blocks", [
    (128, 0, 256, 2), (128, 0, 160, 3), (126, 0, 128, 4), (129, 0, 128, 3), (200, 0, 160, 1), (211, 0, 32, 8), (56, 0, 288, 4), (255, 0, 512, 0),
    (32, 0, 1024, 2), (24, 0, 1024, 2), (16, 0, 32, 32),                         # 64 warps, 32 blocks
    (32, 57 * 1024 - 1024, 128, 4), (32, 57 * 1024 - 1023, 128, 3), (32, 227 * 1024, 128, 1)])
def test_blocks_that_an_sm_holds(lib, regs, smem, threads, blocks):
    assert lib.resident(regs, smem, threads) == blocks


# blocks, resident blocks of the kernel with the weights in registers and of that with them in shared memory, whether the former is faster
@pytest.mark.parametrize("blocks,deep,mma,faster", [
    (118, 1, 3, True),      # 5-15-189-54-1: 76 / 124 us
    (676, 1, 3, False),     # 5-107-29-138-1: 430 / 325
    (836, 1, 1, True),      # 28-145-157-59-8: 661 / 1,159
    (424, 1, 3, False),     # 28-154-13-77-8: 259 / 158
    (288, 1, 2, False),     # 28-168-47-11-8: 168 / 149
    (354, 1, 1, True),      # 28-46-135-132-8: 245 / 486
    (296, 1, 0, True),      # 28-180-180-180-8: 196 / 3,436 through the caches
])
def test_the_faster_kernel_is_taken_above_128_units(tmp_path, blocks, deep, mma, faster):
    src, out = str(tmp_path / "widest.cc"), str(tmp_path / "libwidest.so")
    with open(src, "w") as f:
        f.write('#include "mlp_choice.h"\nextern "C" bool pays(uint64_t b, uint32_t rd, uint32_t rm) { return evo::mlp_widest_pays(b, 148, rd, rm); }\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", out, src], check=True)
    fn = C.CDLL(out).pays
    fn.argtypes, fn.restype = [C.c_uint64, C.c_uint32, C.c_uint32], C.c_bool
    assert fn(blocks, deep, mma) == faster


# hidden layers, widest of them, cart-pole, on k_rollout_mlp2, members, episodes, steps, whether blocks of four episodes are the faster ones
@pytest.mark.parametrize("hidden,widest,cart,registers,members,episodes,steps,faster", [
    (2, 64, True, True, 74, 8, 20, False),       # 5-64-64-1: blocks of eight / of four 15.1 / 16.1 us
    (2, 64, True, True, 74, 8, 200, True),       # 111.4 / 106.6
    (2, 64, True, True, 37, 16, 20, True),       # 16.2 / 15.4 (36 members; both have the second launch)
    (2, 40, True, True, 70, 5, 50, False),       # 5-17-40-1: 28.5 / 28.5
    (1, 30, True, False, 74, 8, 80, False),      # 5-30-1: 30.7 / 31.0
    (1, 20, False, False, 74, 8, 20, False),     # 28-20-8: 11.8 / 12.2
    (1, 20, False, False, 74, 8, 50, True),      # 23.2 / 22.4
    (2, 64, False, True, 16, 5, 20, True),       # 28-64-64-8: 16.8 / 16.1
    (2, 119, False, True, 74, 8, 20, True),      # 28-119-25-8: 23.9 / 21.6
    (2, 119, False, True, 148, 8, 50, True),     # 51.1 / 47.5
    (2, 119, False, True, 149, 8, 50, False),    # more than two blocks an SM
    (3, 64, False, False, 74, 8, 20, True),      # 28-64-64-64-8: 22.6 / 21.7
    (3, 64, False, False, 75, 8, 200, False),
    (0, 0, True, False, 74, 8, 32, False),       # 5-1: 17.3 / 17.6
])
def test_episodes_a_block(tmp_path, hidden, widest, cart, registers, members, episodes, steps, faster):
    src, out = str(tmp_path / "four.cc"), str(tmp_path / "libfour.so")
    with open(src, "w") as f:
        f.write('#include "mlp_choice.h"\nextern "C" bool four(uint32_t h, uint32_t w, bool c, bool r, uint32_t m, uint32_t e, uint32_t t)'
                "{ return evo::mlp_four_pay(h, w, c, r, m, e, t, 148); }\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", out, src], check=True)
    fn = C.CDLL(out).four
    fn.argtypes, fn.restype = [C.c_uint32, C.c_uint32, C.c_bool, C.c_bool, C.c_uint32, C.c_uint32, C.c_uint32], C.c_bool
    assert fn(hidden, widest, cart, registers, members, episodes, steps) == faster

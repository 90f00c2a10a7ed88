"""How the wide chain kernel cuts up a chain, on devices of every size: the header's host functions, compiled alone."""
import ctypes
import os
import subprocess

import pytest

from paper_2411_11925_b200 import build


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src = d / "plan.cpp"
    src.write_text('#include "wideplan.h"\n'
                   'extern "C" int groups(int pairs, int W) { return csd::wide_groups(pairs, W); }\n'
                   'extern "C" int pays(int L, int W, int rows) { return csd::wide_pays(L, W, rows); }\n'
                   'extern "C" void cut(int most, int W, int R, int cfg, int halves, int* o) {\n'
                   '  const csd::WideCut c = csd::wide_cut(most, W, R, cfg, halves);\n'
                   '  o[0] = c.nb; o[1] = c.slots; o[2] = c.part; o[3] = c.ctas;\n}\n')
    lib = d / "plan.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", f"-I{build.CSRC}", str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


def _cut(plan, *a):
    o = (ctypes.c_int * 4)()
    plan.cut(*a, o)
    return list(o)


@pytest.mark.parametrize("W", range(768, 2049, 256))
def test_every_launch_fits_the_device_and_a_device_without_room_for_a_group_is_told(plan, W):
    pairs_of_group = W // 128
    for pairs in (1, 5, 6, 7, 8, 9, 10, 15, 16, 17, 37, 72, 74):
        most = plan.groups(pairs, W)
        assert most == pairs // pairs_of_group            # 0: nothing is cut there, the layer kernels run
        if most == 0:
            continue
        for cfg in (0, 1):
            for R in (129, 257, 300, 1024, 2304, 4608):
                for halves in (1, 2):
                    nb, slots, part, ctas = _cut(plan, most, W, R, cfg, halves)
                    tokens, gs = 64 if cfg else 128, 2 // halves
                    assert nb % 2 == 0 and (nb - 2) * tokens < R <= nb * tokens and slots == nb // 2
                    in_launch = min(part, slots)
                    assert part % gs == 0 and -(-in_launch // gs) <= most
                    assert ctas == -(-in_launch // gs) * 2 * pairs_of_group <= 2 * pairs


def test_cuts_of_a_whole_device(plan):
    # 74 pairs: 1024 rows of 1024 with guidance, 4096 rows of 1536, 3072 of 2048 in the two forms
    assert _cut(plan, plan.groups(74, 1024), 1024, 512, 1, 2) == [8, 4, 4, 64]
    assert _cut(plan, plan.groups(74, 1536), 1536, 2048, 1, 1) == [32, 16, 8, 96]
    assert _cut(plan, plan.groups(74, 2048), 2048, 1536, 1, 2) == [24, 12, 4, 128]


def test_rows_that_take_the_kernel(plan):
    for L, W, least, most in ((1, 768, 683, 4608), (1, 1024, 512, 4608), (1, 1280, 410, 3710), (1, 1536, 342, 3092), (1, 2048, 257, 2319),
                              (2, 768, 257, 4608), (2, 1024, 257, 4608), (12, 1280, 257, 3710), (12, 1536, 257, 3092), (8, 2048, 257, 2319)):
        assert [plan.pays(L, W, r) for r in (1, least - 1, least, most, most + 1, 1 << 30)] == [0, 0, 1, 1, 0, 0], (L, W)

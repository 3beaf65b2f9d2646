"""The layout rules of the vision-encoding calls (host code without CUDA), compiled by themselves: the choices
that timings of both sides of each line are written beside."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_10803_b200", "csrc")
SOURCE = """
#include "vision_plan.h"
extern "C" int merge_fly(int vecs) { return mustdrop::merge_fly(vecs); }
extern "C" int key_rows(int head_dim, int part, int ctas, int sms) {
  return static_cast<int>(mustdrop::key_rows(head_dim, part, ctas, sms));
}
extern "C" int merge_cluster(int batch, int n_win, const int* resident) {
  return mustdrop::merge_cluster(batch, n_win, resident);
}
"""
# clusters of 1 .. 8 CTAs that a B200 holds at once with three CTAs of the merge on an SM
THREE_ON_AN_SM = (444, 222, 142, 104, 82, 71, 56, 48)


(LANE_PER_VECTOR5, LANE_PER_VECTOR3_AHEAD, FOUR1X3_AHEAD, FOUR1X5, FOUR2X2, FOUR2X2_AHEAD, FOUR3X1_AHEAD, EIGHT2X2,
 EIGHT4X1_AHEAD) = range(9)                                             # enum KeyRows


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("vision_plan")
    (d / "rules.cpp").write_text(SOURCE)
    so = str(d / "rules.so")
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Werror", "-I", CSRC, "-o", so, str(d / "rules.cpp")])
    return ctypes.CDLL(so)


def merge_cluster(rules, batch, n_win, resident=THREE_ON_AN_SM):
    return rules.merge_cluster(batch, n_win, (ctypes.c_int * 9)(0, *resident))


@pytest.mark.parametrize("batch,n_win,cluster", [
    (96, 36, 4), (111, 36, 3), (74, 64, 5), (74, 49, 5), (157, 25, 2),   # as many rounds: the fewest waves
    (64, 144, 6), (37, 81, 8), (1, 144, 8), (100, 64, 4), (40, 49, 7),   # fewest rounds, then the most CTAs
    (1, 1, 1), (19, 1, 1), (16, 9, 2), (65535, 576, 1),
])
def test_ctas_per_image_of_the_merge(rules, batch, n_win, cluster):
    assert merge_cluster(rules, batch, n_win) == cluster


def test_the_merge_is_laid_out_without_an_answer_about_the_device(rules):
    # (nothing known: one cluster at a time, whatever its size)
    assert merge_cluster(rules, 5, 144, (1,) * 8) == 8


def test_a_second_vector_in_flight_needs_rows_that_have_one(rules):
    assert [rules.merge_fly(v) for v in (1, 2, 12, 32, 33, 64, 173)] == [1, 1, 1, 1, 2, 2, 2]


@pytest.mark.parametrize("part", [1, 5, 20, 36, 127])
@pytest.mark.parametrize("ctas", [8, 296, 512])
def test_eight_lanes_share_rows_of_more_than_96_dimensions(rules, part, ctas):
    assert [rules.key_rows(d, part, ctas, 148) for d in (96, 104, 128, 136, 256)] == [FOUR3X1_AHEAD, EIGHT2X2, EIGHT2X2, EIGHT4X1_AHEAD,
                                                                               EIGHT4X1_AHEAD]


@pytest.mark.parametrize("head_dim,part,ctas,rows", [
    (8, 121, 96, LANE_PER_VECTOR5), (16, 121, 96, LANE_PER_VECTOR5), (8, 36, 192, LANE_PER_VECTOR5), (8, 16, 768, LANE_PER_VECTOR5),
    (16, 16, 768, FOUR1X3_AHEAD), (16, 19, 32, FOUR1X3_AHEAD), (8, 19, 32, FOUR1X3_AHEAD), (8, 25, 32, LANE_PER_VECTOR5),
    (24, 24, 192, FOUR1X3_AHEAD), (24, 25, 192, FOUR1X5), (32, 36, 8, FOUR1X5), (32, 40, 320, FOUR1X5), (32, 41, 320, FOUR1X3_AHEAD),
])
def test_rows_of_up_to_32_dimensions(rules, head_dim, part, ctas, rows):
    assert rules.key_rows(head_dim, part, ctas, 148) == rows


@pytest.mark.parametrize("part,ctas,sms,rows", [
    (36, 192, 148, FOUR2X2), (109, 312, 148, FOUR2X2), (20, 320, 148, FOUR2X2), (36, 369, 148, FOUR2X2), (36, 370, 148, LANE_PER_VECTOR3_AHEAD),
    (36, 512, 148, LANE_PER_VECTOR3_AHEAD), (36, 512, 296, FOUR2X2), (16, 512, 148, FOUR2X2_AHEAD), (17, 512, 148, LANE_PER_VECTOR5),
    (20, 768, 148, LANE_PER_VECTOR5), (21, 768, 148, LANE_PER_VECTOR3_AHEAD),
])
@pytest.mark.parametrize("head_dim", [40, 64])
def test_rows_of_33_to_64_dimensions(rules, head_dim, part, ctas, sms, rows):
    assert rules.key_rows(head_dim, part, ctas, sms) == rows

"""CPU: the rules that choose between two forms of a kernel (csrc/ssvp_dispatch.h), compiled by the host compiler: on
which side the measured sizes lie.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2102_03011_gb300", "csrc")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")

    def ask(*calls):
        d = tmp_path_factory.mktemp("rules")
        src = d / "r.cpp"
        src.write_text('#include <cstdio>\n#include "ssvp_dispatch.h"\nint main() {\n'
                       + "".join(f'    printf("%d\\n", (int)ssvp::{c});\n' for c in calls) + "}\n")
        subprocess.check_call([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(d / "r")])
        return [int(x) for x in subprocess.check_output([str(d / "r")]).split()]
    return ask


def test_long_hulls(rule):
    def call(T, W, band):
        return f"frustum_long_hulls({2 * T + 1}, {W}, {band}f)"
    yes = [(15, 1280, 3.0), (30, 640, 3.0), (30, 1280, 3.0), (30, 1280, 1.0), (30, 1920, 9.0), (60, 640, 1.5), (15, 1920, 9.0), (60, 1280, 0.5)]
    # short hulls gain nothing, and the instance that can drop their blocks spills
    no = [(0, 1920, 3.0), (15, 1280, 1.0), (15, 1280, 9.0), (30, 640, 9.0), (30, 640, 1.0), (15, 960, 3.0), (30, 320, 3.0), (15, 1920, 1.0), (30, 1280, 0.5)]
    assert rule(*(call(*c) for c in yes)) == [1] * len(yes)
    assert rule(*(call(*c) for c in no)) == [0] * len(no)


def ctas(W, H, n=1):
    return (W + 31) // 32 * ((H + 7) // 8) * n


SMS = 152


def test_frustum_frames_shared(rule):
    def call(W, H, T):
        return f"frustum_shares({ctas(W, H)}, {3 * SMS}, {2 * T + 1})"
    yes = [(96, 54, 1), (160, 90, 1), (256, 144, 2), (320, 180, 2), (320, 180, 3), (320, 180, 15), (480, 270, 3), (480, 270, 15)]
    # one frame has nothing to share; short windows of larger images; full chips
    no = [(96, 54, 0), (320, 180, 0), (320, 180, 1), (480, 270, 0), (480, 270, 2), (640, 360, 3), (640, 360, 15), (1280, 720, 30)]
    assert rule(*(call(*c) for c in yes)) == [1] * len(yes)
    assert rule(*(call(*c) for c in no)) == [0] * len(no)


def test_window_frames_shared(rule):
    def call(W, H, T, k, n=1):
        return f"window_shares({ctas(W, H, n)}, {4 * SMS}, {2 * T + 1}, {k})"
    yes = [(96, 54, 1, 7), (320, 180, 1, 7), (320, 180, 15, 3), (480, 270, 3, 7), (560, 316, 5, 7), (640, 360, 3, 7), (640, 360, 15, 3), (160, 90, 15, 5, 16),
           (320, 180, 15, 7, 6)]
    no = [(96, 54, 0, 7), (320, 180, 0, 3), (480, 270, 0, 7), (480, 270, 1, 3), (480, 270, 2, 7), (560, 316, 1, 7), (640, 360, 2, 7), (640, 360, 5, 3),
          (853, 479, 5, 7), (853, 479, 15, 7), (1280, 720, 30, 7)]
    assert rule(*(call(*c) for c in yes)) == [1] * len(yes)
    assert rule(*(call(*c) for c in no)) == [0] * len(no)


def test_aperture_frames_shared(rule):
    def call(W, H, T, ctas_per_sm=4):
        return f"aperture_shares({ctas(W, H)}, {ctas_per_sm * SMS}, {2 * T + 1})"
    yes = [(96, 54, 1), (320, 180, 1), (320, 180, 2), (480, 270, 2), (640, 360, 1), (640, 360, 3), (853, 479, 15), (640, 360, 3, 3)]
    no = [(96, 54, 0), (320, 180, 0), (640, 360, 0), (640, 360, 2), (853, 479, 2), (853, 479, 15, 3), (1280, 720, 15)]
    assert rule(*(call(*c) for c in yes)) == [1] * len(yes)
    assert rule(*(call(*c) for c in no)) == [0] * len(no)


def test_extraction_ctas(rule):
    sizes = [(160, 90), (320, 180), (480, 270), (532, 293), (640, 360), (1920, 1080)]
    assert rule(*(f"extract_four_ctas({ctas(*s)}, {SMS})" for s in sizes)) == [0, 0, 1, 0, 0, 0]

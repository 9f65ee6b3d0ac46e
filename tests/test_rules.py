"""CPU test of the rules that choose a kernel form by the sizes of a call
(csrc/rbsm_rules.h): each line lies where the two forms' measured times cross,
and calls outside a form's reach do not take it."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """rule(expression): the value of a C++ expression over the rules."""
    def evaluate(expr):
        d = tmp_path_factory.mktemp("rule")
        (d / "rule.cpp").write_text('#include <cstdio>\n#include "rbsm_rules.h"\nusing namespace rbsm;\n'
                                    'int main() { std::printf("%%d", (int)(%s)); }\n' % expr)
        csrc = os.path.join(ROOT, "paper_1711_07793_gb300", "csrc")
        subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", csrc, str(d / "rule.cpp"), "-o", str(d / "rule")],
                       check=True)
        return int(subprocess.run([str(d / "rule")], capture_output=True, text=True, check=True).stdout)
    return evaluate


@pytest.mark.parametrize("size,rects,spheres,scale_in_range,large", [
    (8192, 140, 60, True, True),
    (4096, 1, 0, True, True),
    (2240, 24, 0, True, True),          # 35^2 tiles of 64, two for each of four CTAs on 152 SMs
    (2176, 24, 0, True, False),
    (8192, 0, 0, True, False),          # nothing to cull: the stores alone
    (4096, 0, 0, True, False),
    (4096, 200, 56, True, True),
    (4096, 200, 57, True, False),       # more than one culling round
    (8192, 257, 0, True, False),
    (4096, 100, 50, False, False),      # every covered texel of a sphere in double precision
    (4096, 100, 0, False, True),        # rectangles do not read the depth scale
])
def test_light_pass_tiles(rule, size, rects, spheres, scale_in_range, large):
    assert rule("light_large_tiles(%d, %d, %d, %d, %s, %d)"
                % (size, size, rects, spheres, str(scale_in_range).lower(), SMS)) == large


@pytest.mark.parametrize("w,h,spread", [(128, 128, False), (160, 192, False), (192, 192, True), (512, 512, True),
                                        (1024, 1024, True), (1216 * 32, 32, True), (1216 * 32 + 1, 32, False),
                                        (2048, 2048, False)])
def test_light_pass_rows(rule, w, h, spread):
    assert rule("light_spread_rows(%d, %d, %d)" % (w, h, SMS)) == spread


@pytest.mark.parametrize("w,h,large", [(320, 240, False), (1280, 720, False), (128, 64 * SMS - 1, False),
                                       (127, 64 * SMS, False), (128, 64 * SMS, True), (1920, 1080, True),
                                       (3840, 2160, True), (65536, 65536, True)])
def test_depth_buffer_ctas(rule, w, h, large):
    assert rule("gbuffer_large(%d, %d, %d)" % (w, h, SMS)) == large

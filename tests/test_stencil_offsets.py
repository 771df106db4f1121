"""Offsets into a stored 27-point stencil (component-major, 27 n_x values): they pass 2^31 from 79.6 million points on, and
such levels fit the GPU's memory (Q1 on 128 x 800 x 800 in FP32).  The kernels with 32-bit offsets (k_st27 and the
row kernels' kind 3) are launched on smaller levels only."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_16863_gb300", "csrc")


def _source(name):
    return re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())


@pytest.fixture(scope="module")
def kind(tmp_path_factory):
    """level_kind(fine = 0, d, nx) compiled for the host from its source."""
    mg = _source("mg.cuh")
    rule = re.search(r"constexpr bool sten32_ok\(long long nx\) \{[^}]*\}", mg).group(0)
    fn = mg[mg.index("inline int level_kind("):]
    fn = fn[:fn.index("}") + 1]
    d = tmp_path_factory.mktemp("kind")
    (d / "t.cpp").write_text("#include <cstdio>\n#include <cstdlib>\n" + rule + "\n" + fn +
                             '\nint main(int, char** a) { std::printf("%d", level_kind(atoi(a[1]), atoi(a[2]), atoll(a[3]))); }\n')
    subprocess.run(["g++", "-std=c++17", "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return lambda fine, dim, nx: int(subprocess.run([str(d / "t"), str(fine), str(dim), str(nx)], capture_output=True,
                                                    text=True, check=True).stdout)


@pytest.mark.parametrize("nx", [1, 96 ** 3, 79536431, 79536432, 128 * 800 * 800, 159072863, 2 ** 31 - 1])
def test_kernels_with_32_bit_offsets_take_levels_that_fit(kind, nx):
    largest = 27 * nx - 1                       # the last component's last point
    assert (kind(0, 3, nx) == 3) == (largest < 2 ** 31 - 1)
    assert kind(0, 3, nx) in (0, 3) and kind(0, 2, nx) == 2 and kind(1, 3, nx) == 1


def test_every_launch_asks_the_rule():
    mg, pre = _source("mg.cuh"), _source("precond.cuh")
    body = mg[mg.index("inline bool st27_ok("):]
    assert "sten32_ok(op.g.nx)" in body[:body.index("}")]
    for m in re.finditer(r"launch\(k_st27<", pre):
        before = pre[:m.start()]
        assert "st27_ok(op, B)" in before[before.rindex("if constexpr"):]
    calls = re.findall(r"level_kind\(([^()]*)\)", pre)
    assert calls and all(c == "op.fine, g.d, g.nx" for c in calls)


def test_other_component_offsets_are_64_bit():
    """Outside those two kernels a component times the level's size is a 64-bit product."""
    for path in ("mg.cuh", "cluster_mg.cuh", "precond.cuh", "noalloc.cu"):
        text = _source(path)
        if path == "mg.cuh":
            for start, end in (("constexpr (KIND == 3) {", "diag = s[13];"), ("k_st27(", "sten32_ok(op.g.nx)")):
                i = text.index(start)
                text = text[:i] + text[text.index(end, i):]
        for m in re.finditer(r"\bsten\s*(?:\[[^\]]*\])?\s*(?:\+|\[)[^;,]*", text):
            if re.search(r"\bq \* |\bk \* nx|\d \* nx", m.group(0)):
                assert "(long long)" in m.group(0) or "4 * nx" in m.group(0), m.group(0)

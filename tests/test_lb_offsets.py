"""The stream-collide kernel addresses a population's plane in 64 bits: boxes
are accepted up to 2^30 cells (check_desc in api.cu), whose rows may be padded
to twice that, so that 18 planes pass 2^31 cells from 119 M on.  The rule that
forms the offset is compiled by the host compiler as it stands in the kernel's
source and held against Python's integers, and nothing else in that source
multiplies by the plane's size."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LB = open(os.path.join(ROOT, "paper_2503_20605_gb300", "csrc", "lb.cu")).read()
SIZES = [8, 119304647, 119304648, 134217728, 1 << 30, 1908874353, (1 << 31) - 16]


def test_plane_offsets_pass_32_bits(tmp_path):
    rule = re.search(r"constexpr int64_t plane_offset\(.*?\)\s*\{.*?\}", LB, re.S).group(0)
    src, exe = tmp_path / "o.cpp", tmp_path / "o"
    src.write_text("#include <cstdint>\n#include <cstdio>\n" + rule + "\nint main() {\n" +
                   "".join(f'    std::printf("%lld\\n", (long long)plane_offset({i}, {n}));\n'
                           for n in SIZES for i in range(19)) + "}\n")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-fsanitize=undefined", "-fno-sanitize-recover",
                    "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out] == [i * n for n in SIZES for i in range(19)]


def test_no_other_product_with_a_plane():
    code = re.sub(r"//[^\n]*|/\*.*?\*/", "", LB, flags=re.S)
    assert not re.findall(r"\*\s*(?:c\.)?PC\b|\b(?:c\.)?PC\s*\*", code)
    assert len(re.findall(r"\bplane_offset\(\w+, (?:c\.)?PC\)", code)) == 5

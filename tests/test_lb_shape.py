"""The stream-collide kernel's group size and pipeline depth: they follow from
the boxes and from what the options ask for, whatever was asked for before; a
depth that fits is given, with a group that leaves room for it; every shape
fits a block's shared memory for every row that two stages of one row fit.
The header that the library uses is compiled by the host compiler."""
import os
import random
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_20605_gb300", "csrc")
LAUNCH = 227 * 1024 - 128       # opt-in shared memory of a block less the kernel's 128 bytes of barriers
SHAPE = 227 * 1024 - 1024

MAIN = r"""
#include <cstdio>
#include "lb_shape.h"
using namespace iblb;
int main()
{
    int n, sb, cells, mult, stages;
    while (std::scanf("%d %d %d %d %d", &n, &sb, &cells, &mult, &stages) == 5) {
        std::vector<LbBox> b(n);
        for (auto &x : b)
            if (std::scanf("%d %d %d %d", &x.nx, &x.ny, &x.nzf, &x.mask_pitch) != 4)
                return 1;
        LbRequest ask;
        ask.cells = cells;
        ask.mult = mult;
        ask.stages = stages;
        const LbShape s = lb_shape(b, sb, 152, ask);
        std::printf("%d %d %d", s.cells, s.stages, s.stage_bytes);
        for (auto &x : b) {
            const int r = lb_group_rows(s.cells, s.mult, x, sb, n > 1);
            std::printf(" %d %d", r, (int)lb_mask_staged(r, x, sb, n > 1));
        }
        std::printf("\n");
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    (d / "s.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-o", str(d / "s"), str(d / "s.cpp")],
                   check=True)

    def run(cases):
        """cases: (boxes, bytes per value, cells, mult, stages) -> (cells, stages, stage bytes, [(rows, staged)])"""
        text = "".join(f"{len(b)} {sb} {c} {m} {s} " + " ".join("%d %d %d %d" % x for x in b) + "\n"
                       for b, sb, c, m, s in cases)
        out = subprocess.run([str(d / "s")], input=text, check=True, capture_output=True, text=True).stdout
        res = []
        for line in out.splitlines():
            v = [int(x) for x in line.split()]
            res.append((v[0], v[1], v[2], list(zip(v[3::2], v[4::2]))))
        return res
    return run


def bits(nx):
    return (nx + 127) // 128 * 16


def need(rows, nx, sb, several, mask):
    """Bytes of a stage: 19 populations, 3 forces, bits, header, constants."""
    P = -(-nx // (16 // sb)) * (16 // sb)
    return rows * (19 * P * sb + 12 * P + mask) + 16 + (128 if several else 0)


def test_an_asked_depth_is_given(shapes):
    for sb in (2, 4):
        for box in [(128, 128, 126, 0), (80, 80, 58, 0), (32, 32, 30, 0), (200, 160, 62, bits(200))]:
            for ns in range(2, 9):
                cells, stages, _, rows = shapes([([box], sb, -1, 2, ns)])[0]
                fits = ns * need(1, box[0], sb, False, box[3]) <= SHAPE - 8 * 128
                assert stages == ns if fits else 2 <= stages < ns, (box, sb, ns)


def test_an_asked_group_gets_a_depth_of_its_own(shapes):
    # 128^3 FP32: one depth for groups of 128 cells, whatever stood before, and the default depths are 2 or 3
    for sb, cells in ((4, 128), (4, 768), (2, 128), (2, 512), (2, 768), (2, 2048)):
        c, stages, size, rows = shapes([([(128, 128, 126, 0)], sb, cells, 2, 0)])[0]
        assert c == cells and stages in (2, 3) and stages * size <= SHAPE
        if 3 * need(rows[0][0], 128, sb, False, 0) + 3 * 128 <= 114 * 1024 - 1152:
            assert stages == 3              # two blocks of three stages fit an SM
    # the multiplier: 256 threads' rows
    assert shapes([([(100, 90, 8, 0)], 4, 0, 3, 0)])[0][3][0][0] == 6
    assert shapes([([(300, 90, 8, 0)], 4, 0, 3, 0)])[0][3][0][0] == 3


def test_every_shape_fits(shapes):
    rng = random.Random(5)
    cases = []
    for _ in range(600):
        sb = rng.choice((2, 4))
        top = rng.choice((64, 400, 1316 if sb == 4 else 2320))
        n = rng.choice((1, 1, 2, 5))
        b = []
        for _ in range(n):
            nx = rng.randint(8, top)
            b.append((nx, rng.randint(8, 200), rng.randint(6, 200), rng.choice((0, bits(nx)))))
        cases.append((b, sb, rng.choice((-1, -1, 0, rng.randint(1, 16384))), rng.randint(1, 4), rng.choice((0, 0, 2, 5, 8))))
    edge = [([(nx, 9, 8, m)] + more, sb, -1, 2, s) for sb, xs in ((4, (1309, 1313, 1316)), (2, (2305, 2313, 2320)))
            for nx in xs for m in (0, bits(nx)) for more in ([], [(9, 8, 8, 0)]) for s in (0, 2, 8)]
    for (b, sb, cells, mult, ns), (c, stages, size, rows) in zip(cases + edge, shapes(cases + edge)):
        assert 2 <= stages <= max(3, ns) and stages * size <= LAUNCH and size % 16 == 0
        for (nx, ny, nzf, mask), (r, staged) in zip(b, rows):
            assert 1 <= r <= ny and need(r, nx, sb, len(b) > 1, mask if staged else 0) <= size
            if not staged and mask:
                assert r == 1 and sb == 2 and nx > 2312
    # one cell of padding more does not fit, as it never did
    for sb, nx in ((4, 1317), (2, 2321)):
        assert 2 * shapes([([(nx, 9, 8, 0)], sb, -1, 2, 0)])[0][2] > LAUNCH


def test_the_library_keeps_no_shape_but_the_request():
    api = open(os.path.join(CSRC, "api.cu")).read()
    assert len(re.findall(r"cfg\.lb_stages\s*=", api)) == 1 and "lb_shape(boxes" in api
    body = api[api.index("int iblb_set_option("):api.index("int iblb_get_profile(")]
    assert body.count("return reshape(c, ask);") == 3 and "layout(" not in body

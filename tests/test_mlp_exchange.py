"""The exchanges between the CTAs of the network's kernel: no piece may be sent
while an earlier one could still be on its way to the same place, be read
there, or be copied from the same memory.  The header that the kernel takes its
senders and receivers from is compiled by the host compiler; a second model,
written here from the rules of the copies alone, plays random orders of arrival
and looks for a piece that meets an earlier one.  Both refuse the output
layer's inputs going to CTAs that do not answer them."""
import os
import random
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_20605_gb300", "csrc")
NC = 8
# (buffer, senders, receivers, units)
ALL = {"H1": (0, 8, 8, 32), "H2": (1, 8, 8, 32), "H3": (0, 8, 4, 32), "DY": (1, 4, 8, 16), "D3": (0, 8, 8, 32),
       "D2": (1, 8, 8, 32)}
TRAIN = list(ALL)
# tables with a fault: h3 to CTAs that do not answer it; one buffer for two exchanges in a row; nobody answers
FAULTS = {"h3 to all": {"H3": (0, 8, 8, 32)}, "dy in h3's buffer, d3 unanswered": {"DY": (0, 4, 4, 16)},
          "h2 to half": {"H2": (1, 8, 4, 32), "H3": (1, 4, 8, 32)}}


@pytest.fixture(scope="module")
def header(tmp_path_factory):
    """What the header says of the tables: its own, and those with a fault."""
    d = tmp_path_factory.mktemp("exchange")

    def table(t):
        return "{" + ", ".join("{%d, %d, %d, %d}" % t[n] for n in TRAIN) + "}"
    lines = ["#include <cstdio>", '#include "mlp_exchange.h"', "using namespace iblb;", "int main() {"]
    for n in TRAIN:
        lines.append(f'    std::printf("EX_{n} %d %d %d %d\\n", EX_{n}.buffer, EX_{n}.senders, EX_{n}.receivers, '
                     f"EX_{n}.units);")
    for i, f in enumerate(FAULTS.values()):
        lines.append(f"    const Exchange f{i}[] = {table({**ALL, **f})};")
        lines.append(f'    std::printf("fault {i} %d\\n", (int)ordered(f{i}));')
    lines.append('    std::printf("own %d %d\\n", (int)ordered(EX_FORWARD), (int)ordered(EX_TRAINING));')
    src, exe = d / "x.cpp", d / "x"
    src.write_text("\n".join(lines + ["}"]) + "\n")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [line.split() for line in out.splitlines()]


def test_header_orders_its_exchanges_and_refuses_faults(header):
    assert [tuple(int(v) for v in h[1:]) for h in header if h[0].startswith("EX_")] == [ALL[n] for n in TRAIN]
    assert ["own", "1", "1"] in header
    assert [h[2] for h in header if h[0] == "fault"] == ["0"] * len(FAULTS)


def play(table, rng):
    """One run with arrivals in a random order: True if some piece met an earlier one."""
    at = [0] * NC                       # the exchange that each CTA works on
    sent = [False] * NC
    flying = []                         # (exchange, sender, receiver)
    got = [[set() for _ in table] for _ in range(NC)]
    while any(a < len(table) for a in at):
        moves = [("land", f) for f in flying]
        for c in range(NC):
            k = at[c]
            if k == len(table):
                continue
            b, ns, nr, _ = table[k]
            if not sent[c]:
                moves.append(("send", c))
            elif c >= nr or got[c][k] == set(range(ns)) - {c}:
                moves.append(("done", c))
        kind, m = rng.choice(moves)
        if kind == "land":
            flying.remove(m)
            got[m[2]][m[0]].add(m[1])
        elif kind == "done":
            at[m] += 1
            sent[m] = False
        else:
            k = at[m]
            b, ns, nr, _ = table[k]
            sent[m] = True
            if m >= ns:
                continue
            # its own memory is still being copied from
            if any(f[1] == m and table[f[0]][0] == b and f[0] < k for f in flying):
                return True
            for r in range(nr):
                if r == m:
                    continue
                # the receiver has not finished an earlier exchange of that buffer
                if any(table[e][0] == b and r < table[e][2] and at[r] <= e for e in range(k)):
                    return True
                flying.append((k, m, r))
    return False


@pytest.mark.parametrize("fault", [None, *FAULTS])
def test_random_orders_of_arrival(fault):
    table = [{**ALL, **(FAULTS[fault] if fault else {})}[n] for n in TRAIN]
    rng = random.Random(7)
    met = [play(table, rng) for _ in range(400 if fault else 150)]
    assert any(met) == (fault is not None)


def test_kernel_takes_the_exchanges_in_that_order():
    src = open(os.path.join(CSRC, "mlp.cu")).read()
    assert re.findall(r"^\s*publish\((\w+)", src, re.M) == [n.lower() for n in TRAIN]
    assert re.findall(r"^\s*product\((\w+),", src, re.M) == [n.lower() for n in TRAIN]
    assert len(re.findall(r"\bsend\(sa\[", src)) == 1

"""The rule on late launches (csrc/launch_chain.h), compiled for the host (CPU only): a
launch may start before its predecessor has completed only where nothing that may still be
running -- the last launch that waited at its start, and every late one since -- writes
what it reads or touches what it writes."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_16188_gb300", "csrc")

# Lines "w reads... / writes..." (on time), "l reads... / writes..." (late if it may be) or "u ..."
# (it may be, but is not wanted); a buffer is "address:bytes".  Prints 1 or 0 for each l and u.
PROGRAM = r"""
#include <cstdio>
#include <iostream>
#include <sstream>
#include <string>
#include <vector>
#include "launch_chain.h"
using namespace vmoe;
int main() {
    LaunchChain c;
    std::string line, w;
    while (std::getline(std::cin, line)) {
        std::istringstream in(line);
        std::vector<Span> s[2] = {{}, {}};
        std::string kind;
        in >> kind;
        int k = 0;
        while (in >> w) {
            if (w == "/") { k = 1; continue; }
            const size_t p = w.find(':');
            s[k].push_back(Span{(const void *)std::stoull(w.substr(0, p)), (size_t)std::stoull(w.substr(p + 1))});
        }
        Span none{nullptr, 0};
        for (auto &v : s) v.resize(4, none);
        LaunchChain::Spans r = {s[0][0], s[0][1], s[0][2], s[0][3]}, q = {s[1][0], s[1][1], s[1][2], s[1][3]};
        if (kind == "w") c.on_time(r, q);
        else printf("%d\n", (int)c.late(r, q, kind != "u"));
    }
}
"""


@pytest.fixture(scope="module")
def chain(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("chain")
    (d / "c.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(d / "c"), str(d / "c.cpp")], check=True)

    def run(text):
        r = subprocess.run([str(d / "c")], input=text, check=True, capture_output=True, text=True)
        return [int(x) for x in r.stdout.split()]
    return run


XE, ACT, DYE, W1, W2, DH, DXE, DW1, DW2 = ("%d:1000" % (4096 * i) for i in range(1, 10))


def backward(dw1=DW1, dw2=DW2, dxe=DXE):
    return "w %s %s / %s\nw %s %s / %s\nl %s %s / %s\nl %s %s / %s\n" % (
        DYE, W2, DH, DH, W1, dxe, XE, DH, dw1, ACT, DYE, dw2)


def test_the_backwards_weight_gradients_are_late(chain):
    assert chain(backward()) == [1, 1]


def test_a_gradient_over_what_an_open_launch_reads_waits(chain):
    assert chain(backward(dw1=W1)) == [0, 1]            # dX may still read W1
    assert chain(backward(dw2=W1)) == [1, 0]            # two launches back
    assert chain(backward(dw2=W2)) == [1, 1]            # dA has completed
    assert chain(backward(dw1="%d:1000" % (4096 * 4 + 999))) == [0, 1]  # its last byte
    assert chain(backward(dw1="%d:1000" % (4096 * 4 + 1000))) == [1, 1]


def test_the_output_of_an_open_launch_is_waited_for(chain):
    assert chain("l %s / %s\n" % (XE, DW1)) == [0]      # an entry point's first launch
    assert chain("w %s / %s\nl %s / %s\n" % (XE, DH, DH, DW1)) == [0]
    # a late launch that reads what the launch two back writes
    assert chain("w %s / %s\nl %s / %s\nl %s / %s\n" % (XE, DXE, ACT, DW1, DXE, DW2)) == [1, 0]
    # ... and what a late one writes; behind an on-time launch it is complete
    assert chain("w %s / %s\nl %s / %s\nl %s / %s\n" % (XE, DXE, ACT, DW1, DW1, DW2)) == [1, 0]
    assert chain("w %s / %s\nl %s / %s\nw %s / %s\nl %s / %s\n" % (XE, DXE, ACT, DW1, XE, DH, DXE, DW2)) == [1, 1]


def test_an_unwanted_late_launch_is_on_time(chain):
    lines = "w %s / %s\n%s %s / %s\nl %s / %s\n"
    assert chain(lines % (XE, DXE, "l", ACT, DW1, DXE, DW2)) == [1, 0]
    assert chain(lines % (XE, DXE, "u", ACT, DW1, DXE, DW2)) == [0, 1]  # it has waited: dX has completed


def test_more_buffers_than_the_chain_holds(chain):
    lines = "w %s / %s\n" % (XE, DXE) + "l 1:1 2:1 3:1 4:1 / 5:1 6:1 7:1 8:1\n" * 4
    assert chain(lines)[0] == 1
    many = "w / 1:1\n" + "".join("l / %d:1\n" % (100 * i) for i in range(1, 12))
    got = chain(many)
    assert got[0] == 1 and 0 in got  # full: an on-time launch starts a new chain

"""The tensor-core kernel keeps a weight set in shared memory while items of the same key follow each
other, so a plan's keys name one (stage, output-channel block) each, also in layers of more than 256
blocks.  Checked on the item records themselves, by a program built from the host planner."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_06960_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <utility>
#include "planner.h"
using namespace mafat;
int main() {
    // 8336 = 16 x 521 channels: blocks of 16, 521 of them; the last layer's set is small enough to stay
    const int32_t layers[] = {L_CONV, 3, 1, 1, 8336, L_CONV, 1, 1, 0, 16, L_CONV, 3, 1, 1, 16};
    Net net;
    std::string err = build_net(layers, 3, 4, 4, 16, net);
    for (char& h : net.has_w) h = 1;
    PlanConfig cfg;
    PlanTables t;
    bool unsupported = false;
    if (err.empty()) err = build_plan(net, cfg, t, &unsupported);
    if (!err.empty()) return std::printf("%s\n", err.c_str()), 2;
    std::vector<MafatItemRec> recs;
    build_records(t, recs);
    std::map<uint32_t, std::pair<int, int>> of;
    int most = 0;
    for (size_t i = 0; i < recs.size(); ++i) {
        const std::pair<int, int> set(t.items[i].stage, t.items[i].nb);
        most = most < set.second ? set.second : most;
        auto at = of.insert({recs[i].mma.w[0], set}).first;
        if (at->second != set) return std::printf("stage %d block %d and stage %d block %d share a key\n", set.first, set.second, at->second.first, at->second.second), 1;
    }
    return most > 256 ? 0 : 3;
}
"""


def test_every_weight_set_has_a_key_of_its_own(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    src, exe = tmp_path / "keys.cpp", tmp_path / "keys"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), os.path.join(CSRC, "planner.cpp"),
                    os.path.join(CSRC, "order.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

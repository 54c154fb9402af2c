"""Limits of the device layout that no test machine reaches with real points:
the layout code compiled into a small host program."""
import os
import subprocess

from paper_2310_16668_gb300 import build

MAIN = r"""
#include <cstdio>
#include "host.h"
using namespace skel;
int main() {
    // three sets of 2^30 slots each: more than 2^31 together
    std::vector<Layout> sets(3);
    std::vector<const Layout*> lp;
    for (Layout& l : sets) {
        l.sym_slots = (int64_t)1 << 30;
        l.sym_items.resize(1);
        lp.push_back(&l);
    }
    Layout m;
    merge_layouts(lp, {1, 1, 1}, {1, 1, 1}, 1, m);
    std::printf("%lld %zu\n", (long long)m.sym_slots, m.sym_items.size());
}
"""


def test_merged_plan_has_no_limit_on_slots(tmp_path):
    """The slots of the symmetric translations are numbered within a batch, so
    their total number refuses no plan."""
    src = tmp_path / "main.cpp"
    src.write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-O1", "-std=c++17", "-fopenmp", "-I" + build.CSRC, str(src),
                    os.path.join(build.CSRC, "layout.cpp"), os.path.join(build.CSRC, "tree.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    assert out.stdout.split() == [str(3 << 30), "3"]

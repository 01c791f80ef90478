"""A call on a handle runs on the handle's device whichever is current, and
leaves the caller's current device as it was: the guard that every entry point
holds, against a fake device API."""
import os
import subprocess

CODE = r"""
#include <cassert>
#include <vector>
#include "o2pic_device.h"
struct Fake {
    static int now, fail_get, fail_set;
    static std::vector<int> sets;
    static int get(int *d) { *d = now; return fail_get; }
    static int set(int d) { if (fail_set) return fail_set; now = d; sets.push_back(d); return 0; }
};
int Fake::now = 0, Fake::fail_get = 0, Fake::fail_set = 0;
std::vector<int> Fake::sets;
using On = o2::OnDevice<Fake>;
static int call(int dev, bool early) { On on(dev); if (on.error()) return on.error(); assert(Fake::now == dev); if (early) return 7; return 0; }
int main()
{
    assert(call(0, false) == 0 && Fake::sets.empty() && Fake::now == 0);   // already current: nothing is set
    assert(call(3, false) == 0 && (Fake::sets == std::vector<int>{3, 0}) && Fake::now == 0);
    Fake::sets.clear(); Fake::now = 2;
    assert(call(1, true) == 7 && (Fake::sets == std::vector<int>{1, 2}) && Fake::now == 2);  // an early return too
    Fake::sets.clear();
    { On a(1); On b(1); On c(0); assert(Fake::now == 0); }                                   // nested
    assert(Fake::now == 2);
    Fake::sets.clear(); Fake::fail_set = 101;
    assert(call(1, false) == 101 && Fake::sets.empty() && Fake::now == 2);                   // no such device
    Fake::fail_set = 0; Fake::fail_get = 100;
    assert(call(1, false) == 100 && Fake::sets.empty());
    return 0;
}
"""


def test_the_guard_switches_and_restores(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(root, "paper_0705_0495_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)]).returncode == 0

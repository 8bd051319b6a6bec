"""What the launchers remember of a kernel's occupancy (csrc/resident.h) belongs to one device, cluster size and
shared-memory size.  Checked by a small C++ program built from the header itself (no GPU needed)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "resident.h"
using namespace mvla;
static ResidentClusters r;                       // zero like the launchers' own
#define CHECK(c) if (!(c)) { std::printf("failed: %s\n", #c); return 1; }
int main()
{
    for (int dev = 0; dev < ResidentClusters::kDevices; ++dev) CHECK(r.find(dev, 4, 212992) == 0);
    r.keep(0, 4, 212992, 33);
    CHECK(r.find(0, 4, 212992) == 33);
    CHECK(r.find(1, 4, 212992) == 0);            // another device has to be asked itself
    r.keep(1, 4, 212992, 16);
    CHECK(r.find(0, 4, 212992) == 33 && r.find(1, 4, 212992) == 16);
    CHECK(r.find(0, 8, 212992) == 0 && r.find(0, 4, 212991) == 0);
    r.keep(0, 4, 1024, 90);                      // the last question of a cluster size is kept
    CHECK(r.find(0, 4, 1024) == 90 && r.find(0, 4, 212992) == 0 && r.find(1, 4, 212992) == 16);
    r.keep(0, 2, 0, 0);                          // no answer is not one
    CHECK(r.find(0, 2, 0) == 0);
    r.keep(0, 2, 0, 7);
    CHECK(r.find(0, 2, 0) == 7);
    for (int dev : {-1, ResidentClusters::kDevices, 1 << 20}) { r.keep(dev, 1, 0, 5); CHECK(r.find(dev, 1, 0) == 0); }
    for (int size : {-1, ResidentClusters::kSizes}) { r.keep(2, size, 0, 5); CHECK(r.find(2, size, 0) == 0); }
    std::printf("ok\n");
    return 0;
}
"""


def test_occupancy_of_one_device_is_not_taken_for_another(tmp_path):
    src = tmp_path / "resident.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "resident"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2604_09244_b200", "csrc"),
                    "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


BLOCK_SIZES = r"""
#include <cstdio>
#include <initializer_list>
#include "resident.h"
using namespace mvla;
static ResidentClusters r;
#define CHECK(c) if (!(c)) { std::printf("failed: %s\n", #c); return 1; }
int main()
{
    r.keep(3, 1, 200000, 148, 320);
    CHECK(r.find(3, 1, 200000, 384) == 0);       // the streaming kernel with two more warps has to be asked itself
    r.keep(3, 1, 200000, 74, 384);
    CHECK(r.find(3, 1, 200000, 320) == 148 && r.find(3, 1, 200000, 384) == 74);      // and an answer is kept for each
    CHECK(r.find(3, 1, 200000, 448) == 0);       // (of the same place as 320)
    for (int t : {-1, ResidentClusters::kMaxThreads + 1}) { r.keep(2, 1, 0, 5, t); CHECK(r.find(2, 1, 0, t) == 0); }
    r.keep(3, 2, 1, ResidentClusters::kMaxCount + 1, 320);
    CHECK(r.find(3, 2, 1, 320) == 0);
    std::printf("ok\n");
    return 0;
}
"""


def test_occupancy_of_one_block_size_is_not_taken_for_another(tmp_path):
    src, exe = tmp_path / "blocks.cpp", tmp_path / "blocks"
    src.write_text(BLOCK_SIZES)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2604_09244_b200", "csrc"),
                    "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout

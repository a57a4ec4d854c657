"""The cluster size a kernel is launched with (csrc/cluster_plan.h), against a
stand-in for the CUDA calls: the kernel's attributes are set on every device that
asks, a size that cannot be scheduled gives way to the next one and in the end to
no cluster, and a query that failed is asked again."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_04763_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "cluster_plan.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)
struct Devices {
  int current = 0, asked = 0, limit = 16;
  bool allowed[2] = {false, false}, broken = false;
};
struct Api {
  Devices& d;
  int device() { return d.current; }
  size_t smem_optin() { return 1000; }
  bool allow(size_t cap) { CHECK(cap == 1000); return d.allowed[d.current] = !d.broken; }
  int clusters(int cs, size_t smem) {
    ++d.asked;
    CHECK(smem <= 1000);
    if (d.broken || !d.allowed[d.current]) return -1;
    return cs <= d.limit ? 1 : 0;
  }
};
int main() {
  Devices d;
  rf::ClusterAnswers known;
  auto smem = [](int cs) { return (size_t)(4000 / cs); };   // 4 and more CTAs fit
  auto plan = [&] { return rf::choose_cluster(Api{d}, known, 0, {16, 8, 4, 2, 1}, smem); };
  CHECK(plan() == 16 && d.asked == 1);
  CHECK(plan() == 16 && d.asked == 1);                      // known
  d.current = 1;                                            // a second device has attributes of its own
  CHECK(plan() == 16 && d.allowed[1] && d.asked == 2);
  Devices e;
  rf::ClusterAnswers known_e;
  auto plan_e = [&] { return rf::choose_cluster(Api{e}, known_e, 0, {16, 8, 4, 2, 1}, smem); };
  e.limit = 8;
  CHECK(plan_e() == 8);
  e.current = 1;
  e.limit = 2;                                              // 2 CTAs would run, but need too much memory
  CHECK(plan_e() == 0);
  Devices f;
  rf::ClusterAnswers known_f;
  f.broken = true;
  CHECK(rf::choose_cluster(Api{f}, known_f, 0, {16}, smem) == 0);
  f.broken = false;
  CHECK(rf::choose_cluster(Api{f}, known_f, 0, {16}, smem) == 16);
  CHECK(known_f.fits({9, 9, 9, 9}, [] { return -1; }) == false && known_f.fits({9, 9, 9, 9}, [] { return 1; }));
  return 0;
}
"""


def test_cluster_choice(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "plan.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "plan")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe, "-pthread"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_cluster_kernel_of_this_kind_is_planned_so():
    """No launch parameter of a kernel is remembered from the device that asked first."""
    text = open(os.path.join(CSRC, "levelops.cu")).read()
    plan = text[text.index("static int lu_cluster("):text.index("static cudaError_t launch_lu_cluster(")]
    assert "choose_cluster_of(" in plan
    plan = text[text.index("bool tail_cl_plan("):text.index("cudaError_t launch_vcycle_cl(")]
    assert "choose_cluster_of(" in plan

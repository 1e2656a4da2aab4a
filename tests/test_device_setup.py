"""The one-time set-up of a kernel per device: a set-up that failed is not remembered as done (no GPU needed).

Behind it stand checks without which a kernel may not run at all (a register split that would wait for registers that
never come free), so a second call must be refused like the first.
"""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1511_08486_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "per_device.cuh"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  sfb::PerDeviceOnce once;
  int runs = 0;
  auto fails = [&] { ++runs; return false; };
  auto works = [&] { ++runs; return true; };
  for (int call = 1; call <= 3; ++call) { CHECK(!once.ok(0, fails)); CHECK(runs == call); }
  CHECK(once.ok(0, works) && runs == 4);
  CHECK(once.ok(0, fails) && runs == 4);       // done: not run again
  CHECK(!once.ok(1, fails) && runs == 5);      // another device is on its own
  CHECK(once.ok(1, works) && once.ok(63, works) && runs == 7);
  CHECK(once.ok(63, fails) && runs == 7);
  for (int dev : {64, 127, -1}) { CHECK(!once.ok(dev, fails)); CHECK(once.ok(dev, works)); CHECK(!once.ok(dev, fails)); }
  return 0;
}
"""


def test_a_failed_set_up_stays_failed(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_a_route_is_taken_only_where_its_kernels_can_be_set_up():
    """The context of a large fp32 problem has either the tensor cores' workspace or the CUDA cores': both kernels' set-up is
    asked for before the first of it is allocated, while the other route is still open."""
    text = open(os.path.join(CSRC, "umma_f32.cu")).read()
    create = text[re.search(r"^int f32tc_create\(", text, flags=re.M).start():]
    create = create[:create.index("\n}\n")]
    for kernel in ("pairs_at_once<false>(", "pairs_at_once<true>("):
        assert 0 <= create.find(kernel) < create.index("cudaMalloc")

"""What a kernel needs once before its launches (its opt-in to large shared
memory, its grid) is kept per device: a handle on a second device of the same
process gets its own."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2207_14496_gb300", "csrc")

PROGRAM = r"""
#include "fsl_per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
enum Status { kOk = 0, kFail = 7 };
int main() {
  static fsl::PerDevice known;
  int made[80] = {};
  auto make = [&](int dev, Status st) {
    return [&made, dev, st](int* n) { ++made[dev]; *n = 100 + dev; return st; };
  };
  int n = 0, bad = 0;
  // a failure is returned and asked again
  bad += known.get(1, &n, make(1, kFail), kOk) != kFail;
  bad += known.get(1, &n, make(1, kOk), kOk) != kOk || n != 101 || made[1] != 2;
  // each device once, and its own number
  for (int round = 0; round < 3; ++round)
    for (int dev = 0; dev < fsl::PerDevice::kDevices; ++dev) {
      n = 0;
      bad += known.get(dev, &n, make(dev, kOk), kOk) != kOk || n != 100 + dev;
    }
  for (int dev = 0; dev < fsl::PerDevice::kDevices; ++dev) bad += made[dev] != (dev == 1 ? 2 : 1);
  // devices beyond the table: asked every time
  for (int k = 0; k < 2; ++k) bad += known.get(70, &n, make(70, kOk), kOk) != kOk || n != 170;
  bad += made[70] != 2;
  // threads that come first together
  static fsl::PerDevice other;
  std::vector<std::thread> th;
  int got[8][4] = {};
  for (int t = 0; t < 8; ++t)
    th.emplace_back([&got, t] {
      for (int dev = 0; dev < 4; ++dev)
        other.get(dev, &got[t][dev], [dev](int* m) { *m = 5 + dev; return kOk; }, kOk);
    });
  for (auto& t : th) t.join();
  for (auto& g : got)
    for (int dev = 0; dev < 4; ++dev) bad += g[dev] != 5 + dev;
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_kept_per_device(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"


def test_no_launch_parameter_is_kept_per_process():
    """Function-local statics of the launch code: launch tables and PerDevice only."""
    found = set()
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        # an indented `static` variable (declarations of functions end in a parameter list)
        found |= set(re.findall(r"^ +static (?:const )?(\w+) \w+(?:, \w+)*(?: = [^;(]*|\s*=\s*\w+\([^;]*)?;", text, re.M))
    assert found <= {"PerDevice", "Launch"}, found

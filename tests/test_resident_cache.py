"""The occupancy cache of the persistent kernels (host C++): one answer per kernel,
device, block size and shared memory, whatever was asked before."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2202_07017_gb300", "csrc")

MAIN = """
#include "resident_cache.cuh"
#include <thread>
#include <vector>
int main() {
  sv::ResidentCache c;
  int a = 0, b = 0, asked = 0;
  auto q = [&](int v) { return [&asked, v] { ++asked; return v; }; };
  if (c.get(&a, 0, 64, 1000, q(3)) != 3) return 1;
  if (c.get(&a, 0, 32, 1000, q(7)) != 7) return 2;   // another block size
  if (c.get(&a, 1, 64, 1000, q(5)) != 5) return 3;   // another device
  if (c.get(&b, 0, 64, 1000, q(2)) != 2) return 4;   // another kernel
  if (c.get(&a, 0, 64, 1024, q(1)) != 1) return 5;   // other shared memory
  if (c.get(&a, 0, 64, 1000, q(9)) != 3 || asked != 5) return 6;
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&] { for (int k = 1; k < 500; ++k) c.get(&b, 2, k, 0, [k] { return k; }); });
  for (auto& x : t) x.join();
  for (int k = 1; k < 500; ++k)
    if (c.get(&b, 2, k, 0, [] { return 0; }) != k) return 7;
  return 0;
}
"""


def test_every_part_of_a_configuration_counts(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_kernels_take_their_grids_from_it():
    """No launch keeps an occupancy of its own under a shorter key."""
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        assert "std::map<std::pair<const void*" not in text, name

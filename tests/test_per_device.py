"""Values that belong to a device are made once on each device, also by several threads (per_device.h), and
no launcher keeps one of them for the whole process."""
import glob
import os
import re

from tests.simt import CSRC, run

SRC = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "%s"
int main() {
  bse::PerDevice<int> v;
  std::atomic<int> made[4]{}, wrong{0};
  std::vector<std::thread> t;
  for (int i = 0; i < 16; ++i)
    t.emplace_back([&, i] {
      for (int k = 0; k < 200; ++k) {
        const int dev = (i + k) %% 4;
        if (v.get(dev, [&] { ++made[dev]; return 10 + dev; }) != 10 + dev) ++wrong;
      }
    });
  for (auto& x : t) x.join();
  printf("%%d %%d %%d %%d %%d\n", made[0].load(), made[1].load(), made[2].load(), made[3].load(), wrong.load());
}
"""


def test_made_once_per_device(tmp_path):
    assert run(tmp_path, SRC % os.path.join(CSRC, "per_device.h")) == [[1, 1, 1, 1, 0]]


def test_no_launcher_keeps_a_device_value_for_the_process():
    for f in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(f).read()
        assert not re.search(r"^\s*static\s+(const\s+)?(int|bool)\s+\w+(\[\d\])?\s*=", text, re.M), f

"""Host checks of headers that the kernels share with plain C++, at the limits of what the entry points
accept (sizes no test can run)."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1910_13529_gb300", "csrc")


def run_cpp(tmp_path, source, stdin=""):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(source)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], input=stdin, check=True, capture_output=True, text=True).stdout


def test_box_fit_at_the_limits_of_pic_create(tmp_path):
    """Boxes that span grids pic_create accepts (nz <= 32768, (nz + 2) nx ny < 2^31 - 1) against whole-number
    arithmetic: the 32-bit products 6 z x and 3 z x y wrap to small or negative values there."""
    boxes = [(4, 256, 1), (4, 257, 1), (32, 32, 1), (1024, 1, 1), (1028, 1, 1), (6144, 1, 1), (16, 12, 8), (20, 9, 9), (24, 13, 12),
             (24, 13, 13), (1706, 1, 1), (3754, 1, 1), (32772, 10922, 1), (32772, 21845, 1), (32772, 32764, 1), (32772, 65530, 1), (1028, 1028, 1028),
             (32768, 256, 256), (8, 2 ** 14, 2 ** 14), (4, 2 ** 28, 1), (4, 4, 2 ** 27), (2 ** 15, 2 ** 16, 1),
             (12, 2 ** 15 + 1, 2 ** 12), (1292, 1292, 1292)]
    wrapped = [b for b in boxes if (6 * b[0] * b[1] * b[2] + 2 ** 31) % 2 ** 32 - 2 ** 31 <= 6144 < 6 * b[0] * b[1] * b[2]]
    assert len(wrapped) >= 4                 # boxes that the 32-bit product takes for small ones
    source = """#include "box_fit.h"
    #include <cstdio>
    int main() { int z, x, y;
      while (std::scanf("%d %d %d", &z, &x, &y) == 3)
        std::printf("%d %d %d %d\\n", pic::box_fits<6, 6144>(z, x, y), pic::box_fits<3, 3072>(z, x, y),
                    pic::box_fits<6, 10240>(z, x, y), pic::box_fits<3, 11264>(z, x, y)); }"""
    out = run_cpp(tmp_path, source, "\n".join(" ".join(map(str, b)) for b in boxes))
    got = [[int(v) for v in line.split()] for line in out.splitlines()]
    assert got == [[int(c * z * x * y <= cap) for c, cap in ((6, 6144), (3, 3072), (6, 10240), (3, 11264))]
                   for z, x, y in boxes]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".h"))))
def test_cell_counts_are_not_narrowed(name):
    """nz nx ny reaches 2^31 and three components 3 2^31: no signed 32-bit copy that is then multiplied."""
    text = open(os.path.join(CSRC, name)).read()
    assert not re.search(r"\(int\)\s*\w+(\.|->)ncell", text)
    assert not re.search(r"\bint\s+\w+\s*=\s*\w+(\.|->)ncell", text)


def test_launch_setup_is_kept_per_device(tmp_path):
    """PerDevice: a device that has not been set up is, one that has been is not, a larger amount is granted again, a failure
    is not remembered, and threads that ask together are granted once and for the largest amount."""
    source = r"""#include "per_device.h"
    #include <cstdio>
    #include <thread>
    #include <vector>
    int main() {
      static pic::PerDevice p;
      int calls = 0;
      auto ask = [&](int dev, int amount, int err) { return p.grant(dev, amount, [&] { ++calls; return err; }); };
      ask(0, 100, 0); ask(0, 100, 0); ask(0, 50, 0);
      std::printf("%d ", calls);
      ask(1, 100, 0);
      std::printf("%d ", calls);
      ask(0, 200, 0); ask(0, 150, 0);
      std::printf("%d ", calls);
      const int failed = ask(2, 10, 7), again = ask(2, 10, 0);
      std::printf("%d %d %d ", failed, again, calls);
      ask(-1, 10, 0); ask(-1, 10, 0); ask(1000, 10, 0);
      std::printf("%d\n", calls);
      static pic::PerDevice q, r;
      int sets = 0, last = 0;
      std::vector<std::thread> t;
      for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] { for (int i = 0; i < 2000; ++i)
          q.grant(3, 1 + (i + 250 * k) % 2000, [&] { ++sets; last = 1 + (i + 250 * k) % 2000; return 0; }); });
      for (auto& x : t) x.join();
      int asked = 0;
      auto make = [&] { return ++asked == 1 ? 0 : 5; };
      const int none = r.number(0, make), five = r.number(0, make), kept = r.number(0, make), other = r.number(1, make);
      std::printf("%d %d %d %d %d %d\n", last, none, five, kept, other, asked);
    }"""
    lines = run_cpp(tmp_path, source).splitlines()
    assert lines[0].split() == ["1", "2", "3", "7", "0", "5", "8"]
    # the last amount set is the largest asked for: none was lowered after it
    assert lines[1].split() == ["2000", "0", "5", "5", "5", "3"]


def test_launches_keep_no_state_of_one_device():
    """No launch remembers in a plain static what belongs to the device that was current."""
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            assert not re.search(r"^\s*static (bool|int|size_t|unsigned|long long) \w+\s*(\[\d+\]\s*)?=", text, flags=re.M), name

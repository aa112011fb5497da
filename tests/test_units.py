"""CPU tests of the kernels' work-unit arithmetic (csrc/units.cuh, plain C++ without a GPU compiler)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_07428_gb300", "csrc")


def run(tmp_path, body):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "units.cpp", tmp_path / "units"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "units.cuh"\nusing namespace rbs;\nint main() {\n' + body + "\nreturn 0;\n}\n")
    subprocess.run([gxx, "-std=c++17", "-Wall", "-x", "c++", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("per_item", [1, 2, 3, 4, 16])
def test_counter_at_the_largest_launches(tmp_path, per_item):
    # the last units of launches around 2^31 units and of the largest one, then one more per resident warp: each of those
    # is past the end, none is one of the first units again
    out = run(tmp_path, f"""
  bool ok = !units_fit(kMaxUnits + 1) && !units_fit(4LL << 31);
  for (long long n : {{2147483647LL, 2147483648LL, 2147483653LL, kMaxUnits}}) {{
    ok = ok && units_fit(n);
    const unit_t nunits = (unit_t)n;
    unit_t counter = nunits - 5;
    for (int warp = 0; warp < 152 * 64; ++warp) {{
      const unit_t unit = counter++;
      if (warp < 5) {{
        const UnitPart u = unit_part(unit, {per_item});
        ok = ok && unit < nunits && u.part >= 0 && u.part < {per_item} && (long long)u.item * {per_item} + u.part == (long long)unit;
      }} else {{
        ok = ok && unit >= nunits;
      }}
    }}
  }}
  std::printf("%d\\n", (int)ok);""")
    assert out == ["1"]

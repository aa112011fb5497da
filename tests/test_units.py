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


def near_units(tmp_path, pairs, sm_count, one_part=0):
    targets, sources = (", ".join(str(p[k]) for p in pairs) for k in (0, 1))
    out = run(tmp_path, f"""
  for (const NearUnitItem& u : list_near_units({{{targets}}}, {{{sources}}}, {sm_count}, {one_part}))
    std::printf("%d %d %d %d ", u.pair, u.t, u.part, u.parts);""")
    v = [int(w) for w in out]
    return [tuple(v[k:k + 4]) for k in range(0, len(v), 4)]


@pytest.mark.parametrize("one_part", [0, 1])
@pytest.mark.parametrize("pairs,sm_count", [
    ([(144, 688)] * 12, 152),                                # a short list: runs of 128 sources
    ([(144, 688)] * 2000, 152),                              # a long one: as few runs as 512 sources allow
    ([(2112, 260)] + [(40, 20680)] + [(40, 260)] * 400, 152),  # one p = 32 particle among small ones
    ([(12, 52), (33, 127), (32, 128), (1, 1)], 4)])
def test_near_units_cover_each_pair_once(tmp_path, pairs, sm_count, one_part):
    units = near_units(tmp_path, pairs, sm_count, one_part)
    want = []
    for k, (nt, ns) in enumerate(pairs):
        parts = {u[3] for u in units if u[0] == k}
        assert len(parts) == 1
        p = parts.pop()
        assert p == 1 if one_part else (ns + 511) // 512 <= p <= max(ns // 128, (ns + 511) // 512)
        want += [(k, t, q, p) for t in range(0, nt, 32) for q in range(p)]
    assert units == want  # in order, none empty and none twice

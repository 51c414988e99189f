"""Host rules of the library that need no GPU, compiled from their headers."""
import subprocess

import pytest

from paper_2505_23970_gb300 import build as gbuild

INT_MAX = 2**31 - 1


def compile_and_run(tmp_path, program, *args):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(program)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", gbuild.CSRC, str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    return r.stdout.split()


# (requests x kv heads, capacity of a block table): calls whose 128-key tiles can be
# numbered, from small ones to the last that can
CALLS = [(8, 9216), (512, 131072), (2048, 2**24), (2048, 2**24 - 4096), (65536, 32767 * 128),
         (65536, 32765 * 128), (65536, 32763 * 128), (1, INT_MAX // 128 * 128), (3, 16),
         (8192 * 64, 4094 * 128)]


@pytest.mark.parametrize("pairs,cap", CALLS)
def test_decode_units_can_be_counted(tmp_path, pairs, cap):
    """Every pair's units, the allowance in front of its keys included, sum up in
    32 bits with the margin for the kernel's rounding."""
    margin = 448
    tiles = -(-cap // 128)
    assert pairs * tiles + margin <= INT_MAX  # what the call itself accepts
    shift, lead = map(int, compile_and_run(tmp_path, """
#include "decode_units.h"
#include <cstdio>
#include <cstdlib>
int main(int, char** v) {
  const auto u = gc::decode_units(atoll(v[1]), atoll(v[2]), atoll(v[3]));
  printf("%d %d", u.shift, u.lead);
}""", pairs, cap, margin))
    units = ((cap - 1) >> shift) + 1
    assert pairs * (units + lead) + margin <= INT_MAX
    # the finest units that fit, with the allowance wherever it fits
    if pairs * (-(-cap // 16) + 16) + margin <= INT_MAX:
        assert (shift, lead) == (4, 16)
    else:
        assert (shift, lead) == (7, 2 if pairs * (tiles + 2) + margin <= INT_MAX else 0)

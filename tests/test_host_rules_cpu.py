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


SHARED = r"""
#include "shared_by_context.h"
#include <cassert>
#include <cstdio>
#include <vector>

// handles made and destroyed, by contexts that can go and take theirs with them
char values[8];
std::vector<char*> destroyed;
gc::ContextId alive_context;
gc::SharedByContext<char*> shared;

char* acquire(gc::ContextId c, char* made, int device = 0) {
  return shared.acquire(device, c, [=] { return made; });
}
void release(gc::ContextId c, char* h, int device = 0) {
  shared.release(device, c, h, [=] { return c == alive_context; },
                 [](char* x) { destroyed.push_back(x); });
}

int main() {
  char *a = values, *b = values + 1;
  // two users of one context: one handle, destroyed with the last
  alive_context = 1;
  assert(acquire(1, a) == a && acquire(1, b) == a);
  release(1, a);
  assert(destroyed.empty());
  release(1, a);
  assert(destroyed.size() == 1 && destroyed[0] == a);
  // a reset before the last user gives its handle back: nothing to destroy
  assert(acquire(1, a) == a);
  alive_context = 2;
  release(1, a);
  assert(destroyed.size() == 1);
  // ... and the new context's handle has the old one's value: the old users do not
  // count as its users
  alive_context = 3;
  assert(acquire(3, a) == a && acquire(3, b) == a);
  alive_context = 4;
  assert(acquire(4, a) == a);
  release(3, a);
  release(3, a);
  assert(destroyed.size() == 1);
  assert(acquire(4, b) == a);
  release(4, a);
  assert(destroyed.size() == 1);
  release(4, a);
  assert(destroyed.size() == 2);
  // another device, no context, nothing made, more places than there are
  alive_context = 5;
  assert(acquire(5, a) == a && acquire(5, b, 1) == b);
  release(5, b, 1);
  release(5, a);
  assert(destroyed.size() == 4);
  assert(acquire(0, a) == nullptr && acquire(5, nullptr) == nullptr);
  release(5, nullptr);
  for (int c = 10; c < 74; ++c) assert(acquire(c, a) == a);
  assert(acquire(99, a) == nullptr);
  release(10, a);
  assert(acquire(99, a) == a);
  puts("ok");
}
"""


def test_what_a_context_shares(tmp_path):
    """The scratch allocator of the pools of a device and context: made once,
    destroyed with its last user, and only forgotten when a device reset took it,
    also where the next context's has the same handle value."""
    assert compile_and_run(tmp_path, SHARED) == ["ok"]

"""Kept tensor maps are found by everything they were encoded from, never by a hash of it."""
import os
import subprocess

from paper_2608_01651_b200.build import CSRC

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include <cstring>
#include "tv_map_cache.h"
using namespace tvtc;

static long made = 0;
static bool fails = false;   // of the encode
// a set of maps that says what it was made from
static void stamp(CUtensorMap* m, const MapKey& k) {
  std::memcpy(&m[0], &k.view[0], sizeof(NodeView));
  std::memcpy(&m[1], &k.view[1], sizeof(NodeView));
  std::memcpy(&m[2], &k.items, sizeof(k.items));
  std::memcpy(&m[3], k.ptr, sizeof(k.ptr));
}
static bool serves(const MapKey& k) {
  const MapSet* s = cached_maps(k, [&](CUtensorMap* m) { stamp(m, k); ++made; return !fails; });
  CUtensorMap want[5];
  std::memset(want, 0, sizeof(want));
  stamp(want, k);
  return s && !std::memcmp(&s->map[0], &want[0], sizeof(NodeView)) && !std::memcmp(&s->map[1], &want[1], sizeof(NodeView)) &&
         !std::memcmp(&s->map[2], &want[2], sizeof(k.items)) && !std::memcmp(&s->map[3], &want[3], sizeof(k.ptr));
}
static NodeView view(uint64_t heads, uint64_t T, uint64_t Z, bool token) {
  const int64_t d = 128;
  return token ? NodeView{128, T, heads, Z, (int64_t)(T * heads) * d, d, (int64_t)heads * d}
               : NodeView{128, T, heads, Z, (int64_t)(T * heads) * d, (int64_t)T * d, d};
}

int main() {
  char mem[8];
  long bad = 0, calls = 0;
  const int Ts[] = {15, 24, 63, 64, 128};
  for (int H = 1; H <= 32; ++H)
    for (int G = 1; G <= 4; G *= 2) {
      if (H % G) continue;
      for (int T : Ts)
        for (int token = 0; token < 2; ++token)
          for (uint64_t z = 1; z <= 8; ++z)      // batches that share the buffers of a larger one
            for (uint64_t step = 1; step <= 256; step *= 2)
              for (int out = 0; out < 2; ++out)
                for (uint64_t Z : {z, z + step - 1, z + step}) {
                  MapKey k{{mem, mem + 1, mem + 2, mem + 3}, {view(H / G, T, Z, token), view(H, T, Z, token)}, H * Z, T, 9};
                  if (out) k.view[2] = k.view[1];
                  bad += !serves(k);
                  ++calls;
                }
    }
  // found again, in the order of use; one field away is another set
  MapKey k{{mem, mem + 1, mem + 2, mem + 3, mem + 4}, {view(8, 64, 4, 0), view(8, 64, 4, 0), view(8, 64, 4, 1)}, 32, 64, 0};
  bad += !serves(k);
  long before = made;
  for (int i = 0; i < 3; ++i) bad += !serves(k);
  if (made != before) bad += 1000;
  for (int i = 0; i < 5; ++i) { MapKey x = k; x.ptr[i] = mem + 7; before = made; bad += !serves(x) + 1000 * (made != before + 1); }
  { MapKey x = k; x.view[2].st += 8; before = made; bad += !serves(x) + 1000 * (made != before + 1); }
  { MapKey x = k; x.T = 63; before = made; bad += !serves(x) + 1000 * (made != before + 1); }
  { MapKey x = k; x.kind = 4; before = made; bad += !serves(x) + 1000 * (made != before + 1); }
  // an encode that fails is not kept
  MapKey f = k;
  f.kind = 77;
  fails = true;
  for (int i = 0; i < 2; ++i) { before = made; bad += serves(f) + 1000 * (made != before + 1); }
  fails = false;
  before = made;
  bad += !serves(f) + 1000 * (made != before + 1) + !serves(k);
  std::printf("%ld lookups, %ld bad\n", calls, bad);
  return bad != 0;
}
"""


def test_lookup_serves_what_was_asked_for(tmp_path):
    src, exe = tmp_path / "maps.cpp", tmp_path / "maps"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

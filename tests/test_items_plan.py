"""The plan of the perturbation passes (zo_items.h): which thread changes which
element with which sign, computed on the host from the tables that the kernel
gets (the kernel places its threads with the same item_place), over random
lists of every type, alignment and size, with entries and launches short
enough that tensors are split over both. Every element is changed exactly
once, with the byte of the virtual block that belongs to it."""
import os
import shutil
import subprocess

import pytest

from paper_2609_38095_gb300 import build as zo_build

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "zo_items.h"
using namespace zo;
static int fail(const char* what, int round, int t, long long e) {
  std::printf("round %d tensor %d element %lld: %s\n", round, t, e, what);
  return 1;
}
template <int N> int check(int round, std::mt19937& g) {
  auto pick = [&](long long n) { return static_cast<long long>(g() % static_cast<unsigned long long>(n)); };
  const int n = 1 + pick(round % 7 == 0 ? 3 * N : 12);
  std::vector<zo_tensor> list(n);
  std::vector<long long> first(n);           // virtual index of element 0
  std::vector<std::vector<int>> hits(n);
  long long v = round % 3 == 0 ? 0 : pick(1 << 20);
  for (int t = 0; t < n; ++t) {
    const int dt = pick(3);
    const long long esz = dt == ZO_F32 ? 4 : 2;
    const long long numel = pick(8) == 0 ? 0 : pick(4) == 0 ? 1 + pick(40) : 1 + pick(3000);
    const long long off = pick(2) ? 0 : esz * pick(32 / esz);
    list[t] = {reinterpret_cast<void*>((t + 1) * 1048576ll + off), numel, dt, 1};
    hits[t].assign(numel, 0);
  }
  ItemsCursor cur;
  cur.v = v;
  for (int t = 0; t < n; ++t) { first[t] = 16 * v; v += (list[t].numel + 15) / 16; }
  const long long piece = round % 2 ? 2 * (16 + pick(200)) : kItemsPiece;
  const long long launch = round % 2 ? 64 + 2 * piece + pick(5000) : kItemsLaunch;
  static ItemsParams<N> ip;
  while (cur.t < n) {
    const bool one = fill_items(ip, list.data(), n, cur, [](auto&, int32_t, int64_t) {}, piece, launch);
    if (!one) return fail("high word", round, cur.t, 0);
    if (ip.n == 0) { if (cur.t < n) return fail("nothing taken", round, cur.t, 0); break; }
    std::vector<ItemPlace> place(ip.total + 32);
    std::vector<int> entry(ip.total + 32);
    for (uint32_t wb = 0; wb < ip.total; wb += 32) {
      int t = ip.hint[wb >> ip.hint_shift];
      if (t > 0 && ip.e[t - 1].end > wb) return fail("hint past its tensor", round, t, wb);
      while (wb >= ip.e[t].end) ++t;
      for (uint32_t lane = 0; lane < 32; ++lane) { place[wb + lane] = item_place(ip.e[t], wb + lane); entry[wb + lane] = t; }
    }
    for (uint32_t b = 0; b < (ip.total + 31) / 32 * 32; ++b) {
      const ItemPlace& k = place[b];
      const ItemsEntry& e = ip.e[entry[b]];
      if (!k.act) continue;
      const uint64_t at = e.base + 32 * k.i;
      const int t = static_cast<int>(at / 1048576) - 1;
      const bool f32 = (e.meta & kDtypeMask) == kF32, shift = (e.meta & kShift) != 0;
      const long long esz = f32 ? 4 : 2, per = 32 / esz, a = e.meta >> 16;
      if (list[t].dtype != static_cast<int>(e.meta & kDtypeMask)) return fail("type", round, t, b);
      int lo, hi;
      item_range(e, k.i, &lo, &hi);
      if (k.full != (lo == 0 && hi == per)) return fail("full", round, t, b);
      for (int j = lo; j < hi; ++j) {
        const long long el = static_cast<long long>(at + esz * j - reinterpret_cast<uint64_t>(list[t].ptr)) / esz;
        if (el < 0 || el >= list[t].numel) return fail("outside", round, t, el);
        ++hits[t][el];
        // element j of the chunk: byte j - a of the lane's block (half block), or of the one below (lane - 1)
        long long pos = j - (shift ? a : 0);
        int32_t from = k.i;
        if (pos < 0) {
          if (!shift || b % 32 == 0) return fail("no lane below", round, t, el);
          from = place[b - 1].i;
          pos += per;
        }
        const long long index = 16 * item_block(e, from) + (f32 && (from & 1) ? 8 : 0) + pos;
        if (index != first[t] + el) return fail("sign of another element", round, t, el);
      }
    }
  }
  for (int t = 0; t < n; ++t)
    for (size_t e = 0; e < hits[t].size(); ++e)
      if (hits[t][e] != 1) return fail("not changed exactly once", round, t, static_cast<long long>(e));
  return 0;
}
// Lists past 2^32 blocks: a launch that fill_items calls one of a single counter high word uses no block of another,
// in the first and the last warp of each entry.
static int check_high_words(const std::vector<long long>& blocks, const std::vector<int>& offsets) {
  static ItemsParams<kItemsMany> ip;
  const int n = static_cast<int>(blocks.size());
  std::vector<zo_tensor> list(n);
  for (int t = 0; t < n; ++t)
    list[t] = {reinterpret_cast<void*>((t + 1) * (1ll << 44) + 2 * offsets[t]), 16 * blocks[t], ZO_BF16, 1};
  ItemsCursor cur;
  for (int l = 0; cur.t < n; ++l) {
    if (!fill_items(ip, list.data(), n, cur, [](auto&, int32_t, int64_t) {})) continue;
    const int64_t high = ip.e[0].vb >> 32;
    for (int t = 0; t < ip.n; ++t) {
      const ItemsEntry& e = ip.e[t];
      for (uint32_t wb : {e.begin, e.begin + (e.end - 1 - e.begin) / 32 * 32})
        for (uint32_t b = wb; b < wb + 32 && b < e.end; ++b) {
          const ItemPlace k = item_place(e, b);
          if (!k.act) continue;
          int lo, hi;
          item_range(e, k.i, &lo, &hi);
          const int a = static_cast<int>(e.meta >> 16);
          if (hi > a && item_block(e, k.i) >> 32 != high) return fail("high word", l, t, b);
          if (lo < a && item_block(e, item_place(e, b - 1).i) >> 32 != high) return fail("high word below", l, t, b);
        }
    }
  }
  return 0;
}
int main() {
  std::mt19937 g(12345);
  const long long b30 = 1ll << 30;
  for (int off : {0, 1, 9}) {
    if (check_high_words({b30, b30, b30, 2 * b30 - 100}, {0, 0, 0, off})) return 1;
    if (check_high_words({b30, b30, b30 - 5, 2 * b30 - 100}, {0, 0, 0, off})) return 1;
    if (check_high_words({2 * b30 - 1, 2 * b30 - 1, 2, 700}, {off, off, off, off})) return 1;
  }
  for (int r = 0; r < 600; ++r)
    if (check<kItemsFew>(r, g)) return 1;
  for (int r = 0; r < 20; ++r)
    if (check<kItemsMany>(7 * r, g)) return 1;
  std::printf("ok\n");
  return 0;
}
"""


def test_every_element_once_with_its_own_sign(tmp_path):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not found")
    src = tmp_path / "plan.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "plan"
    subprocess.run([zo_build.nvcc(), "-std=c++17", "-O1", *zo_build.ARCH, "-I", zo_build.INCLUDE, "-I", zo_build.CSRC,
                    "-o", str(exe), str(src)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout

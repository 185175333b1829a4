// zo_items.h -- host-side planning of the tables of the launches by items
// (perturb_items_kernel, pair_items_kernel, update_items_kernel).
#pragma once

#include <cstdint>

#include "zo.h"
#include "zo_device.cuh"

namespace zo {

// A position in a parameter list: the next tensor, how many of its items are
// already in earlier entries, and the virtual block of its first element.
struct ItemsCursor {
  int32_t t = 0;
  int64_t done = 0;
  int64_t v = 0;
};

// log2 of a storage type's bytes (a division by a variable costs a long list's
// call more than the rest of its loop).
inline int size_shift(int32_t dtype) { return dtype == ZO_F32 ? 2 : 1; }

// Items of a tensor in a launch's numbering, up to the next tensor's start.
inline int64_t tensor_items(const zo_tensor& p) {
  if (p.numel == 0) return 0;
  const int sh = size_shift(p.dtype);
  const int64_t off = static_cast<int64_t>(reinterpret_cast<uintptr_t>(p.ptr) % 32) >> sh;
  const int64_t items = (p.numel + off + (32 >> sh) - 1) >> (5 - sh);
  return off == 0 ? (items + kLaunchAlign - 1) / kLaunchAlign * kLaunchAlign
                  : (items + kShiftLanes - 1) / kShiftLanes * kLaunchAlign;
}

// Most items of one entry (an even number, so that a later piece of an fp32
// tensor starts with a whole block) and of one launch. A longer tensor takes
// several entries.
constexpr int64_t kItemsPiece = INT64_C(1) << 30;
constexpr int64_t kItemsLaunch = INT64_C(1) << 31;

// Fill `ip` (ItemsParams, PairItemsParams) from `cur` on, as far as its entries
// and `launch` items go; more(entry, tensor, bytes) sets what an entry has
// besides, `bytes` being the entry's base minus the tensor's address. Returns
// whether the launch's virtual blocks share the counter's high word.
template <class Params, class More>
bool fill_items(Params& ip, const zo_tensor* params, int32_t n, ItemsCursor& cur, const More& more,
                int64_t piece = kItemsPiece, int64_t launch = kItemsLaunch) {
  constexpr int N = Params::kEntries;
  ip.n = 0;
  int64_t b = 0, last = 0;  // items so far, and the last virtual block
  while (cur.t < n) {
    const zo_tensor& p = params[cur.t];
    if (p.numel == 0) {
      ++cur.t;
      continue;
    }
    if (ip.n == N) break;
    const int sh = size_shift(p.dtype);
    const uintptr_t addr = reinterpret_cast<uintptr_t>(p.ptr);
    const int64_t off = static_cast<int64_t>(addr % 32) >> sh;
    const int64_t whole = (p.numel + off) >> (5 - sh), rem = (p.numel + off) & ((32 >> sh) - 1);
    const int64_t items = whole + (rem != 0);
    const int64_t left = items - cur.done, take = left < piece ? left : piece;
    const int64_t start = (b + kLaunchAlign - 1) / kLaunchAlign * kLaunchAlign;
    const int64_t end = start + (off == 0 ? take : (take + kShiftLanes - 1) / kShiftLanes * kLaunchAlign);
    if (ip.n > 0 && end > launch) break;
    b = end;
    auto& e = ip.e[ip.n++];
    e.base = static_cast<uint64_t>(addr - addr % 32) + static_cast<uint64_t>(32 * cur.done);
    e.vb = cur.v + (p.dtype == ZO_F32 ? cur.done / 2 : cur.done);
    e.begin = static_cast<uint32_t>(start);
    e.end = static_cast<uint32_t>(end);
    e.whole = static_cast<uint32_t>(whole - cur.done < take ? whole - cur.done : take);
    e.meta = static_cast<uint32_t>(p.dtype) | (off == 0 ? 0u : static_cast<uint32_t>(kShift)) |
             (cur.done == 0 ? 0u : kItemsCont) | static_cast<uint32_t>(take == left ? rem : 0) << 8 |
             static_cast<uint32_t>(off) << 16;
    more(e, cur.t, static_cast<int64_t>(e.base - static_cast<uint64_t>(addr)));
    last = e.vb + take;
    cur.done += take;
    if (cur.done == items) {
      ++cur.t;
      cur.done = 0;
      cur.v += (p.numel + 15) / 16;
    }
  }
  ip.total = static_cast<uint32_t>(b);
  if (ip.n == 0) return true;
  // hint[k]: the first entry that ends past item k << hint_shift
  ip.hint_shift = 5;
  while ((ip.total - 1) >> ip.hint_shift >= static_cast<uint32_t>(kItemsHints)) ++ip.hint_shift;
  int t = 0;
  for (uint32_t k = 0; k <= (ip.total - 1) >> ip.hint_shift; ++k) {
    while (static_cast<uint64_t>(ip.e[t].end) <= static_cast<uint64_t>(k) << ip.hint_shift) ++t;
    ip.hint[k] = static_cast<uint16_t>(t);
  }
  // the first block: of a later piece off the grid, the one below, whose tail is the piece's first elements
  const bool below = (ip.e[0].meta & kItemsCont) && (ip.e[0].meta & kShift);
  return (ip.e[0].vb - (below ? 1 : 0)) >> 32 == last >> 32;
}

}  // namespace zo

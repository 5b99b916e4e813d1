// Row order of the sliced storage (host, standard library only).
#pragma once

#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

namespace bamg {

// Rows per slice of the sliced block storage: one warp, one row per lane.
constexpr int kSlice = 32;

// Row orders: identity, rows sorted by decreasing length within windows of 1,024
// rows, the slices then by decreasing width; or sorted only where that removes
// at least a tenth of the stored slots.
constexpr int kSortNever = 0, kSortAlways = 1, kSortAuto = 2;

struct Placement {
  std::vector<int> order;  // block row of each of the 32 * nslices row positions, -1 at the padding positions
  bool sorted = false;     // order is not the identity
};

// The padding positions are the last ones in every order, so positions
// 0 .. nbr - 1 hold every row once: the multi-vector kernels run over these
// alone.
inline Placement place_rows(const std::vector<int>& rowptr, int64_t nbr, int sort_rows) {
  const int64_t nslices = (nbr + kSlice - 1) / kSlice;
  Placement p;
  p.order.resize((size_t)(nslices * kSlice));
  for (size_t r = 0; r < p.order.size(); ++r) p.order[r] = (int64_t)r < nbr ? (int)r : -1;
  if (sort_rows == kSortNever) return p;
  auto len = [&](int i) { return i < 0 ? -1 : rowptr[i + 1] - rowptr[i]; };
  auto stored_chunks = [&](const std::vector<int>& ord) {
    int64_t c = 0;
    for (int64_t s = 0; s < nslices; ++s) {
      int w = 0;
      for (int64_t r = s * kSlice; r < (s + 1) * kSlice; ++r) w = std::max(w, len(ord[r]));
      c += w;
    }
    return c;
  };
  std::vector<int> sorted = p.order;
  constexpr size_t kWindow = 1024;
  for (size_t w0 = 0; w0 < sorted.size(); w0 += kWindow) {
    const size_t w1 = std::min(sorted.size(), w0 + kWindow);
    std::stable_sort(sorted.begin() + w0, sorted.begin() + w1, [&](int a, int b) { return len(a) > len(b); });
  }
  // auto: only where the sort removes a tenth of the stored slots or more
  // (rows of very uneven length, e.g. Q2 vertex and mid-edge nodes); evenly
  // filled slices keep the identity order and its contiguous vectors
  if (sort_rows != kSortAlways && 10 * stored_chunks(sorted) > 9 * stored_chunks(p.order)) return p;
  // Slices in order of decreasing width over the whole matrix.  CTAs go to
  // the SMs in turn, and with the windows one after another (32 slices
  // each, wide to narrow) an SM's CTAs came from the same few places of
  // every window: its work was up to 1.3 times another's, with about one
  // wave of CTAs nothing evened that out, and a wide slice could come last
  // (21^3 Q2 elements: SMs busy 62,000 to 100,000 cycles).  Wide to narrow,
  // each SM gets a like share of every width: FP32 product 50.7 to 47.1 us,
  // FP64 84.6 to 74.4, a whole 16^3 Q2 step 17.5 to 15.3 ms; the assembly
  // gains too (345 to 322 us).  A row's sum does not depend on its place.
  // A partly filled slice (the last one of the last window) stays last whatever
  // its width, with its padding.
  std::vector<int64_t> by((size_t)nslices);
  for (size_t q = 0; q < by.size(); ++q) by[q] = (int64_t)q;
  auto width = [&](int64_t q) { return len(sorted[(size_t)q * kSlice]); };
  std::stable_sort(by.begin(), by.begin() + nbr / kSlice, [&](int64_t a, int64_t b) { return width(a) > width(b); });
  for (size_t q = 0; q < by.size(); ++q)
    std::copy_n(sorted.begin() + by[q] * kSlice, kSlice, p.order.begin() + q * kSlice);
  p.sorted = true;
  return p;
}

}  // namespace bamg

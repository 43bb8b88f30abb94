// Balanced tile lists for the persistent tensor-core kernels, and the choice of kernel
// for calls of few tokens (host code only).
#include "gs_plan.cuh"

#include <algorithm>
#include <utility>

namespace gs {

void plan_tiles(const std::vector<int32_t>& cost, int n_owners, TileList& L) {
  const int n = (int)cost.size();
  L.on = 0;
  if (n > kTileListMax || n_owners > kTileOwnersMax || n_owners <= 0) return;
  std::vector<int> idx(n);
  for (int i = 0; i < n; ++i) idx[i] = i;
  std::stable_sort(idx.begin(), idx.end(), [&](int a, int b) { return cost[a] > cost[b]; });
  // min-heap of (load, owner)
  std::vector<std::pair<int64_t, int>> heap;
  heap.reserve(n_owners);
  for (int b = 0; b < n_owners; ++b) heap.emplace_back(0, b);
  auto later = [](const std::pair<int64_t, int>& x, const std::pair<int64_t, int>& y) { return x > y; };
  std::vector<int> owner(n);
  std::vector<int> count(n_owners + 1, 0);
  for (int t : idx) {
    std::pop_heap(heap.begin(), heap.end(), later);
    auto& h = heap.back();
    owner[t] = h.second;
    h.first += cost[t];
    std::push_heap(heap.begin(), heap.end(), later);
    ++count[owner[t] + 1];
  }
  for (int b = 0; b < n_owners; ++b) count[b + 1] += count[b];
  for (int b = 0; b <= n_owners; ++b) L.off[b] = (uint16_t)count[b];
  // each owner's tiles longest first (the order they were handed out)
  for (int t : idx) L.order[count[owner[t]]++] = (uint16_t)t;
  L.on = 1;
}

// The lines below are fitted to both kernels' times, eager and as graph replays with
// weights past L2, over 54 sets of 1 to 32 layers (16.8 M to 537 M weights, 1 x 128 and
// 1 x 256), kept fractions of 0.05 to 1 and 1 to 16 tokens: 3930 points.  The choice made
// here is more than 4 % behind the decode kernel at 1 % of them and 0.5 % behind the better
// kernel on average (eager calls); a line at 20 M weights in all (250 M for batches at two
// tokens) was behind the decode kernel at 14 % and 3.7 % behind the better one.  us a call,
// decode kernel against zero-filled one:
//  - below 20 M weights both take 6 to 11 us: 4096 x 4096 at T = 4 8 / 9;
//  - one launch of either.  While all of the decode kernel's units are resident at once it
//    is ahead up to eight tokens (1024 x 20480 at d = 0.1: 8.4 / 10.1 at T = 1, 9.9 / 10.9 at
//    T = 8, 14.0 / 11.6 at T = 16); from the second wave on it is not (5120 x 5120 at d = 0.1:
//    10.5 / 9.3, 12.6 / 9.7, 17.6 / 10.3; 7B block at d = 0.2, T = 1: 47 / 29);
//  - batches of layers so small that the host sets the pace: a zero-filled launch is
//    prepared 3 to 5 us later (eight layers of 1024 x 4096 at T = 8 16 / 22, eight of
//    2048 x 2048 20 / 18, seven of a 60 M block 25 / 18);
//  - at one or two tokens, 1 x 256 batches whose weights stream as fast on either stay on
//    the decode kernel (7B block at d = 0.5: 38.8 / 39.1) up to 250 M weights (13B block
//    61 / 56);
//  - more than eight layers: each further zero-filled launch adds its start, its own
//    ragged end and 7 us on the host, so both times are estimated (32 layers of
//    1024 x 1024 at T = 8 54 / 68, 9 of 2048 x 2048 at T = 1 19 / 29, two 7B blocks with
//    1 x 128 groups 115 / 81).
bool zero_filled_first(const std::vector<FewTokenLayer>& layers, int kw, int T, int sms) {
  const int n = (int)layers.size();
  const double ctas = 2.0 * sms, pairs = std::max(1.0, sms / 2.0);
  // the decode kernel's units, as it makes them, and their 64-row chunk steps
  double weights = 0.0, kept = 0.0, steps = 0.0, units = 0.0, fine = 0.0;
  int longest = 0, longest_fine = 0;   // chunks of the longest unit
  for (const FewTokenLayer& L : layers) {
    const double blocks = (double)((L.out + 63) / 64);
    weights += (double)L.out * (double)L.in;
    kept += L.kept_bytes;
    steps += blocks * L.chunks;
    units += blocks * ((L.chunks + L.cpu - 1) / L.cpu);
    fine += blocks * ((L.chunks + L.cpu_fine - 1) / L.cpu_fine);
    longest = std::max(longest, L.cpu);
    longest_fine = std::max(longest_fine, L.cpu_fine);
  }
  if (units < 2.0 * ctas) {
    units = fine;
    longest = longest_fine;
  }
  if (weights < 20e6) return false;
  // us of the decode kernel's walk over its chunks, with the end of its longest unit, and
  // of its stream of kept weights (tokens take their share of the copies)
  const bool wide = kw == 256;
  const double walk = units / ctas * (1.8 + 0.22 * T) + steps / ctas * (wide ? 0.42 : 0.465) + 0.3 * longest;
  const double stream = kept / (6.9e6 - 0.11e6 * T);
  if (n <= 8) {
    if (units <= ctas && T <= 8) return false;
    if (n > 1) {
      const double work = (steps + 3.0 * units) / ctas;   // per resident CTA; a unit costs what three chunks do
      if (work < n * (T <= 2 ? 4.0 : T <= 8 ? 2.0 : 1.6)) return false;
      if (T <= 2 && wide && weights < 250e6 && stream >= walk) return false;
    }
    return true;
  }
  const auto both = [](double a, double b) { return std::max(a, b) + 0.2 * std::min(a, b); };
  const double decode = std::max((wide ? 3.6 : 1.8) + both(walk, stream), 3.2 + 1.6 * n);
  // launches of eight layers, widest input first: 256-column items of the busiest CTA pair
  std::vector<FewTokenLayer> by_width(layers);
  std::stable_sort(by_width.begin(), by_width.end(),
                   [](const FewTokenLayer& a, const FewTokenLayer& b) { return a.in > b.in; });
  double zero_filled = 0.7 + 0.05 * T;
  for (int b = 0; b < n; b += 8) {
    double total = 0.0, widest = 0.0, bytes = 0.0;
    for (int k = b; k < std::min(n, b + 8); ++k) {
      const double items = (double)((by_width[k].in + 255) / 256);
      total += items * (double)((by_width[k].out + 255) / 256);
      widest = std::max(widest, items);
      bytes += by_width[k].kept_bytes;
    }
    zero_filled += 4.7 + both((wide ? 0.47 : 0.55) * std::max(widest, total / pairs), bytes / (wide ? 6.7e6 : 6.3e6));
  }
  zero_filled = std::max(zero_filled, 7.0 * ((n + 7) / 8) + 1.5 * n);
  return zero_filled < 0.97 * decode;
}

}  // namespace gs

// Every entry that row_walk hands out, against the rows' definition: the CSR
// position, item and payload of entry x of the list, and the place of a lane's
// window item in the batch.  Rows too long to hold in memory are walked by a few
// warps of many, whose chunks lie all over the list.
#include <cstdio>
#include <atomic>
#include <thread>
#include <vector>

#include "cc_device.cuh"

using namespace ccg;

namespace {

struct List {
  std::vector<int64_t> pos, row;
  std::vector<int32_t> len;
  int64_t E = 0;
  void add(int32_t n) {
    pos.push_back(E);
    row.push_back(E + 17 * (int64_t)pos.size() + 5);       // gaps between the rows
    len.push_back(n);
    E += n;
  }
};

std::atomic<long long> wrong{0}, seen{0};

template <int kB>
void walk(const List& L, int gwarp, int nwarps) {
  std::vector<std::thread> lanes;
  for (unsigned lane = 0; lane < 32; ++lane)
    lanes.emplace_back([&, lane] {
      threadIdx.x = lane;
      const int32_t n = (int32_t)L.pos.size();
      long long bad = 0, got = 0;
      row_walk<kB>(gwarp, nwarps, n, L.E, host_warp::columns, WalkShape{},
                   [&](int32_t j) { return L.pos[(size_t)j]; },
                   [&](int32_t j) { return RowItem{L.pos[(size_t)j], L.row[(size_t)j], L.len[(size_t)j], 3 * j + 1}; },
                   [&](const RowBatch<kB>& X) {
                     int32_t counted = 0;                  // entries of this lane's window item in the batch
                     if (X.from < 32 * kB) counted = X.to - (X.from > 0 ? X.from : 0);
                     int32_t mine[kB];
                     for (int q = 0; q < kB; ++q) mine[q] = X.w[q] >= 0 ? X.item[q] : -1;
                     const int32_t j0 = __shfl_sync(FULL, X.w[0] >= 0 ? X.item[0] : -1, 0);
                     if (j0 < 0) ++bad;                    // a batch has at least one entry
                     int32_t total = counted > 0 ? counted : 0;
                     for (int q = 0; q < kB; ++q) {
                       if (X.w[q] < 0) continue;
                       ++got;
                       const int32_t j = X.item[q];
                       if (j < 0 || j >= n || X.aux[q] != 3 * j + 1) { ++bad; continue; }
                       // the position names an entry of row j
                       const int64_t k = (X.w[q] - L.row[(size_t)j]) & 0x7FFFFFFF;
                       if (k >= L.len[(size_t)j]) ++bad;
                     }
                     // the items' shares of the batch add up to its entries
                     int32_t entries = 0;
                     for (int q = 0; q < kB; ++q) entries += X.w[q] >= 0 ? 1 : 0;
                     if (__reduce_add_sync(FULL, entries) != __reduce_add_sync(FULL, total)) ++bad;
                     // neighbouring lanes hold neighbouring entries of a row
                     for (int q = 0; q < kB; ++q) {
                       const int32_t w = __shfl_up_sync(FULL, X.w[q], 1), it = __shfl_up_sync(FULL, mine[q], 1);
                       if (lane > 0 && mine[q] >= 0 && it == mine[q] && ((X.w[q] - w) & 0x7FFFFFFF) != 1) ++bad;
                     }
                   });
      wrong += bad;
      seen += got;
    });
  for (auto& t : lanes) t.join();
}

// Entries of the chunks of warp gwarp.
long long share(const List& L, int kB, int gwarp, int nwarps) {
  const int64_t kW = 32 * kB, most = (int64_t)nwarps * kW * 4 * kLbsBatches;
  int64_t nb = L.E >= most ? 2 * kLbsBatches : L.E / (nwarps * kW * 2);
  nb = nb < 1 ? 1 : nb;
  long long sum = 0;
  for (int64_t c = gwarp * nb * kW; c < L.E; c += nwarps * nb * kW) sum += L.E - c < nb * kW ? L.E - c : nb * kW;
  return sum;
}

int check(const char* name, const List& L, std::initializer_list<int> warps, int nwarps) {
  long long want = 0;
  wrong = seen = 0;
  for (int g : warps) {
    walk<4>(L, g, nwarps);
    walk<1>(L, g, nwarps);
    want += share(L, 4, g, nwarps) + share(L, 1, g, nwarps);
  }
  const bool ok = wrong == 0 && seen == want;
  std::printf("%s: %zu rows, %lld entries: %s (%lld of %lld seen, %lld wrong)\n", name, L.pos.size(), (long long)L.E,
              ok ? "ok" : "FAILED", (long long)seen, want, (long long)wrong);
  return ok ? 0 : 1;
}

}  // namespace

int main() {
  int bad = 0;
  List one, window, two, mixed, hubs32, hubs33, longest;
  one.add(1);
  for (int i = 0; i < 32; ++i) window.add(1 + i * 37 % 61);
  for (int i = 0; i < 33; ++i) two.add(1 + i * 37 % 61);
  for (int i = 0; i < 100; ++i) mixed.add(i % 50 == 7 ? 1000 : 1 + i * 7 % 5);
  // lists of more than 2^31 entries, of one window (walked from item 0 on) and of two
  for (int i = 0; i < 32; ++i) hubs32.add(140'000'003 - i);
  for (int i = 0; i < 33; ++i) hubs33.add(140'000'003 - i);
  longest.add(INT32_MAX - 1);
  longest.add(5);
  longest.add(INT32_MAX - 1);
  bad += check("one entry", one, {0, 1}, 2);
  bad += check("one window", window, {0, 1, 2}, 3);
  bad += check("two windows", two, {0, 1, 2}, 3);
  bad += check("mixed rows", mixed, {0, 1}, 2);
  const int many = 1 << 21;
  bad += check("32 hubs", hubs32, {1, many - 1}, many);
  bad += check("33 hubs", hubs33, {1, many - 1}, many);
  bad += check("longest rows", longest, {0}, 1 << 20);
  return bad;
}

// CopyQueue against copies made one after the other: the destinations of a
// random sequence overlap in part, wholly and not at all.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "lg_copies.h"

int main(int argc, char** argv) {
  const unsigned threads = argc > 1 ? (unsigned)atoi(argv[1]) : 4;
  std::mt19937_64 rng(threads + 7);
  constexpr size_t N = 1 << 20, K = 3000;
  std::vector<unsigned char> src(N + K), got(N), want(N);
  for (auto& x : src) x = (unsigned char)rng();
  std::vector<std::atomic<int>> done(K);
  for (auto& d : done) d = 0;
  {
    lg::CopyQueue q(threads, [&](uint64_t t) { done[t]++; });
    for (uint64_t t = 0; t < K; t++) {
      const size_t bytes = t % 50 == 0 ? 0 : t % 3 == 0 ? rng() % 300000 : rng() % 3000;
      const size_t at = t % 7 == 0 ? 4096 : rng() % (N - 300000), from = rng() % (N - 300000) + t;
      memcpy(want.data() + at, src.data() + from, bytes);
      q.push(got.data() + at, src.data() + from, bytes, t);
    }
  }
  for (uint64_t t = 0; t < K; t++)
    if (done[t] != 1) return printf("ticket %d done %d times\n", (int)t, (int)done[t]), 1;
  if (got != want) return printf("the copies differ from those in order\n"), 1;
  // a push waits for the copy that it overlaps, and for no other
  if (threads) {
    std::atomic<bool> first{false};
    lg::CopyQueue q(threads, [&](uint64_t t) {
      if (t) return;
      std::this_thread::sleep_for(std::chrono::milliseconds(500));
      first = true;
    });
    q.push(got.data(), src.data(), 1000, 0);
    q.push(got.data() + 1000, src.data(), 1000, 1);
    if (first) return printf("waited for another range\n"), 1;
    q.push(got.data() + 999, src.data(), 2, 2);
    if (!first) return printf("did not wait for its range\n"), 1;
  }
  printf("ok\n");
  return 0;
}

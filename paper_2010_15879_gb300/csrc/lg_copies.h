// Copies of results to the caller's buffers by a few helper threads.  Copies
// whose destinations overlap are made in the order in which they were pushed
// (a caller may give one buffer to several requests), all others in any order.
// Nothing here throws: what a thread or a list entry cannot be had for is
// copied by the caller of push().
#pragma once

#include <condition_variable>
#include <cstdint>
#include <cstring>
#include <exception>
#include <functional>
#include <iterator>
#include <list>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

namespace lg {

class CopyQueue {
 public:
  // done(ticket) follows each copy, on the thread that made it
  CopyQueue(unsigned threads, std::function<void(uint64_t)> done) : done_(std::move(done)) {
    try {
      threads_.reserve(threads);
      for (unsigned k = 0; k < threads; k++) threads_.emplace_back([this] { work(); });
    } catch (const std::exception&) {  // those there copy, or the caller
    }
  }
  // ends when everything is copied
  ~CopyQueue() {
    {
      std::lock_guard<std::mutex> l(mu_);
      end_ = true;
    }
    pushed_.notify_all();
    for (auto& t : threads_) t.join();
  }
  CopyQueue(const CopyQueue&) = delete;
  CopyQueue& operator=(const CopyQueue&) = delete;

  // One thread pushes.  Waits for earlier copies into any of the same bytes.
  void push(void* to, const void* from, uint64_t bytes, uint64_t ticket) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(to), b = a + bytes;
    {
      std::unique_lock<std::mutex> l(mu_);
      copied_.wait(l, [&] { return !overlaps(a, b); });
      if (bytes && !threads_.empty()) {
        try {
          const auto at = open_.emplace(a, b).first;
          try {
            queue_.push_back(Copy{to, from, bytes, ticket});
            l.unlock();
            pushed_.notify_one();
            return;
          } catch (const std::exception&) {
            open_.erase(at);
          }
        } catch (const std::exception&) {
        }
      }
    }
    if (bytes) memcpy(to, from, bytes);
    done_(ticket);
  }

 private:
  struct Copy {
    void* to;
    const void* from;
    uint64_t bytes, ticket;
  };

  // open_ holds disjoint ranges, so only the last one that starts below b can reach past a
  bool overlaps(uintptr_t a, uintptr_t b) const {
    const auto it = open_.lower_bound(b);
    return it != open_.begin() && std::prev(it)->second > a;
  }

  void work() {
    for (;;) {
      Copy c;
      {
        std::unique_lock<std::mutex> l(mu_);
        pushed_.wait(l, [&] { return end_ || !queue_.empty(); });
        if (queue_.empty()) return;
        c = queue_.front();
        queue_.pop_front();
      }
      memcpy(c.to, c.from, c.bytes);
      done_(c.ticket);
      {
        std::lock_guard<std::mutex> l(mu_);
        open_.erase(reinterpret_cast<uintptr_t>(c.to));
      }
      copied_.notify_one();
    }
  }

  std::function<void(uint64_t)> done_;
  std::mutex mu_;
  std::condition_variable pushed_, copied_;
  std::list<Copy> queue_;
  std::map<uintptr_t, uintptr_t> open_;  // destinations not yet written: start, end
  bool end_ = false;
  std::vector<std::thread> threads_;
};

}  // namespace lg

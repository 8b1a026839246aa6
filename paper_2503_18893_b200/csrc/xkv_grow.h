// A setting that only ever grows, shared by host threads (plain C++).
#pragma once

#include <stddef.h>

#include <atomic>
#include <mutex>

namespace xkv {

// Makes sure that the setting is at least `to`: `set(to)` applies it and returns a status that is zero when it worked.  What
// is on record is never above what is set: the check, the setting and the record are one step under `lock`, so a smaller
// value that another thread asks for at the same time cannot end up set behind a larger one.  A call that finds enough on
// record is one load.
template <class Set>
auto grow(std::atomic<size_t>& have, std::mutex& lock, size_t to, Set&& set) -> decltype(set(to)) {
  using Status = decltype(set(to));
  if (have.load(std::memory_order_acquire) >= to) return Status{};
  const std::lock_guard<std::mutex> held(lock);
  if (have.load(std::memory_order_relaxed) >= to) return Status{};
  const Status st = set(to);
  if (st == Status{}) have.store(to, std::memory_order_release);
  return st;
}

}  // namespace xkv

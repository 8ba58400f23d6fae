// Settings that belong to a CUDA context (kernel attributes), made once in each.
#pragma once
#include <deque>
#include <mutex>

namespace ha {

class ContextOnce {
 public:
  // Runs set() unless it has succeeded before for setting `bit` (a power of two) in the context
  // with this id.  Ids are never reused within a process, so a device reset makes the settings
  // anew; id 0 (unknown) always runs.  Returns what set() returns, 0 meaning success.  Threads
  // may call at the same time: each finds the setting made when its call returns.
  template <class F>
  int run(unsigned long long ctx_id, unsigned bit, F&& set) {
    if (ctx_id == 0) return set();
    std::lock_guard<std::mutex> lock(mutex_);
    Entry* e = find(ctx_id);
    if (e && (e->done & bit)) return 0;
    if (const int rc = set()) return rc;
    if (e) {
      e->done |= bit;
      return 0;
    }
    if (seen_.size() == kContexts) seen_.pop_front();
    seen_.push_back({ctx_id, bit});
    return 0;
  }

 private:
  static constexpr size_t kContexts = 64;   // the latest ones; older ones would be set again
  struct Entry {
    unsigned long long ctx_id;
    unsigned done;
  };
  Entry* find(unsigned long long ctx_id) {
    for (Entry& e : seen_)
      if (e.ctx_id == ctx_id) return &e;
    return nullptr;
  }
  std::mutex mutex_;
  std::deque<Entry> seen_;
};

}  // namespace ha

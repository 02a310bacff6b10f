// Idle workspaces kept for later calls of an entry point without a handle.
#pragma once

#include <cstddef>
#include <memory>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

namespace rtcc {

// A call takes a workspace of its CUDA context for itself, so calls from several
// threads never share one, and gives it back; up to kIdle of a context stay
// allocated.  Workspaces of a context that is gone went with it: they are
// dropped, untouched, when a call next has to make one, so a process keeps
// kIdle for each context it has and nothing for those it had.
//
// Space: `ctx`, the id of its context; create(ctx) and destroy(), with that
// context current; gone(), whether the context is (with any context current).
template <class Space, size_t kIdle>
class KeptPool {
 public:
  // Null if there is none idle and none can be made.
  std::unique_ptr<Space> take(unsigned long long ctx) {
    {
      std::lock_guard<std::mutex> lk(mu_);
      for (size_t i = idle_.size(); i-- > 0;)
        if (idle_[i]->ctx == ctx) {
          std::unique_ptr<Space> s = std::move(idle_[i]);
          idle_.erase(idle_.begin() + (std::ptrdiff_t)i);
          return s;
        }
      for (size_t i = idle_.size(); i-- > 0;)
        if (idle_[i]->gone()) idle_.erase(idle_.begin() + (std::ptrdiff_t)i);
    }
    std::unique_ptr<Space> s(new (std::nothrow) Space);
    if (s && !s->create(ctx)) {
      s->destroy();
      s.reset();
    }
    return s;
  }

  void give(std::unique_ptr<Space> s) {
    {
      std::lock_guard<std::mutex> lk(mu_);
      size_t n = 0;
      for (const auto& i : idle_) n += i->ctx == s->ctx ? 1 : 0;
      if (n < kIdle) {
        try {
          idle_.push_back(std::move(s));
          return;
        } catch (const std::bad_alloc&) {        // s is still here: not kept
        }
      }
    }
    s->destroy();
  }

 private:
  std::mutex mu_;
  std::vector<std::unique_ptr<Space>> idle_;
};

}  // namespace rtcc

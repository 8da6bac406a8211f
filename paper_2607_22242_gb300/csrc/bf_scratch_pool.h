// bf_scratch_pool.h -- scratch of scenario handles that are gone, for the next
// handles, and the record of calls that decides whether a handle's scratch may
// go there.  Host code only; no CUDA calls.
#pragma once

#include <stdint.h>

#include <mutex>

namespace bfcapi {

// A handle's calls that have put work out and not seen its end.  One that
// failed or stopped waiting stays open for good: a later call's wait, perhaps
// on another stream, says nothing of its work.
struct OpenCalls {
  uint32_t open;
  void begin() { ++open; }
  void end() { --open; }
  bool none_open() const { return open == 0u; }
};

// A device block and its pinned mirror (14 KB each): allocating and freeing them
// took most of a one-off search (12-tool fan-out through bf_create_scenario,
// bf_search_best and bf_destroy_scenario: 547 -> 118 us).  At most kMost pairs
// are kept; a pair belongs to the context it was made in and is only handed out
// there.  `context` gives the ID of the current context (never 0), or false.
template <typename Scratch>
class ScratchPool {
 public:
  struct Pair {
    Scratch* d;
    Scratch* h;
  };
  using ContextFn = bool (*)(unsigned long long*);

  explicit ScratchPool(ContextFn context) : context_(context) {}

  // ID of the current context, 0 when it cannot be told.
  unsigned long long context() const {
    unsigned long long id = 0;
    return context_(&id) ? id : 0;
  }

  // A pair made in the current context, or false.
  bool take(Pair* out) {
    const unsigned long long id = context();
    if (id == 0) return false;
    std::lock_guard<std::mutex> lock(mu_);
    for (unsigned i = 0; i < count_; ++i)
      if (slots_[i].ctx == id) {
        *out = slots_[i].pair;
        slots_[i] = slots_[--count_];
        return true;
      }
    return false;
  }

  // Keep a pair made in context `made_in`; false (the caller frees it) when the
  // pool is full or another context is current: the device may have been reset
  // since, and the pair be gone.
  bool keep(const Pair& pair, unsigned long long made_in) {
    if (made_in == 0 || made_in != context()) return false;
    std::lock_guard<std::mutex> lock(mu_);
    if (count_ == kMost) return false;
    slots_[count_++] = Slot{made_in, pair};
    return true;
  }

 private:
  static constexpr unsigned kMost = 16;
  struct Slot {
    unsigned long long ctx;
    Pair pair;
  };
  const ContextFn context_;
  std::mutex mu_;
  Slot slots_[kMost];
  unsigned count_ = 0;
};

}  // namespace bfcapi

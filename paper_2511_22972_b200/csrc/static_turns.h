// Turns at the parts of the static entry point's scratch.  Host code only.
#pragma once
#include <mutex>

namespace fly {

// A call runs on one of N parts and empties the next one for the call after it.  That holds only if calls are launched in the order of
// their turns, and if a call that was not launched had none: so launch(part, next) runs under the lock that the turn is taken under, and
// the turn passes on when it returns true.
template <unsigned N>
struct Turns {
  std::mutex mu;
  unsigned part = 0;

  template <typename Launch>
  bool take(Launch&& launch) {
    std::lock_guard<std::mutex> lock(mu);
    const unsigned next = (part + 1) % N;
    if (!launch(part, next)) return false;
    part = next;
    return true;
  }
};

}  // namespace fly

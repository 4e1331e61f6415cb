// sg_spans.h -- disjoint address ranges: which of the buffers a scheduler holds
// share memory (sg_sched.cu).  Host code only.
#pragma once

#include <cstdint>
#include <iterator>
#include <map>

namespace sg {

// A set of address ranges no two of which meet.
class Spans {
  public:
    // Add [start, start + bytes); false, and nothing added, if it meets one held.
    bool add(uintptr_t start, uint64_t bytes)
    {
        const auto next = at_.lower_bound(start);
        if (next != at_.end() && next->first - start < bytes) return false;
        if (next != at_.begin()) {
            const auto prev = std::prev(next);
            if (start - prev->first < prev->second) return false;
        }
        at_.emplace_hint(next, start, bytes);
        return true;
    }
    void remove(uintptr_t start) { at_.erase(start); }
    void clear() { at_.clear(); }

  private:
    std::map<uintptr_t, uint64_t> at_;     // start -> bytes
};

}  // namespace sg

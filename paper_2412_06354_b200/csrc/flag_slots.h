// Words of pinned host memory, each with an event, that calls borrow to wait for something a kernel reports to the host.
// Slots are handed out one per call in progress and kept for the next ones: making one takes some 20 us.
// Api makes and frees them (CUDA in the library), so that the rules below hold for any source of memory.
#pragma once
#include <mutex>
#include <vector>

namespace gnn {

constexpr size_t FLAG_SLOTS_KEPT = 8;  // idle slots; more exist only while more calls than that run at once

template <class Api>
class FlagSlots {
  public:
    struct Slot {
        int* word = nullptr;
        typename Api::Event event{};
        int device = -1;
    };

    bool take(int device, Slot* s) {
        {
            std::lock_guard<std::mutex> lock(mutex_);
            for (size_t k = 0; k < idle_.size(); ++k)
                if (idle_[k].device == device) {
                    *s = idle_[k];
                    idle_.erase(idle_.begin() + (long)k);
                    return true;
                }
        }
        s->device = device;
        if (!Api::make_word(&s->word)) return false;
        if (!Api::make_event(&s->event)) {
            Api::free_word(s->word);
            return false;
        }
        return true;
    }

    // quiet: nothing in any stream can still write the word.  If that is not known (a call failed and its stream could not be
    // waited for), the slot is neither reused nor freed.
    void give(const Slot& s, bool quiet) {
        if (!quiet) return;
        {
            std::lock_guard<std::mutex> lock(mutex_);
            if (idle_.size() < FLAG_SLOTS_KEPT) {
                idle_.push_back(s);
                return;
            }
        }
        Api::free_event(s.event);
        Api::free_word(s.word);
    }

  private:
    std::mutex mutex_;
    std::vector<Slot> idle_;
};

}  // namespace gnn

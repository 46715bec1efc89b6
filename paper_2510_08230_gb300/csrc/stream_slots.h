// stream_slots.h - a few scratch buffers of a matrix, each for one stream (plain
// C++, tested on the host).
#pragma once

#include <atomic>

namespace gk {

// The first COUNT streams that ask get a slot each and keep it; -1 for any
// other.  Streams are named by cudaStreamGetId's ids, which are never used
// again, unlike handles.
class StreamSlots {
public:
    static constexpr int COUNT = 4;
    int of(unsigned long long id) {
        for (int k = 0; k < COUNT; ++k) {
            unsigned long long seen = owner_[k].load();
            if (seen == 0 && owner_[k].compare_exchange_strong(seen, id + 1)) return k;
            if (seen == id + 1) return k;
        }
        return -1;
    }

private:
    std::atomic<unsigned long long> owner_[COUNT] = {};  // id + 1, 0: nobody
};

}  // namespace gk

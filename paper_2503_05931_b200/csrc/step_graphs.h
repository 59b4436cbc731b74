// Which steps are replayed as CUDA graphs, and what is kept of them.  Plain C++: the graph and its recording come from the caller, so that
// the rules are also checked on the host.
#pragma once
#include <cstdint>
#include <map>

namespace aed {

// Steps of the caller's own loop of one key that are launched kernel by kernel before its graph is recorded.  A recording costs about what
// a replay saves in that many steps, so a caller whose sizes never come again pays little, and one whose sizes do come again at most
// twice what the better way would have taken.  Beyond the row count of the ready-made activation planes (`many_rows`) a replay saves more.
// Recording, beside the step itself: 24 layers 0.9 to 1.0 ms up to 128 rows, 1.3 at 200; 4 layers 0.2 to 0.35 (and 5 to 40 ms when the
// driver takes more device memory for its graphs, 2 MB for five or six graphs of 24 layers).  us per step, launched / replayed, 24 layers, 1 / 8 /
// 24 / 48 / 64 / 128 / 200 / 400 rows: 474 / 430, 526 / 485, 666 / 632, 910 / 874, 1019 / 987, 1498 / 1463, 1936 / 1833, 2735 / 2602; 4 layers, 8 /
// 64 / 128 / 256 / 400 rows: 108 / 103, 193 / 189, 277 / 272, 402 / 384, 506 / 484.  (The kernels of a graph follow each other more closely, and a host
// that takes 3 us and more per launch is the slower of the two up to 32 rows.)
inline int steps_before_recording(bool many_rows) { return many_rows ? 16 : 32; }

template <class Key, class Exec>
class StepGraphs {
public:
    struct Entry {
        Exec exec{};
        int64_t nodes = 0;
        bool usable = false;
    };

    // Counts a step of the caller's loop: true once `before` of its key have come before it.
    bool due(const Key &key, int before)
    {
        int &n = seen_[key];
        if (n >= before) return true;
        ++n;
        return false;
    }

    // The graph of a key, from record(Entry &) -> bool at first use; null where recording failed.  That is not tried again: the steps of this
    // key are launched kernel by kernel then (a device that is full refuses the graph's memory and still runs its kernels).
    template <class Record>
    const Entry *get(const Key &key, Record record)
    {
        auto it = entries_.find(key);
        if (it == entries_.end()) {
            Entry e;
            e.usable = record(e);
            it = entries_.emplace(key, e).first;
        }
        return it->second.usable ? &it->second : nullptr;
    }

    template <class Destroy>
    void clear(Destroy destroy)
    {
        for (auto &e : entries_)
            if (e.second.usable) destroy(e.second.exec);
        entries_.clear();
        seen_.clear();
    }

private:
    std::map<Key, Entry> entries_;
    std::map<Key, int> seen_;
};

}  // namespace aed

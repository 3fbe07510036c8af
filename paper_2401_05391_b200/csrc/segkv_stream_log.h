// Which of the library's launches came last on each stream (host only, no CUDA headers).
#pragma once

#include <mutex>

namespace segkv_impl {

// A stream as a launch sees it.  Its handle alone does not name it: the default stream's is the same on every device, and
// the per-thread default stream's in every thread.
struct StreamKey {
    int device;
    const void* stream;
    const void* thread;           // per-thread default stream only: something of the calling thread's own
    bool operator==(const StreamKey& o) const { return device == o.device && stream == o.stream && thread == o.thread; }
};

// Where and when data was last written: the stream and the per-process sequence number of the launch.
struct WriteMark {
    StreamKey at;
    unsigned long long seq;       // 0: never written
};

enum Release { kAfterWait, kAtOnce, kAtOnceSerialised };      // when a launch lets its successor begin

// A kernel launched with programmatic stream serialisation may begin before its predecessor P in the stream has
// finished, but not before P lets it.  Most kernels do so behind their own grid-dependency wait (kAfterWait): everything older
// than P is complete then, and data whose producing launch is strictly older than P may be read by the new
// kernel from its very first instruction.  A kernel that lets its successor go at once vouches for less: for everything
// older if it was itself launched behind the whole kernel before (kAtOnceSerialised), else only for what was
// complete when IT began (kAtOnce).  (A launch of the caller's own in between only helps: it does not release its dependents
// early.)
class StreamLog {
public:
    // Record a launch; returns its sequence number.
    unsigned long long note(const StreamKey& at, Release rel) {
        std::lock_guard<std::mutex> lk(mu_);
        const unsigned long long seq = ++seq_;
        int slot = -1, oldest = 0;
        for (int i = 0; i < kSlots; ++i) {
            if (s_[i].used && s_[i].at == at) { slot = i; break; }
            if (!s_[i].used) { if (slot < 0) slot = i; }
            else if (s_[i].last < s_[oldest].last || !s_[oldest].used) oldest = i;
        }
        if (slot < 0) slot = oldest;          // more streams than slots: forget the one idle longest
        Slot& s = s_[slot];
        if (rel != kAtOnce) s.complete = seq;
        else if (!s.used || !(s.at == at)) s.complete = 0;       // (nothing is known of its predecessor)
        s.at = at;
        s.last = seq;
        s.used = true;
        return seq;
    }

    // Is what the launch behind `m` wrote complete when the next kernel on `at` begins?
    bool complete_for_next(const StreamKey& at, const WriteMark& m) {
        if (m.seq == 0 || !(m.at == at)) return false;
        std::lock_guard<std::mutex> lk(mu_);
        for (int i = 0; i < kSlots; ++i)
            if (s_[i].used && s_[i].at == at) return m.seq < s_[i].complete;
        return false;
    }

private:
    static constexpr int kSlots = 32;
    struct Slot {
        StreamKey at;
        unsigned long long last;      // sequence number of the latest launch there
        unsigned long long complete;  // launches older than this are complete when the next kernel there begins
        bool used;
    };
    std::mutex mu_;
    Slot s_[kSlots] = {};
    unsigned long long seq_ = 0;
};

}  // namespace segkv_impl

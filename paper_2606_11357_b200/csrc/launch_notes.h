// What this library launched last on a stream, as far as it is known.  Host only, no CUDA in it.
//
// Two decisions rest on it.  (1) Order: the GEMV and the GEMM read packed weights before they wait for the kernels ahead of them,
// so behind the device packer they have to be launched as ordinary kernels.  They are launched to start early only where a GEMV or
// GEMM is known to have been launched on the stream since the last packing there; that one was behind the packer as an ordinary
// kernel, or behind another such.  Whatever is not known -- a stream not seen before, an entry given up for another stream, a
// question to the runtime that failed -- is an ordinary launch, which costs overlap and never order.  (2) Overlap only: whether a
// half-SM GEMV follows another (see launch_one in gemv.cu).
//
// A stream is named by the runtime's number for it, which is the same for every handle of one stream (NULL and cudaStreamLegacy),
// another one for every device's NULL and every thread's cudaStreamPerThread, and never given out again.  While it is capturing it is
// named by its handle and the capture: a captured launch says nothing about what runs on the stream.  (A graph that is launched on the
// stream is waited for as a whole.)
#pragma once
#include <stdint.h>

#include <mutex>

namespace tf {

enum class LaunchKind : int { kNone = 0, kHalfSm, kWholeSm };

struct StreamName {
    unsigned long long stream, capture;     // capture 0: none
    bool known;                             // false: the runtime did not say
};

class LaunchNotes {
public:
    static constexpr int kEntries = 32;
    struct Seen {
        LaunchKind kind;               // kNone: nothing is known
        uint64_t packings;             // how many packings there had been when it was read
    };
    Seen look(const StreamName& s) noexcept {
        std::lock_guard<std::mutex> hold(mutex_);
        const Entry* e = s.known ? find(s) : nullptr;
        return {e ? e->kind : LaunchKind::kNone, packings_};
    }
    // A kernel that is not the packer has been launched, going by `seen`.  If another host thread has packed since then, the launch may have
    // come before the packing: nothing is known.
    void launched(const StreamName& s, const Seen& seen, LaunchKind kind) noexcept {
        std::lock_guard<std::mutex> hold(mutex_);
        if (!s.known) return;
        Entry* e = find(s);
        if (seen.packings != packings_) {
            if (e) e->kind = LaunchKind::kNone;
            return;
        }
        if (!e) e = free_entry();
        *e = {s.stream, s.capture, kind};
    }
    // The packer has been launched (noted after the launch: a caller may use the blob when the call has returned).  In a capture every stream of it
    // is forgotten, since a dependency between two of them need not be a wait.
    void packed(const StreamName& s) noexcept {
        std::lock_guard<std::mutex> hold(mutex_);
        ++packings_;
        for (Entry& e : entries_)
            if (!s.known || (e.capture == s.capture && (s.capture != 0 || e.stream == s.stream))) e.kind = LaunchKind::kNone;
    }

private:
    struct Entry {
        unsigned long long stream, capture;
        LaunchKind kind;               // kNone: empty
    };
    Entry* find(const StreamName& s) noexcept {
        for (Entry& e : entries_)
            if (e.kind != LaunchKind::kNone && e.stream == s.stream && e.capture == s.capture) return &e;
        return nullptr;
    }
    Entry* free_entry() noexcept {      // an empty one, else that of the stream whose turn it is
        for (Entry& e : entries_)
            if (e.kind == LaunchKind::kNone) return &e;
        next_ = (next_ + 1) % kEntries;
        return &entries_[next_];
    }
    std::mutex mutex_;
    Entry entries_[kEntries] = {};
    int next_ = 0;
    uint64_t packings_ = 0;
};

}  // namespace tf

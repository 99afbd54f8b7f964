// Which GEMM launches may begin before the previous kernel of their stream has ended.  Host code without CUDA calls.
//
// Programmatic dependent launch lets a GEMM kernel request packed weights while the previous kernel of its stream still runs.
// That kernel may be a w4a16_pack that writes those weights (pack_kernel lets the next launch start as soon as all of its CTAs
// are there), or may itself have started before such a pack ended.  So the first GEMM launched on a stream after any pack on
// the device is a plain, fully ordered launch; behind a GEMM that was itself ordered behind the pack, the next ones may
// overlap their predecessor again.
#pragma once

#include <stdint.h>

namespace w4a16 {

constexpr uintptr_t kPerThreadStream = 0x2;          // cudaStreamPerThread: one handle for a stream of each host thread

class PackOrder {
public:
    void pack_issued() { ++epoch_; }

    // May a pack, or a kernel that may come behind one, start early and let the next launch start early?  Not in a capture (id
    // `capture`, 0 = none): the replays of a graph are not counted, so that a GEMM behind one may be allowed to overlap.
    static bool may_release(unsigned long long capture) { return capture == 0; }

    // Has a GEMM been launched on `stream` (a cudaStream_t) since the last pack, or captured since then in the capture that the
    // stream is in?  capture_of() tells its id, and is asked only where the stream's own record does not allow the overlap,
    // because asking the runtime costs 50 to 100 ns of a call's 3.5 us: with no pack since then there is none in the capture
    // either, and the graph's replays are ordered behind whatever is on their stream.
    template <typename Capture>
    bool may_overlap(uintptr_t stream, const Capture& capture_of) const {
        if (current({own(stream), 0})) return true;
        const unsigned long long capture = capture_of();
        return capture != 0 && current({own(stream), capture});
    }

    // f(overlap) launches a GEMM kernel and tells whether it got onto the stream.  A launch that was refused orders nothing:
    // only one that is there stands between the pack and what comes behind.  Nor does a captured one on the stream: it does
    // not run there.
    template <typename Capture, typename F>
    bool launch(uintptr_t stream, const Capture& capture_of, const F& f) {
        const bool overlap = may_overlap(stream, capture_of);
        const bool ok = f(overlap);
        if (ok && !overlap) launched({own(stream), capture_of()});
        return ok;
    }

private:
    // The epoch counts the packs; a slot holds the epoch of its queue's last GEMM launch: a stream, or a capture of it.  (A
    // queue without a slot gets a plain launch, so that what is evicted costs no more than that.)
    struct Queue { uintptr_t stream; unsigned long long capture; };
    struct Slot {
        Queue queue;
        unsigned long long epoch;
        bool of(const Queue& q) const { return epoch != 0 && queue.stream == q.stream && queue.capture == q.capture; }
    };
    static constexpr int kSlots = 32;

    // The calling thread's own stream of that handle.  (An address is no handle of another stream; the next thread that gets
    // it inherits a record like the one that a new stream inherits with a handle: older than any pack still to come.)
    static uintptr_t own(uintptr_t stream) {
        static thread_local char thread;
        return stream == kPerThreadStream ? reinterpret_cast<uintptr_t>(&thread) : stream;
    }

    bool current(const Queue& queue) const {
        for (const Slot& s : slots_)
            if (s.of(queue)) return s.epoch == epoch_;
        return false;
    }

    void launched(const Queue& queue) {
        Slot* slot = nullptr;
        for (Slot& s : slots_)
            if (s.of(queue)) { slot = &s; break; }
        for (int i = 0; slot == nullptr && i < kSlots; ++i)
            if (slots_[i].epoch == 0) slot = &slots_[i];
        if (slot == nullptr) {
            slot = &slots_[evict_];
            evict_ = (evict_ + 1) % kSlots;
        }
        *slot = {queue, epoch_};
    }

    unsigned long long epoch_ = 1;
    Slot slots_[kSlots] = {};
    int evict_ = 0;
};

}  // namespace w4a16

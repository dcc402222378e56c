// When a product may start early behind the library's own producers of sign words and scales (pack, compress).
//
// A product launched with an early start fetches W_base, sign words and scales while the kernel ahead of it on its stream is still running, so
// one that follows a producer has to be launched without.  Every producer call leaves a mark; a product starts early only if one on the same
// stream of the same device has been launched without since the last mark.  The mark is one for all streams (a producer may reach this stream
// through an event or the default stream's implicit order), what has been seen of it belongs to (device, stream): a product on
// another stream, device or thread says nothing about the order on this one.  A capture has a mark of its own, from the producers recorded
// in it: those outside run before or after a whole replay, and a call that is only recorded orders nothing outside (one mark for both would cost
// the first product of every graph its early start).
// What is forgotten costs a launch without the early start, never the order.  (Host code only.)
#pragma once
#include <atomic>
#include <cstdint>
#include <mutex>

namespace bd {

struct StreamKey {
    int device = -1;
    const void* stream = nullptr;
    unsigned long long capture = 0;   // the capture that the call is recorded in, 0: none
    bool operator==(const StreamKey& o) const { return device == o.device && stream == o.stream && capture == o.capture; }
};

class ProducerNote {
public:
    // Before a producer's first launch and after its last one, launched or not: a product that another thread puts between them is held back, too,
    // and is no answer for the next one.  capture: the one that its stream is in (0: none), known: whether the stream could say.
    void produced(bool known, unsigned long long capture) {
        std::lock_guard<std::mutex> lock(mu_);
        const unsigned long long v = count_.fetch_add(1) + 1;
        if (!known || capture == 0) eager_ = v;
        if (!known) forgotten_ = v;
        if (known && capture == 0) return;
        for (Recorded& r : recorded_) {
            if (!known && r.mark != 0) r.mark = v;
            if (known && r.capture == capture) {
                r.mark = v;
                return;
            }
        }
        if (!known) return;
        Recorded& r = recorded_[next_];
        next_ = (next_ + 1) % kCaptures;
        if (r.mark > forgotten_) forgotten_ = r.mark;
        r = {capture, v};
    }
    // False: there has been no producer at all, every product may start early.
    bool any() const { return count_.load() != 0; }
    // The last mark that concerns a product in `capture` (0: an eager one); 0: none.
    unsigned long long mark(unsigned long long capture) {
        std::lock_guard<std::mutex> lock(mu_);
        if (capture == 0) return eager_;
        for (const Recorded& r : recorded_)
            if (r.capture == capture) return r.mark;
        return forgotten_;
    }
    // Whether a product on `key` was launched without the early start at `mark` (as read before the question) or later.
    bool settled(const StreamKey& key, unsigned long long mark) {
        std::lock_guard<std::mutex> lock(mu_);
        const Set& s = sets_[set_of(key)];
        for (int i = 0; i < kWays; ++i)
            if (s.seen[i] >= mark && s.key[i] == key) return true;
        return false;
    }
    // ... it has been, after its launch (not before: a product of another thread could slip in ahead of it).
    void settle(const StreamKey& key, unsigned long long mark) {
        std::lock_guard<std::mutex> lock(mu_);
        Set& s = sets_[set_of(key)];
        int at = -1;
        for (int i = 0; i < kWays && at < 0; ++i)
            if (s.seen[i] != 0 && s.key[i] == key) at = i;
        if (at < 0) {
            at = s.next;
            s.next = (at + 1) % kWays;
            s.seen[at] = 0;
            s.key[at] = key;
        }
        if (s.seen[at] < mark) s.seen[at] = mark;
    }

private:
    static constexpr int kSets = 64, kWays = 4;   // 256 streams and captures at a time
    static constexpr int kCaptures = 16;          // captures with producers in them
    struct Recorded {
        unsigned long long capture, mark;   // 0: free
    };
    struct Set {
        StreamKey key[kWays];
        unsigned long long seen[kWays] = {};   // 0: free
        int next = 0;
    };
    static unsigned set_of(const StreamKey& k) {
        uint64_t h = reinterpret_cast<uint64_t>(k.stream) ^ ((uint64_t)(unsigned)k.device << 56) ^ (k.capture * 0xD1B54A32D192ED03ull);
        h *= 0x9E3779B97F4A7C15ull;
        return (unsigned)(h >> 58);
    }
    std::atomic<unsigned long long> count_{0};
    std::mutex mu_;
    Set sets_[kSets];
    Recorded recorded_[kCaptures] = {};
    int next_ = 0;
    unsigned long long eager_ = 0, forgotten_ = 0;   // (forgotten_: the last mark of the captures that are no longer held)
};

// Around a producer's launches.  key_of as below.
class Producing {
public:
    template <class KeyOf>
    Producing(ProducerNote& note, KeyOf key_of) : note_(note) {
        known_ = key_of(&key_);
        note_.produced(known_, key_.capture);
    }
    ~Producing() { note_.produced(known_, key_.capture); }

private:
    ProducerNote& note_;
    StreamKey key_;
    bool known_;
};

// One product call: `early` says how to launch it; `launched` after a successful launch.
// key_of(StreamKey*): false if the stream cannot say whether it is being captured (then no early start, and nothing learned).
class ProductStart {
public:
    template <class KeyOf>
    ProductStart(ProducerNote& note, bool enabled, KeyOf key_of) : early(enabled), note_(note) {
        if (!enabled || !note_.any()) return;
        const bool known = key_of(&key_);
        mark_ = known ? note_.mark(key_.capture) : 0;
        early = known && (mark_ == 0 || note_.settled(key_, mark_));
        held_back_ = known && !early;
    }
    void launched() {
        if (held_back_) note_.settle(key_, mark_);
    }
    bool early;

private:
    ProducerNote& note_;
    StreamKey key_;
    unsigned long long mark_ = 0;
    bool held_back_ = false;
};

}  // namespace bd

// When a product may start early behind the library's own producers of sign words and scales (pack, compress).
//
// A product launched with an early start fetches W_base, sign words and scales while the kernel ahead of it on its stream is still running, so
// one that follows a producer has to be launched without.  A producer call counts up; a product starts early only if one on the same stream
// of the same device has been launched without since the count last moved.  The count is one for the process (a producer may reach this stream
// through an event or the default stream's implicit order), what has been seen of it belongs to (device, stream, capture): a product on
// another stream, device or thread, or one that is only being captured, says nothing about the order on this one.
// A forgotten entry costs one launch without the early start, never the order.  (Host code only.)
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
    // and is no answer for the next one.
    void produced() { count_.fetch_add(1); }
    // 0: there has been no producer, every product may start early.
    unsigned long long count() const { return count_.load(); }
    // Whether a product on `key` was launched without the early start at `count` (as read before the question).
    bool settled(const StreamKey& key, unsigned long long count) {
        std::lock_guard<std::mutex> lock(mu_);
        const Set& s = sets_[set_of(key)];
        for (int i = 0; i < kWays; ++i)
            if (s.seen[i] == count && s.key[i] == key) return true;
        return false;
    }
    // ... it has been, after its launch (not before: a product of another thread could slip in ahead of it).
    void settle(const StreamKey& key, unsigned long long count) {
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
        if (s.seen[at] < count) s.seen[at] = count;
    }

private:
    static constexpr int kSets = 64, kWays = 4;   // 256 streams and captures at a time
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
};

// Around a producer's launches.
struct Producing {
    ProducerNote& note;
    explicit Producing(ProducerNote& n) : note(n) { note.produced(); }
    ~Producing() { note.produced(); }
};

// One product call: `early` says how to launch it; `launched` after a successful launch.
// key_of(StreamKey*): false if the stream cannot say whether it is being captured (then no early start, and nothing learned).
class ProductStart {
public:
    template <class KeyOf>
    ProductStart(ProducerNote& note, bool enabled, KeyOf key_of) : note_(note), count_(note.count()) {
        early = enabled;
        if (count_ == 0 || !enabled) return;
        known_ = key_of(&key_);
        early = known_ && note_.settled(key_, count_);
        known_ = known_ && !early;
    }
    void launched() {
        if (known_) note_.settle(key_, count_);
    }
    bool early;

private:
    ProducerNote& note_;
    StreamKey key_;
    unsigned long long count_;
    bool known_ = false;
};

}  // namespace bd

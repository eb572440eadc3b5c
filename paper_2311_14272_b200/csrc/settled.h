// Host-side bookkeeping: whether a product may read its handle's weight tiles and walk lists before the kernel in front of it in the stream has
// finished.  That kernel must not be one that writes them.  Plain C++ without CUDA.
#pragma once
#include <atomic>
#include <cstdint>

namespace crisp {

// The encode calls of the process, and the moments between them at which nothing was being encoded.
class EncodeCount {
public:
    // Around the launches of an encode call.
    void begin() { begun_.fetch_add(1); }
    void end() { ended_.fetch_add(1); }
    // Launches that go into a graph happen again whenever it is replayed, and nobody counts that: as long as there is such a graph, there is no moment of
    // which it is known that nothing has been encoded since another.
    void graph_made() { graphs_.fetch_add(1); }
    void graph_gone() { graphs_.fetch_sub(1); }
    // The present moment: the same number as long as nothing is encoded.  0: something is just being, or a graph may at any time.
    uint64_t now() const {
        const uint64_t ended = ended_.load();                // (read first: where it equals what has begun, all that had begun by then has ended)
        return begun_.load() == ended && graphs_.load() == 0 ? ended + 1 : 0;
    }

private:
    std::atomic<uint64_t> begun_{0}, ended_{0}, graphs_{0};
};

// What a handle keeps of its last product that ran: the stream, and the moment before it was launched.  A product may read ahead where one went before
// in the same stream and nothing has been encoded since.  The kernel in front then either is that product or came after it, began when that product had
// waited for all that came before, and everything up to the last encode had finished by then.  (A product in another stream, or one that was
// captured, says nothing about the kernel in front.)
class Settled {
public:
    bool holds(const void *stream, uint64_t now) const { return now != 0 && at_ == now && stream_ == stream; }
    void note(const void *stream, uint64_t now, bool ran) {
        stream_ = stream;
        at_ = ran ? now : 0;
    }

private:
    const void *stream_ = nullptr;
    uint64_t at_ = 0;
};

// Launches a product whose parameters p say whether it reads early, decided at `moment`.  An encode that another host thread has called meanwhile may have
// come between the decision and the launch: the product is then made once more, behind everything (its results are the same buffer).
// launch() returns 0 where it succeeded.
template <typename Params, typename Launch>
auto launch_product(const EncodeCount &encodes, Params &p, uint64_t moment, const Launch &launch) {
    auto error = launch();
    if (error == 0 && p.early && encodes.now() != moment) {
        p.early = 0;
        error = launch();
    }
    return error;
}

}  // namespace crisp

// Which freed device blocks of the valid lists are kept for the next handle's
// lists (host side only; the blocks and their events are the caller's to
// create and free).
#pragma once

#include <stddef.h>

#include <utility>
#include <vector>

namespace tmk {

constexpr size_t kSpareListBlocks = 2;  // kept per device
// A block that so many requests in a row could not use for its size gives way to
// the next one that comes back, smaller or larger: batches that have shrunk
// for good find their block again and the peak's memory is returned, while
// every eighth batch may still be a large one and find its own.
constexpr int kSpareUnfit = 8;

struct SpareBlock {
    int dev = -1;
    void *p = nullptr;
    size_t bytes = 0;
    void *ready = nullptr;  // event after the block's last use (null: none pending)
    int unfit = 0;          // requests since then that it was too small or too large for
};

class SpareBlocks {
public:
    // The smallest kept block of device dev for `bytes`, at most twice as
    // large, whose last use is over by done(event); p is null if there is none.
    template <typename Done>
    SpareBlock take(int dev, size_t bytes, Done done) {
        size_t best = kept_.size();
        for (size_t i = 0; i < kept_.size(); i++) {
            SpareBlock &b = kept_[i];
            if (b.dev != dev) continue;
            if (b.bytes < bytes || b.bytes > 2 * bytes) {
                b.unfit++;
                continue;
            }
            if (best < kept_.size() && kept_[best].bytes <= b.bytes) continue;
            if (!b.ready || done(b.ready)) best = i;
        }
        if (best == kept_.size()) return SpareBlock();
        SpareBlock b = kept_[best];
        kept_.erase(kept_.begin() + long(best));
        b.unfit = 0;
        return b;
    }

    // Keeps the block; returns the one to free instead (p null: none). With
    // kSpareListBlocks kept it takes the place of one whose last use is over:
    // of the one that most requests could not use, from kSpareUnfit on, else of
    // the smallest smaller one (so that sizes in turn end up with the largest
    // blocks, which serve the others too).
    template <typename Done>
    SpareBlock give(SpareBlock block, Done done) {
        size_t held = 0;
        SpareBlock *out = nullptr;
        for (SpareBlock &b : kept_) {
            if (b.dev != block.dev) continue;
            held++;
            const bool stale = b.unfit >= kSpareUnfit;
            if (!stale && b.bytes >= block.bytes) continue;
            if (out) {
                const bool out_stale = out->unfit >= kSpareUnfit;
                if (out_stale && (!stale || b.unfit <= out->unfit)) continue;
                if (!out_stale && !stale && b.bytes >= out->bytes) continue;
            }
            if (!b.ready || done(b.ready)) out = &b;
        }
        if (held < kSpareListBlocks) {
            kept_.push_back(block);
            return SpareBlock();
        }
        if (out) std::swap(*out, block);
        return block;
    }

private:
    std::vector<SpareBlock> kept_;
};

}  // namespace tmk

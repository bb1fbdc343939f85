// nls_ring.h -- which entries of a handle's ring of device counters a flush
// takes, and when they are zeroed (host arithmetic only).
#pragma once

#include <algorithm>

namespace nls {

// Entries [pos, zeroed) are free and zero, by memsets of which the last went to
// the stream zero_on.  Blocks are zeroed as the position reaches them, on the
// stream of the flush that reaches them, so that most flushes need no memset.
//
// A flush may take entries of two memsets: the rest of a block that another
// stream zeroed, then a block that it zeroes itself.  The memset of the later
// block is therefore ordered after the earlier one's, and one event, recorded
// behind it, stands for both.
//
// A flush recorded by a stream capture zeroes its own entries each time it
// runs.  Its replays also write them at times that the ring does not see,
// before and after they are handed out again: from the first such flush on,
// every flush zeroes exactly its own entries.
template <class Stream>
struct CounterRing {
    int size, block;
    int pos = 0, zeroed = 0;
    bool any = false;      // a memset was made, on:
    Stream zero_on{};
    bool recorded = false; // a capture has recorded a flush

    CounterRing(int size_, int block_) : size(size_), block(block_) {}

    // Takes `count` <= size consecutive entries for a flush on `st`; the first
    // one's index goes to *start.  ops.release(i): entry i's request is complete
    // and its count kept; ops.zero(first, end, st): memset, then the event;
    // ops.after_zero(st): st waits for the event.  All return 0 or an error code.
    template <class Ops>
    int take(int count, Stream st, bool captured, Ops &&ops, int *start)
    {
        if (pos + count > size) pos = zeroed = 0;
        recorded = recorded || captured;
        if (recorded) zeroed = pos;
        if (!captured && any && st != zero_on)
            if (int rc = ops.after_zero(st)) return rc;
        const int end = pos + count;
        if (end > zeroed) {
            const int z1 = recorded ? end : std::min(size, (end + block - 1) / block * block);
            for (int i = zeroed; i < z1; ++i)
                if (int rc = ops.release(i)) return rc;
            if (!captured) {
                if (int rc = ops.zero(zeroed, z1, st)) return rc;
                any = true;
                zero_on = st;
            }
            zeroed = z1;
        }
        *start = pos;
        pos = end;
        return 0;
    }
};

} // namespace nls

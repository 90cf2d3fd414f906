// Which launch chains are kept captured: plain C++, no device code.
//
// A chain is captured when its geometry comes back (a stream whose geometries never repeat is launched kernel by kernel),
// and kept in one of a few slots.  Once all are taken a chain gives way, the least recently used first, and only to a
// geometry that has come twice since that chain was last used: a stream that goes round more geometries than there are
// slots replays as many as fit and captures none over and over.
#pragma once

#include <cstdint>

namespace rp {

struct ChainStore {   // all zero: empty
    static constexpr int SLOTS = 16, SEEN = 32;
    uint64_t now;                                 // batches asked about so far
    uint64_t key[SLOTS], used[SLOTS];             // used: when last replayed, 0 = empty slot
    uint64_t seen_key[SEEN], seen_at[SEEN];       // geometries without a chain, and when each last came

    // the slot of this geometry's chain, or -1
    int find(uint64_t k) {
        ++now;
        for (int i = 0; i < SLOTS; ++i)
            if (used[i] && key[i] == k) {
                used[i] = now;
                return i;
            }
        return -1;
    }

    // after a find that failed: the slot to capture this geometry's chain into (put() enters it), or -1
    int place(uint64_t k) {
        int at = 0, slot = 0;
        for (int i = 0; i < SEEN; ++i) {
            if (seen_at[i] && seen_key[i] == k) { at = i; break; }
            if (seen_at[i] < seen_at[at]) at = i;
        }
        const uint64_t before = seen_at[at] && seen_key[at] == k ? seen_at[at] : 0;
        seen_key[at] = k;
        seen_at[at] = now;
        for (int i = 1; i < SLOTS; ++i)
            if (used[i] < used[slot]) slot = i;
        return before > used[slot] ? slot : -1;
    }

    void put(int slot, uint64_t k) {
        key[slot] = k;
        used[slot] = now;
    }

    void drop(int slot) { used[slot] = 0; }
    void clear() { *this = ChainStore{}; }
};

}  // namespace rp

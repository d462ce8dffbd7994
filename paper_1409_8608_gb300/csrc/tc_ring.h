// Books of the rings into which a producer copies tiles: one of bytes, tiles of
// their own sizes released by their readers in order (tc_stream.cu), and what
// a producer of any ring waits for before its block may leave, since another
// role may have given up with copies on their way.  Plain C++, so that they can
// be run on the host too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define TC_RING_FN __host__ __device__ __forceinline__
#else
#define TC_RING_FN inline
#endif

namespace tc {

// Tiles take [pos, pos + size) in order, none wrapping the end; each has one of
// SLOTS slots, in order too.
template <int BYTES, int SLOTS>
struct ByteRing {
    int used = 0, pos = 0;               // bytes taken (with the ends skipped); where the next tile goes
    int slot = 0, oldest = 0, busy = 0;  // next slot, the oldest not known released, how many of those
    uint32_t ph = 0;                     // parity of the oldest slot's phase

    TC_RING_FN void next_oldest() {
        --busy;
        if (++oldest == SLOTS) oldest = 0, ph ^= 1u;
    }

    // Waits for releases until `size` bytes in one piece and a slot are free;
    // skip: bytes left out at the end of the ring.  wait(slot, parity): the
    // slot's tile has been released; held(slot): the bytes that it took.  False
    // when a wait gave up: its tile then still counts as in flight.
    template <class Wait, class Held>
    TC_RING_FN bool make_room(int size, int &skip, Wait wait, Held held) {
        skip = pos + size > BYTES ? BYTES - pos : 0;
        while (used + skip + size > BYTES || busy == SLOTS) {
            if (!wait(oldest, ph)) return false;
            used -= held(oldest);
            next_oldest();
        }
        return true;
    }

    // The place of a tile that make_room found room for; it takes size + skip
    // bytes, in slot `slot` as it was before.
    TC_RING_FN int take(int size, int skip) {
        if (pos + size > BYTES) pos = 0;
        const int at = pos;
        used += size + skip;
        pos += size;
        ++busy;
        if (++slot == SLOTS) slot = 0;
        return at;
    }

    // landed(slot, parity) for every tile not known released, oldest first.
    template <class Landed>
    TC_RING_FN void drain(Landed landed) {
        while (busy > 0) {
            landed(oldest, ph);
            next_oldest();
        }
    }
};

// f(slot, parity) for the last fillings of a ring's slots that nothing may have
// read: filling q goes to slot q % slots and completes phase q / slots of its
// barrier.
template <class F>
TC_RING_FN void last_filled(int64_t filled, int slots, F f) {
    for (int64_t q = filled > slots ? filled - slots : 0; q < filled; ++q) f((int)(q % slots), (uint32_t)((q / slots) & 1));
}

}  // namespace tc

// How the warps of a CTA take pieces of work that are shared out among CTAs that join while it runs.
//
// Pieces come in lots from one counter of the launch: a CTA takes a lot, its warps the pieces of it.  One word of the CTA holds the number of
// its lot << 12 | calls since; another the lot after it, which was asked for one lot ago (-1: not here yet).  Of the calls of a lot the
// first `pieces` get one each, the next one fetches the lot behind it and gets its first piece, and any further ones wait for that.  A caller
// that waits leaves again as soon as the count is down to `pieces`, too: the new lot may be used up before it looks, and then it is the one
// to fetch the lot after that.  (Waiting for a piece to be free, it waited for others to come; behind the last lot nobody does.)
//
// Cell: add() adds one to the word and returns what was there, swap(x) replaces it, peek() reads it; next() reads the other word, put(x) writes it
// (writes of a caller are seen in their order); ask() takes a number from the launch's counter.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MVLA_LOTS_FN __host__ __device__ __forceinline__
#else
#define MVLA_LOTS_FN inline
#endif

namespace mvla {

// The caller's next piece; at or past lots * pieces: there is none, nor will there be.  More than `limit` tries in all: gives up
// (*gave_up), as if there were none.
template <class Cell>
MVLA_LOTS_FN uint32_t take_piece(Cell& c, uint32_t pieces, uint32_t lots, uint32_t limit, bool* gave_up)
{
    for (uint32_t it = 0;;) {
        const uint32_t got = c.add(), used = got & 0xFFFu;
        if (used < pieces) return (got >> 12) * pieces + used;
        if (used == pieces) {
            int32_t lot = c.next();
            for (; lot < 0 && it < limit; ++it) lot = c.next();        // (the caller that has asked for it waits for nobody)
            if (lot < 0) break;
            c.put(-1);
            c.swap(static_cast<uint32_t>(lot) << 12 | 1u);
            c.put(static_cast<uint32_t>(lot) < lots ? c.ask() : lot);
            return static_cast<uint32_t>(lot) * pieces;
        }
        while ((c.peek() & 0xFFFu) > pieces && it < limit) ++it;
        if (it >= limit) break;
    }
    *gave_up = true;
    return lots * pieces;
}

}  // namespace mvla

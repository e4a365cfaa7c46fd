// warp_table.cuh -- an open-addressing table that the 32 lanes of one warp
// fill together without atomics.  Plain C++ but for the warp intrinsics, so
// that a host program can run it with lanes of its own.
#pragma once

namespace fq {

// Every lane with `open` looks for its record e in `tab` (slots of mask + 1,
// free ones hold `none`) from slot s on and returns the record that holds its
// place: e itself, or the record x already there with same(x).
// A turn has three steps, each complete in all lanes before the next begins:
// read the slot; lanes that found it free write their record there; they read
// back whose claim stayed.  Without the first barrier a lane may read a claim
// that is overwritten at once, compare its key with the wrong record and
// insert a determinant a second time.
template <typename TAB, typename SLOT, typename SAME>
__device__ __forceinline__ int warp_claim(TAB tab, unsigned mask, unsigned s, SLOT e, SLOT none, bool open, SAME same)
{
    int target = -1;
    while (__any_sync(0xffffffffu, open)) {
        SLOT x = none;
        if (open) x = tab[s];
        __syncwarp();
        const bool claims = open && x == none;
        if (claims) tab[s] = e;
        __syncwarp();
        if (open) {
            if (claims) x = tab[s];
            if (x == e || same(x)) {
                target = (int)x;
                open = false;
            } else {
                s = (s + 1) & mask;
            }
        }
    }
    return target;
}

}  // namespace fq

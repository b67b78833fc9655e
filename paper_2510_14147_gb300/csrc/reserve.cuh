// reserve.cuh -- room in a list that many warps fill.
#pragma once

#ifndef CT_HD
#define CT_HD __host__ __device__ __forceinline__
#endif

namespace ct {

// Takes n entries of a list of `cap` entries: the first one, or -1 when they
// do not fit.  used: the count as last seen; cas(expected, desired) returns the
// count it found and stores `desired` where that was `expected`.  The count
// never passes cap.  (An atomic add also counts what does not fit: a walk that
// stops below a vertex of a million children asks for up to 16 thousand
// entries, and some hundred thousand such walks wrap a 32-bit count, after
// which the stores go before the list.)  A compare-and-swap that fails means
// that another warp took entries, so the loop ends after at most cap of them.
template <class Cas>
CT_HD int list_reserve(int used, int n, int cap, Cas cas) {
    while (n <= cap - used) {
        const int found = cas(used, used + n);
        if (found == used) return used;
        used = found;
    }
    return -1;
}

}  // namespace ct

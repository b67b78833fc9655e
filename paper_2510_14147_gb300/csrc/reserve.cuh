// reserve.cuh -- room in a list that many warps fill.
#pragma once

#ifndef CT_HD
#define CT_HD __host__ __device__ __forceinline__
#endif

namespace ct {

// A list of `cap` entries is filled by atomic adds of the entries wanted to a
// 64-bit count, which goes past cap once they do not fit.  (A walk that stops
// below a vertex of a million children asks for up to 16 thousand entries, and
// some hundred thousand such walks wrap a 32-bit count, after which the stores
// go before the list.  A compare-and-swap that leaves the count alone when the
// entries do not fit is no way out: many walks stop at the same time, and the
// walk of a million 256-bit codes took 11.2 ms instead of 5.1.)
struct ListRoom {
    int begin;  // the first entry, cap if there is none
    bool fits;  // all the entries have room; else those from begin on are marked empty
};
// The n entries asked for after `first` others.
CT_HD ListRoom list_room(unsigned long long first, int n, int cap) {
    const unsigned long long end = (unsigned long long)cap;
    return ListRoom{first < end ? (int)first : cap, first + (unsigned long long)n <= end};
}
// Entries stored or marked empty of those asked for.
CT_HD int list_length(unsigned long long asked, int cap) {
    return asked < (unsigned long long)cap ? (int)asked : cap;
}

}  // namespace ct

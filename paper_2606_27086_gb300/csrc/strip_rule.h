// When the strip-ordered passes (strip.cu) serve a list of items at all, from
// the items' lengths alone: plain C++, evaluated at create before anything is
// built.
#pragma once

#include <algorithm>
#include <climits>
#include <vector>

namespace suppy {

// Ring bytes: CT 512x512 ran the same from 96 to 192 KB (254-257 us a row
// pass), so the rest stays with L1.  Strips are taken while their padding stays
// below kStripSlots slots per entry: at 1.4 an entry costs 8.6 bytes, about the
// streamed passes' 8, and CT and travel-time rows lie at 1.05-1.10, their
// columns at 1.11-1.38.  Where the packets stay in L2 bytes matter less (dose
// matrices: rows 1.19, columns 1.40).  Packets of up to 8 MB are taken whatever
// their padding: a pass over them is a few microseconds of latency, which the
// streamed passes' rings make more of (row pass in us, streamed and strips:
// 16x16 in 16 angles 18.4 / 8.0 at 2.2 slots an entry, 32x32 in 500 angles, 7.5
// MB, 49.5 / 22.8 at 1.74; columns of 200 travel-time rows over 100x200, 3.7 MB,
// 70.1 / 12.4 at 22).  Above, the strips lose where padding is common: 26 MB at
// 2.6 slots 34.9 / 48.3.
constexpr int kStripRing = 160 * 1024;
constexpr double kStripSlots = 1.4, kStripSlotsL2 = 1.6;
constexpr long long kStripL2 = 80LL * 1024 * 1024, kStripSmall = 8LL * 1024 * 1024;

// `packets` packets of pbytes, `most` in one strip, for `entries` entries.
inline bool strips_pay(long long packets, long long most, int pbytes, long long entries) {
    const long long bytes = packets * pbytes;
    const double slots = bytes <= kStripL2 ? kStripSlotsL2 : kStripSlots;
    return packets >= 1 && (bytes <= kStripSmall || (double)packets * 128.0 <= slots * (double)entries + 128.0) &&
           most * pbytes <= kStripRing / 2 && (bytes >> 4) <= 0xffffffffLL;
}

// Whether they can: item numbers are 32 bits (blocks x columns may pass 2^31
// where the entries do not), and a strip takes at least as many packets as its
// longest item has windows of 32 entries.  False only where the count made on
// the device would say no as well.  block_of: first item of every block, and
// the end; len(t, i): entries of item i of block t.
template <class Len>
bool strips_possible(const std::vector<long long>& block_of, Len len, int pbytes, long long entries) {
    if (block_of.back() > INT_MAX) return false;
    long long packets = 0, most = 0;
    for (size_t t = 0; t + 1 < block_of.size(); ++t)
        for (long long i = block_of[t]; i < block_of[t + 1]; i += 4) {
            long long longest = 0;
            for (long long k = i; k < std::min(i + 4, block_of[t + 1]); ++k)
                longest = std::max(longest, (long long)len(t, k));
            const long long p = (longest + 31) / 32;
            packets += p;
            most = std::max(most, p);
        }
    return strips_pay(packets, most, pbytes, entries);
}

}  // namespace suppy

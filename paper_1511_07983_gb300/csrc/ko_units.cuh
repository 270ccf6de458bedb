// Work units of a simulator pass: whole work items, or parts of them.
//
// An exhaustive item (a prefix of d0 kernels) of m = n - d0 kernels can be cut
// by x further kernels into m (m-1) .. (m-x+1) units, each the walk below one
// longer prefix; unit s is the s-th such prefix in lexicographic order, so its
// first order is the item's first plus s (m-x)!.  Two uses:
//   * the last items of a whole-space pass, so that all threads end together
//     instead of waiting for whole items;
//   * passes over abandoned items, which are few: their orders run side by side
//     instead of one after another.
// What both are worth, with abandoned items going to a larger one-thread state
// first: a 10-kernel / 15-SM space 13.9 -> 12.0 ms, an 11-kernel / 148-SM one
// 218 -> 198 ms, 48 mixed sets in one graph 131 -> 105 ms.
// Sets of one launch may differ in m: a pass numbers its units with the factor
// of the largest m, and a unit past its own item's number of parts is skipped.
//
// A list entry of an abandoned unit: item | part << 44 | x << 58.
#pragma once

#include "ko_fast.h"

namespace kounits {

constexpr int kItemBits = 44, kPartBits = 14;
constexpr unsigned long long kItemMask = (1ull << kItemBits) - 1ull, kPartMask = (1ull << kPartBits) - 1ull;

struct Unit {
    unsigned long long item;
    unsigned part;   // lexicographic number of the prefix among the item's
    int x;           // kernels the unit fixes beyond the item's
    bool valid;
};

__host__ __device__ inline unsigned long long entry_of(unsigned long long item, unsigned part, int x)
{
    return item | ((unsigned long long)part << kItemBits) | ((unsigned long long)x << (kItemBits + kPartBits));
}

// Parts of m kernels' orders when x more are fixed (m >= 1).
__host__ __device__ inline unsigned parts(int m, int x)
{
    unsigned f = 1;
    for (int i = 0; i < x && m - i > 1; i++) f *= (unsigned)(m - i);
    return f;
}

// How a pass numbers its units.  Units [0, a) are whole items, the next ones
// parts cut by x1 of the items from `a` to b, the rest parts cut by x2 of the
// items from b on.
struct Numbering {
    unsigned long long a, b, items, units;
    unsigned f1, f2;
    int x1, x2;
};

// A whole-space pass of `threads` simulations: once one whole item is left per
// thread, items are cut by one kernel; once one such part is left, by two.
__host__ __device__ inline Numbering number_space(unsigned long long items, int levels, unsigned long long threads)
{
    Numbering u;
    const int m = levels + 1;
    u.items = items;
    u.x1 = 1;
    u.x2 = 2;
    u.f1 = parts(m, 1);
    u.f2 = parts(m, 2);
    u.a = items > threads ? items - threads : 0ull;
    u.b = items > threads / u.f1 ? items - threads / u.f1 : 0ull;
    u.units = u.a + (u.b - u.a) * u.f1 + (items - u.b) * u.f2;
    return u;
}

// A pass of `threads` simulations over `items` list entries, every one cut as
// far as a thread is left for each part; with `fine`, down to walks of at most
// three kernels (six orders) whatever the threads, or as many of them as there
// is room for by one kernel more than the rest.  `room`, the entries of the
// list the pass writes, bounds the units of any: a pass may abandon all it
// numbers (840 two-level items in 2,520 parts against a list of 1,024 lost
// 2,992 of 5,040 orders).
__host__ __device__ inline Numbering number_list(unsigned long long items, int levels, unsigned long long threads,
                                                 unsigned long long room, bool fine = false)
{
    Numbering u;
    const int m = levels + 1;
    if (threads > room) threads = room;
    u.items = items;
    u.a = u.b = 0ull;
    u.x1 = u.x2 = 0;
    u.f1 = u.f2 = 1;
    while (m - u.x2 > 1 && items * u.f2 * (unsigned)(m - u.x2) <= (m - u.x2 > 3 && fine ? room : threads)) {
        u.f2 *= (unsigned)(m - u.x2);
        u.x2++;
    }
    if (fine && m - u.x2 > 3 && items) {  // the last items one kernel further
        u.x1 = u.x2++;
        u.f1 = u.f2;
        u.f2 *= (unsigned)(m - u.x1);
        u.b = items - (room - items * u.f1) / (u.f2 - u.f1);
    }
    u.units = u.b * u.f1 + (items - u.b) * u.f2;
    return u;
}

// The numbering of a list as single orders, if there are few enough of them (and
// no more than a list holds): run from the start, a warp per order, they take
// 10 to 50 us a thousand, and none is too large for that pass, where walking them in
// 16-lane segments abandons most of what one thread could not hold.
constexpr unsigned long long kSinglesMax = 2ull << 20;
__host__ __device__ inline bool number_singles(unsigned long long items, int levels, unsigned long long room,
                                               Numbering &u)
{
    u = number_list(items, levels, kSinglesMax, room);
    return levels + 1 - u.x2 <= 1;
}

// The item (or list entry) of unit `unit`, the part's number and its cut.
__host__ __device__ inline Unit unit_at(const Numbering &u, unsigned long long unit)
{
    if (unit < u.a) return Unit{unit, 0u, 0, true};
    unit -= u.a;
    const unsigned long long mid = (u.b - u.a) * u.f1;
    if (unit < mid) return Unit{u.a + unit / u.f1, (unsigned)(unit % u.f1), u.x1, true};
    unit -= mid;
    return Unit{u.b + unit / u.f2, (unsigned)(unit % u.f2), u.x2, true};
}

// Cuts an item or an already cut unit (`part`, `x` of an item of m kernels) by
// `cut` more kernels: part number `s` of it, not valid when it has fewer.
__host__ __device__ inline Unit cut_unit(unsigned long long item, unsigned part, int x, int m, int cut, unsigned s)
{
    const int left = m - x;                       // kernels the unit still walks
    if (cut > left) cut = left > 0 ? left : 0;
    const unsigned f = parts(left, cut);
    return Unit{item, part * f + s, x + cut, s < f};
}

#ifdef __CUDACC__
// Record an abandoned unit for the next pass.  Every pass numbers at most as many
// units as its list has entries; one that found its list full all the same is
// counted, and the call's status tells.
__device__ __forceinline__ void hand_on(const KoWork &a, unsigned long long entry)
{
    const unsigned long long slot = atomicAdd(a.ov_count, 1ull);
    if (slot < a.ov_cap) a.ov_list[slot] = entry;
    else atomicAdd(a.lost, 1ull);
}
#endif

}  // namespace kounits

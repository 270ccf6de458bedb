// One simulation per warp, one run of SMs per lane: the pass over short lists of
// explicit orders (and over spaces walked order by order), where the time of a
// single simulation decides.
//
// Same model and runs as the run-length simulator (ko_fast.cu), laid out for a
// short chain of dependent instructions per event:
//   * runs are unordered (a split appends a lane), so a split moves no lanes;
//   * a lane keeps what its SMs have free and the earliest end of its groups in
//     registers and its groups (end, descriptor) in its own column of shared
//     memory, free of bank conflicts; an event reads the column once, in one
//     burst of independent loads, for what ends and for the next end;
//   * between a kernel's first and last burst an event changes only the run
//     whose groups end, and that one takes its full capacity, so every lane has
//     its next event worked out ahead (release, room, the new group's duration)
//     and a turn takes the events of all lanes that come before the earliest
//     one not worked out yet: four warp reductions, three more where several
//     runs end together and decide the pointer.  The joint water-fill runs once
//     per kernel, for the burst that empties the queue.
//   * the slot and descriptor of a lane's next group to end are at hand, so its
//     release does not wait for a look through the column.
// It is bound by instruction latency (570 orders of N=20 on 13 SMs, one warp per
// SM sub-partition: 145 warp instructions per event at 4.2 cycles each, half of
// that waits for the previous instruction; 229 while a turn took one event
// time).  The run-length kernel took 3,200 cycles per event here (its groups in
// registers behind select chains, more reductions per event, lanes shifted by
// every split).  570 orders, us before -> with one event time a turn -> now:
// N=8 on 13 SMs 124 -> 60 -> 55, N=20 on 13 SMs 608 -> 268 -> 185, N=20 on 148
// SMs 573 -> 283 -> 146.
#include "ko_fast.h"
#include "ko_units.cuh"

namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kWarps = 4;        // at most, per block
constexpr int kSlots16 = 16;     // group slots of a run
constexpr int kPosBits = 12;     // a pointer move is 1 .. N_SM <= 1024

__constant__ unsigned long long c_warp_fact[21] = {
    1ull, 1ull, 2ull, 6ull, 24ull, 120ull, 720ull, 5040ull, 40320ull, 362880ull, 3628800ull,
    39916800ull, 479001600ull, 6227020800ull, 87178291200ull, 1307674368000ull,
    20922789888000ull, 355687428096000ull, 6402373705728000ull, 121645100408832000ull,
    2432902008176640000ull};

// One kernel's constants: a block's needs and cycles, blocks, and the reciprocals
// of the needs rounded down (ko_lane_sim.cuh's cap() says why that is exact).
struct __align__(16) WarpKern {
    int r, s, w, c;
    int m, b;
    float frr, frs;
    float frw, fsb;
    int pad0, pad1;
};

struct WarpMem {
    uint32_t end[kSlots16][32];
    uint32_t desc[kSlots16][32];  // kernel | blocks per SM << 5
    WarpKern k[KO_MAX_KERNELS];
};

// a / b for capacities that are no power of two; one copy of the long division.
__device__ __noinline__ uint32_t quotient(unsigned long long a, uint32_t b) { return (uint32_t)(a / b); }

// A lane's run and the simulation's warp-uniform state.
struct WarpSim {
    WarpMem &mem;
    int lane;
    int S;
    uint32_t ccap, mcap;
    int cshift, mshift;
    bool shifts;                    // both capacities are powers of two
    // run
    int beg, cnt, fr, fs, fw, fb;   // SMs; free registers, shared memory, warps, blocks of each
    uint32_t sc, sm, re;            // SumC, SumM, earliest end of its groups (where it has any)
    uint32_t used, pend;            // group slots in use; of groups whose burst is open
    int rslot;                      // the group that ends at re: its slot and descriptor
    uint32_t rdesc;
    // simulation
    unsigned long long t;
    int p, nr;

    __device__ void init(const KoSet *set)
    {
        beg = 0;
        cnt = lane == 0 ? S : 0;
        fr = set->R; fs = set->Sh; fw = set->W; fb = set->Bk;
        sc = sm = re = 0;
        used = pend = 0;
        rslot = 0;
        rdesc = 0;
        t = 0;
        p = 0;
        nr = 1;
    }

    __device__ __forceinline__ int cap(const WarpKern &h) const
    {
        float f = (float)fr * h.frr;
        f = fminf(f, fminf((float)fw * h.frw, (float)fs * h.frs + h.fsb));
        int q = (int)fminf(f, 40.0f);
        if ((q + 1) * h.r <= fr && (q + 1) * h.w <= fw && (q + 1) * h.s <= fs) q++;
        return min(q, fb);
    }

    // Cycles of a block started when its SM's sums are c_sum / m_sum.
    __device__ __forceinline__ uint32_t duration(uint32_t c, uint32_t m, uint32_t c_sum, uint32_t m_sum) const
    {
        const unsigned long long pc = (unsigned long long)c * max(c_sum, ccap) + (ccap - 1u);
        const unsigned long long pm = (unsigned long long)m * max(m_sum, mcap) + (mcap - 1u);
        if (shifts) return max((uint32_t)(pc >> cshift), (uint32_t)(pm >> mshift));
        return max(quotient(pc, ccap), quotient(pm, mcap));
    }

    // q blocks per SM of kernel k as a new group in a slot outside `taken`; the
    // slot, or -1 without one.
    __device__ __forceinline__ int place(const WarpKern &h, int k, int q, uint32_t taken)
    {
        const int g = __ffs((int)(~taken & 0xffffu)) - 1;
        if (g < 0) return -1;
        used |= 1u << g;
        mem.desc[g][lane] = (uint32_t)k | ((uint32_t)q << 5);
        fr -= q * h.r; fs -= q * h.s; fw -= q * h.w; fb -= q;
        sc += (uint32_t)(q * h.c); sm += (uint32_t)(q * h.m);
        return g;
    }

    // Group g (descriptor d), started now, ends after dur.
    __device__ __forceinline__ void start(uint32_t now, int g, uint32_t d, uint32_t dur)
    {
        mem.end[g][lane] = now + dur;
        // the slots besides g decide whether `re` holds an end
        if ((used & ~pend & ~(1u << g)) == 0u || dur < re - now) {
            re = now + dur;
            rslot = g;
            rdesc = d;
        }
    }

    // Durations of the groups whose burst closes now.
    __device__ void close_burst()
    {
        while (__any_sync(kAll, pend != 0u)) {
            if (pend) {
                const int g = __ffs((int)pend) - 1;
                const uint32_t d = mem.desc[g][lane];
                const WarpKern &q = mem.k[d & 31u];
                start((uint32_t)t, g, d, duration((uint32_t)q.c, (uint32_t)q.m, sc, sm));
                pend &= pend - 1u;
            }
        }
    }

    // Release the groups that end now -- the one at rslot and any others -- and
    // find the earliest end of the rest.  The first group's descriptor is at hand
    // since the last time the lane looked, so its constants load while the ends
    // are read.
    __device__ __forceinline__ void release(uint32_t now)
    {
        uint32_t gone = 1u << rslot, d = rdesc, next;
        do {
            const WarpKern &k = mem.k[d & 31u];
            const int q = (int)(d >> 5);
            const int4 a = *reinterpret_cast<const int4 *>(&k);
            const int km = k.m;
            used &= ~gone;
            uint32_t e[8];
#pragma unroll
            for (int g = 0; g < 8; g++) {
                e[g] = mem.end[g][lane] - now;
                if (!((used >> g) & 1u)) e[g] = 0xffffffffu;
            }
            next = min(min(min(e[0], e[1]), min(e[2], e[3])), min(min(e[4], e[5]), min(e[6], e[7])));
            gone = 0;
#pragma unroll
            for (int g = 0; g < 8; g++) gone |= e[g] == next ? 1u << g : 0u;
            if (used >> 8) {
                for (uint32_t m = used >> 8; m; m &= m - 1u) {
                    const int g = __ffs((int)m) + 7;
                    const uint32_t x = mem.end[g][lane] - now;
                    if (x < next) { next = x; gone = 0; }
                    if (x == next) gone |= 1u << g;
                }
            }
            gone &= used;
            gone &= 0u - gone;  // the first of equal ones
            rslot = gone ? __ffs((int)gone) - 1 : 0;
            d = mem.desc[rslot][lane];
            fr += q * a.x; fs += q * a.y; fw += q * a.z; fb += q;
            sc -= (uint32_t)(q * a.w); sm -= (uint32_t)(q * km);
        } while (next == 0u);
        rdesc = d;
        re = now + next;
    }

    // How far past `p` (in SMs, cyclically) the run's last SM lies, 1 .. S.
    __device__ __forceinline__ int last_past(int p) const
    {
        const int d = beg + cnt - p;
        if (beg < p && d > 0) return S;  // p lies inside: its last SM from p on is p - 1
        return d <= 0 ? d + S : d;
    }

    // Lane j keeps the run's first x SMs (0 < x < its count); lane nr takes the rest.
    __device__ void split(int j, int x)
    {
        const int k = nr++;
        __syncwarp();
        if (lane < kSlots16) {
            mem.end[lane][k] = mem.end[lane][j];
            mem.desc[lane][k] = mem.desc[lane][j];
        }
        const int b = __shfl_sync(kAll, beg, j), n = __shfl_sync(kAll, cnt, j);
        const int r = __shfl_sync(kAll, fr, j), s = __shfl_sync(kAll, fs, j), w = __shfl_sync(kAll, fw, j),
                  bl = __shfl_sync(kAll, fb, j);
        const uint32_t c = __shfl_sync(kAll, sc, j), m = __shfl_sync(kAll, sm, j), e = __shfl_sync(kAll, re, j);
        const uint32_t masks = __shfl_sync(kAll, used | (pend << 16), j);
        const uint32_t rd = __shfl_sync(kAll, rdesc, j);
        const int rs = __shfl_sync(kAll, rslot, j);
        if (lane == j) cnt = x;
        if (lane == k) {
            beg = b + x; cnt = n - x;
            fr = r; fs = s; fw = w; fb = bl;
            sc = c; sm = m; re = e;
            used = masks & 0xffffu; pend = masks >> 16;
            rdesc = rd; rslot = rs;
        }
        __syncwarp();
    }

    // The burst that empties the queue: `left` blocks over lanes with room q, of
    // which there is more in all.  Every SM ends with min(room, L - 1) blocks of
    // it and the first ones past p with more room have one more; runs are cut at p
    // and where the last sweep stops.  False if a run or a slot is missing.
    __device__ bool place_last(const WarpKern &h, int kern, int left, int q, int run_limit)
    {
        int lo = 1, hi = (int)__reduce_max_sync(kAll, (unsigned)q);
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((int)__reduce_add_sync(kAll, (unsigned)(cnt * min(q, mid))) >= left) hi = mid; else lo = mid + 1;
        }
        const int rem = left - (int)__reduce_add_sync(kAll, (unsigned)(cnt * min(q, lo - 1)));  // >= 1
        const unsigned inside = __ballot_sync(kAll, q >= lo && beg < p && p < beg + cnt);
        if (inside) {
            if (nr >= run_limit) return false;
            const int j = __ffs((int)inside) - 1, k = nr;
            const int room = __shfl_sync(kAll, q, j);
            split(j, p - __shfl_sync(kAll, beg, j));
            if (lane == k) q = room;
        }
        // the runs with room in the last sweep, in cyclic order from p: SMs before this one
        const bool in = q >= lo && cnt > 0;
        const int e = in ? cnt : 0;
        int d = beg - p;
        if (d < 0) d += S;
        int before = 0;
        for (unsigned m = __ballot_sync(kAll, in); m; m &= m - 1u) {
            const int j = __ffs((int)m) - 1;
            const int dj = __shfl_sync(kAll, d, j), ej = __shfl_sync(kAll, e, j);
            if (dj < d) before += ej;
        }
        int give = min(q, lo - 1) + (in && before < rem ? 1 : 0);
        const unsigned here = __ballot_sync(kAll, in && before < rem && rem <= before + e);
        const int star = __ffs((int)here) - 1;  // exactly one: 1 <= rem <= SMs with room
        const int x = rem - __shfl_sync(kAll, before, star);
        p = __shfl_sync(kAll, beg, star) + x;
        if (p >= S) p -= S;
        if (x < __shfl_sync(kAll, cnt, star)) {
            if (nr >= run_limit) return false;
            const int k = nr;
            const int room = __shfl_sync(kAll, give, star);
            split(star, x);
            if (lane == k) give = room - 1;
        }
        bool ok = true;
        if (give > 0) {
            const int g = place(h, kern, give, used);
            ok = g >= 0;
            if (ok) pend |= 1u << g;
        }
        return __all_sync(kAll, ok);
    }

    // Every lane takes its room q: p moves past the last SM with the most.  False
    // if a lane has no slot.
    __device__ __forceinline__ bool move_pointer(int q)
    {
        unsigned key = q > 0 ? ((unsigned)q << kPosBits) | (unsigned)last_past(p) : 0u;
        if (q > 0 && used == 0xffffu) key = 0xffffffffu;
        const unsigned top = __reduce_max_sync(kAll, key);
        p += (int)(top & ((1u << kPosBits) - 1u));
        if (p >= S) p -= S;
        return top != 0xffffffffu;
    }

    // p after a burst in which lanes with key > 0 placed: past the last SM of those
    // with the largest key.  p always lies where a run begins (it is set to the end
    // of a run, and runs only ever split), so one such lane alone decides it;
    // -1 where several do and `from`, the pointer before, is not known (< 0).
    __device__ __forceinline__ int pointer_after(unsigned key, int from) const
    {
        const unsigned top = __reduce_max_sync(kAll, key);
        const unsigned who = __ballot_sync(kAll, key == top);
        if ((who & (who - 1u)) == 0u) {
            const int end = __shfl_sync(kAll, beg + cnt, __ffs((int)who) - 1);
            return end >= S ? end - S : end;
        }
        if (from < 0) return -1;
        const int to = from + (int)__reduce_max_sync(kAll, key == top ? (unsigned)last_past(from) : 0u);
        return to >= S ? to - S : to;
    }

    // The state a run has after its next event, worked out ahead of time.
    struct Ahead {
        int fr, fs, fw, fb;
        uint32_t sc, sm, re, used, rdesc;
        int rslot;
        int q;   // blocks per SM it takes
    };

    // The run's next event: releases at `re`, room for the head kernel, the new
    // group.  The run itself stays as it is; the new group may go to the released
    // group's slot (put_back() restores that one) or a free one.
    __device__ __forceinline__ void look_ahead(const WarpKern &h, int kern, Ahead &a)
    {
        const Ahead was{fr, fs, fw, fb, sc, sm, re, used, rdesc, rslot, 0};
        release(was.re);
        const int q = cap(h);
        if (q > 0) {
            const int g = place(h, kern, q, used | (was.used & ~(1u << was.rslot)));
            start(was.re, g, (uint32_t)kern | ((uint32_t)q << 5), duration((uint32_t)h.c, (uint32_t)h.m, sc, sm));
        }
        a = Ahead{fr, fs, fw, fb, sc, sm, re, used, rdesc, rslot, q};
        set(was);
    }
    __device__ __forceinline__ void set(const Ahead &a)
    {
        fr = a.fr; fs = a.fs; fw = a.fw; fb = a.fb;
        sc = a.sc; sm = a.sm; re = a.re; used = a.used; rdesc = a.rdesc;
        rslot = a.rslot;
    }
    __device__ __forceinline__ void put_back()
    {
        mem.end[rslot][lane] = re;
        mem.desc[rslot][lane] = rdesc;
    }

    // Queue all blocks of kernel `kern` behind the current queue and simulate until
    // the last of them is placed (its burst stays open).  False if the state
    // cannot hold it.
    //
    // Between the kernel's first burst and the one that empties the queue a run's
    // events depend on no other run, so every lane has its next event worked out,
    // and a turn takes, of all runs side by side, the next events before the
    // earliest event that is not worked out yet -- if the queue is longer than what
    // they take.
    __device__ bool place_kernel(int kern, int limit, int run_limit)
    {
        const WarpKern h = mem.k[kern];
        int left = h.b;
        {   // the first burst continues the open one: every run is offered the kernel
            const int q = cnt > 0 ? cap(h) : 0;
            const int total = (int)__reduce_add_sync(kAll, (unsigned)(q * cnt));
            if (total > left) return place_last(h, kern, left, q, run_limit);
            if (!move_pointer(q)) return false;
            left -= total;
            if (q > 0) pend |= 1u << place(h, kern, q, used);
            if (left == 0) return true;
            close_burst();
        }
        Ahead a{};
        if (used) look_ahead(h, kern, a);
        __syncwarp();
        for (int it = 0; it < limit; it++) {
            const uint32_t now = (uint32_t)t, none = 0xffffffffu;
            const uint32_t e1 = used ? re - now : none, e2 = used && a.used ? a.re - now : none;
            const uint32_t bound = __reduce_min_sync(kAll, e2);
            bool in = e1 < bound;
            const int take = a.q * cnt;
            int total = (int)__reduce_add_sync(kAll, in ? (unsigned)take : 0u);
            uint32_t adv = __reduce_max_sync(kAll, in ? e1 : 0u);
            int to = p;
            if (total > 0 && total < left) {
                // the pointer: the last of these bursts decides, with the one before it
                // where several runs end together
                const uint32_t at = in && a.q > 0 ? e1 : 0u;
                const uint32_t last = __reduce_max_sync(kAll, at);
                const unsigned key = at == last ? (unsigned)a.q : 0u;
                to = pointer_after(key, -1);
                if (to < 0) {
                    const uint32_t prev = at == last ? 0u : at;
                    const uint32_t before = __reduce_max_sync(kAll, prev);
                    const int from = before ? pointer_after(prev == before ? (unsigned)a.q : 0u, -1) : p;
                    if (from >= 0) to = pointer_after(key, from);
                }
            }
            if (total >= left || to < 0) {  // the earliest end alone
                adv = __reduce_min_sync(kAll, e1);
                in = e1 == adv && used != 0u;
                total = (int)__reduce_add_sync(kAll, in ? (unsigned)take : 0u);
                if (total >= left) {        // the queue runs empty
                    if (used) put_back();
                    t += adv;
                    if (in) release((uint32_t)t);
                    __syncwarp();
                    const int q = in ? cap(h) : 0;
                    if (total > left) return place_last(h, kern, left, q, run_limit);
                    if (!move_pointer(q)) return false;
                    if (q > 0) pend |= 1u << place(h, kern, q, used);
                    return true;
                }
                to = total > 0 ? pointer_after(in ? (unsigned)a.q : 0u, p) : p;
            }
            if (!__any_sync(kAll, in)) return false;  // nothing runs: not reached
            p = to;
            t += adv;
            left -= total;
            if (in) {
                set(a);
                if (used) look_ahead(h, kern, a);
            }
            __syncwarp();
        }
        return false;  // each event frees a block: not reached
    }

    // Close the last burst; the makespan is the latest end.
    __device__ unsigned long long finish()
    {
        close_burst();
        const uint32_t now = (uint32_t)t;
        uint32_t last = 0;
#pragma unroll
        for (int g = 0; g < kSlots16; g++)
            if ((used >> g) & 1u) last = max(last, mem.end[g][lane] - now);
        return t + __reduce_max_sync(kAll, last);
    }
};

__global__ void __launch_bounds__(kWarps * 32) warp_kernel(KoWork a)
{
    __shared__ WarpMem mems[kWarps];
    const int lane = threadIdx.x & 31;
    WarpSim sim{mems[threadIdx.x >> 5], lane};
    const int run_limit = a.run_limit < 32 ? a.run_limit : 32;
    int loaded = -1, n = 0, limit = 0;
    const KoSet *set = nullptr;
    kounits::Numbering units{};
    if (a.item_list) {
        const unsigned long long have = *a.item_count < a.ov_cap ? *a.item_count : a.ov_cap;
        if (!kounits::number_singles(have, a.space ? a.levels : 0, a.ov_cap, units)) return;  // the next pass walks them
    } else {
        units.units = (unsigned long long)a.n_items;
    }
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(a.counter, 1ull);
        item = __shfl_sync(kAll, item, 0);
        if (item >= units.units) break;
        unsigned part = 0, list_part = 0;
        int cut = 0, list_cut = 0;
        if (a.item_list) {
            const kounits::Unit un = kounits::unit_at(units, item);
            const unsigned long long entry = a.item_list[un.item];
            item = entry & kounits::kItemMask;
            list_part = (unsigned)((entry >> kounits::kItemBits) & kounits::kPartMask);
            list_cut = (int)(entry >> (kounits::kItemBits + kounits::kPartBits));
            part = un.part;
            cut = un.x;
            if (item >= (unsigned long long)a.n_items) continue;
        }
        int lo = 0, hi = a.nchunks - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.chunks[mid].first <= (long long)item) lo = mid; else hi = mid - 1;
        }
        const KoChunk ch = a.chunks[lo];
        if (a.item_list) {
            const kounits::Unit un =
                kounits::cut_unit(item, list_part, list_cut, ch.mode == 0 ? a.sets[ch.set].n - ch.d0 : 0, cut, part);
            if (!un.valid) continue;
            part = un.part;
            cut = un.x;
        }
        if (ch.set != loaded) {
            loaded = ch.set;
            set = a.sets + ch.set;
            n = set->n;
            int blocks = 0;
            __syncwarp();
            if (lane < n) {
                const KoKern k = set->k[lane];
                const float down = 1.0f - 1.0f / 262144.0f;
                blocks = k.b;
                sim.mem.k[lane] = WarpKern{k.r, k.s, k.w, k.c, k.m, k.b, __fdividef(down, (float)k.r),
                                           k.s > 0 ? __fdividef(down, (float)k.s) : 0.0f,
                                           __fdividef(down, (float)k.w), k.s > 0 ? 0.0f : 40.0f, 0, 0};
            }
            limit = (int)__reduce_add_sync(kAll, (unsigned)blocks) + 64;
            sim.S = set->S;
            sim.ccap = (uint32_t)set->ccap; sim.mcap = (uint32_t)set->mcap;
            sim.cshift = set->cshift; sim.mshift = set->mshift;
            sim.shifts = set->cshift >= 0 && set->mshift >= 0;
            __syncwarp();
        }
        // lane d holds the kernel at position d
        const long long local = (long long)item - ch.first;
        long long outpos = ch.out_off + local;
        int mine = -1;
        bool valid = true;
        if (ch.mode == 2) {
            const int8_t *row = a.perms + ch.list_off + local * (a.perm_stride ? a.perm_stride : n);
            const int v = lane < n ? row[lane] : 0;
            const bool range = lane >= n || (v >= 0 && v < n);
            const unsigned seen = __reduce_or_sync(kAll, lane < n && range ? 1u << v : 0u);
            valid = __all_sync(kAll, range) && seen == (n < 32 ? (1u << n) - 1u : kAll);
            mine = v;
        } else {
            // a Lehmer index; a prefix of all kernels but one leaves no choice either
            unsigned long long k;
            if (ch.mode == 1) {
                k = a.idx[ch.list_off + local];
                valid = k < c_warp_fact[n];
            } else {
                k = (unsigned long long)(ch.list_off + local) * c_warp_fact[n - ch.d0] +
                    part * c_warp_fact[n - ch.d0 - cut];
                outpos = ch.out_off + (long long)k;
            }
            unsigned rest = (1u << n) - 1u;
            for (int d = 0; valid && d < n; d++) {
                const unsigned long long f = c_warp_fact[n - 1 - d];
                const unsigned digit = (unsigned)(k / f);
                k -= (unsigned long long)digit * f;
                unsigned u = rest;
                for (unsigned q = 0; q < digit; q++) u &= u - 1u;
                const int v = __ffs((int)u) - 1;
                rest &= ~(1u << v);
                if (lane == d) mine = v;
            }
        }
        if (!valid) {
            if (lane == 0 && a.out) a.out[outpos] = -1;
            continue;
        }
        sim.init(set);
        bool ok = true;
        for (int d = 0; ok && d < n; d++) ok = sim.place_kernel(__shfl_sync(kAll, mine, d), limit, run_limit);
        if (!ok) {
            if (lane == 0) {
                kounits::hand_on(a, kounits::entry_of(item, part, cut));
                if (!a.item_list) atomicAdd(a.abandoned, 1ull);
            }
            continue;
        }
        const unsigned long long ms = sim.finish();
        if (lane == 0) {
            if (a.out) a.out[outpos] = (int64_t)ms;
            if (a.accs) {
                KoAccum *acc = a.accs + ch.set;
                const unsigned long long ref = (unsigned long long)(a.refs ? a.refs[ch.set] : set->ref_makespan);
                atomicMin(&acc->min, ms);
                atomicMax(&acc->max, ms);
                atomicAdd(ms < ref ? &acc->n_better : ms == ref ? &acc->n_equal : &acc->n_worse, 1ull);
            }
        }
    }
}

}  // namespace

cudaError_t ko_launch_warp(const KoWork &a, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // as few warps per block as give every warp one order, up to one per sub-partition.  A list's
    // length is not known here: its pass gets the warps that are resident at once (96 registers a
    // thread: 5 blocks per SM; an empty list costs no more than with one).  100,003 orders that the
    // one-thread pass hands on for their set's limits, us with one block per SM / with five: N=8 on
    // 13 SMs 3520 / 1048, N=12 on 148 SMs 7280 / 2267; in 16 lanes 2081 and 5889
    const long long work = a.item_list ? (long long)sms * 5 * kWarps : a.n_items;
    const long long per_sm = (work + sms - 1) / sms;
    const int warps = per_sm < 1 ? 1 : per_sm < kWarps ? (int)per_sm : kWarps;
    long long blocks = (work + warps - 1) / warps;
    const long long resident = (long long)sms * 8;
    if (blocks > resident) blocks = resident;
    if (blocks < 1) blocks = 1;
    warp_kernel<<<(unsigned)blocks, warps * 32, 0, st>>>(a);
    ko_count_launch();
    return cudaGetLastError();
}

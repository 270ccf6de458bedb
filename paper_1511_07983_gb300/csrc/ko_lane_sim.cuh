// One simulation per thread: the block-dispatch model (Sec. 2 dispatch rule,
// durations fixed at burst end from the SM's SumC / SumM) advanced by a single
// thread, one run of SMs at a time.
//
// State.  SMs with identical state form a run of consecutive SM indices; the
// runs themselves are kept in no particular order (a split appends the new run).
// A run holds usage (registers, blocks and warps packed in one word, shared
// memory, SumC, SumM), the earliest end of its groups, and a list of up to ten
// 6-bit slot numbers into a pool of groups, sorted by end.  A group is the
// blocks of one kernel started in one burst on every SM of a run (kernel,
// blocks per SM, end).  When a run splits, both halves list the groups already
// started; a group that is still pending (its burst is open) is copied to a
// new slot for the new half, so each pending group has exactly one owner run,
// whose SumC / SumM fixes its duration when the burst closes.
//
// Events.  Between a kernel's first and last burst the queue holds more blocks
// than any event frees room for, so a run whose groups end takes its full
// capacity whatever the other runs do: event() takes ONE run per call --
// release, capacity, placement and durations of that run alone -- also when
// several runs end at the same time (the rest wait in `todo`).  Only the burst
// that would empty the queue needs all its runs together: event() then reports
// the last burst, and place_partial() releases the runs still in `todo`, takes
// back what the burst had placed and fills all of them jointly.  A step without
// loops over runs keeps the 32 simulations of a warp in step.
//
// What bounds it: instruction issue at the lanes that are active (a warp's
// threads wait for each other at the control step) and the latency of nine
// warps per SM; it moves no data to speak of.  The loops over released runs
// and their slots that an event step had before made a warp run as long as its
// worst thread.  All 39.9M orders of an 11-kernel / 148-SM set: 470 ms with the
// looping event step over ordered runs, 260 ms with this one, 184 with a kernel's
// first burst and the close of a burst as such steps too; 3.6M orders of a
// ten-kernel / 15-SM set 31.9 -> 22.6 -> 15.3 ms.
//
// Measured on the N=12 / 148-SM set: about 11 runs and 34 groups live, 1.24
// runs released per event, 34 events per order, a split every 15 events.  56
// slots hold every group of about 99 % of the 120-order work items; the rest
// move on to other passes.
//
// Layout.  The state of one simulation is a column of kWords 32-bit words in
// shared memory, word f of the thread's column at col[f * STRIDE]; with STRIDE
// = the block's thread count (a multiple of 32) every access of a warp is free
// of bank conflicts whatever run or slot each thread touches.  Registers hold
// the clock, the round-robin pointer, the number of runs, the free and pending
// slot masks and the head kernel's constants.
//
// Time.  Ends are 32-bit values modulo 2^32 beside a 64-bit clock; the host
// uses this path only when every possible duration is below 2^31, so every
// comparison of (end - now) is exact.
#pragma once

#include <stdint.h>

#ifndef KO_HD
#define KO_HD __host__ __device__ __forceinline__
#endif

// Reconvergence point of the threads in `mask` (device only).
#ifdef __CUDA_ARCH__
#define KO_RECONVERGE(mask) __syncwarp(mask)
#else
#define KO_RECONVERGE(mask) ((void)(mask))
#endif

namespace kolane {

// State shape of one simulation: RUNS runs and POOL group slots, laid out as
// the column words below.  Smaller shapes let more simulations share an SM's
// shared memory; a work item that needs more is handed on (see LaneSim).
template <int RUNS, int POOL>
struct Shape {
    static_assert(RUNS <= 16 && POOL <= 62 && POOL % 2 == 0, "run masks are 32 bits; slot 63 marks an empty list entry");
    static constexpr int kRuns = RUNS;   // runs one simulation may hold
    static constexpr int kPool = POOL;   // group slots of one simulation
    static constexpr unsigned long long kPoolAll = (1ull << POOL) - 1ull;
    static constexpr int W_RB = 0;                 // run: first SM | SM count << 11 | capacity at the last offer << 22
    static constexpr int W_RU = W_RB + RUNS;       // run: registers | blocks << 19 | warps << 25 in use per SM
    static constexpr int W_RS = W_RU + RUNS;       // run: shared memory in use per SM
    static constexpr int W_RC = W_RS + RUNS;       // run: SumC
    static constexpr int W_RM = W_RC + RUNS;       // run: SumM
    static constexpr int W_RE = W_RM + RUNS;       // run: earliest end of its listed groups (where it lists any)
    static constexpr int W_L0 = W_RE + RUNS;       // run: its listed groups' slots in order of end, low word
    static constexpr int W_L1 = W_L0 + RUNS;       // run: high word
    static constexpr int W_GE = W_L1 + RUNS;       // slot: end (mod 2^32)
    static constexpr int W_GD = W_GE + POOL;       // slots 2w, 2w+1: 16-bit descriptors
    static constexpr int kWords = W_GD + POOL / 2; // 8 words per run, 1.5 per slot
    static constexpr int kSaveWords = kWords + 8;  // with the registers of a node state
    static_assert(kWords % 4 == 0, "node states are copied in 16-byte pieces");
};
// The shapes the one-thread simulator is built for: 14 runs / 56 slots (196
// words), 12 / 40 (156 words), 10 / 32 (128 words).
using ShapeL = Shape<14, 56>;
using ShapeM = Shape<12, 40>;
using ShapeS = Shape<10, 32>;

// Descriptor: kernel (bits 0-4) | blocks per SM - 1 (bits 5-10) | owner run (bits 11-14).
constexpr uint32_t kDescKernel = 31u, kDescOwnerShift = 11;
// Packed usage word: registers in bits 0-18, blocks 19-24, warps 25-31.
constexpr uint32_t kRegMask = (1u << 19) - 1u;
// Slot lists: ten 6-bit entries from bit 0 of a 64-bit word, 63 = none; bits 60-63 stay set.
constexpr int kListBits = 6, kListLen = 10;
constexpr uint32_t kNoSlot = 63u;

// Run word: N_SM <= 1024, so a first SM and a count take 11 bits each.
constexpr uint32_t kSmMask = 0x7ffu;
constexpr int kCntShift = 11, kCapShift = 22;
constexpr uint32_t kSpanMask = (1u << kCapShift) - 1u;

// Registers saved with a node state (beside the column words).
constexpr int kRegWords = 8;

// a / b for capacities that are no power of two; one copy of the long division.
#ifdef __CUDACC__
static __host__ __device__ __noinline__ uint32_t quotient(unsigned long long a, uint32_t b)
#else
static inline uint32_t quotient(unsigned long long a, uint32_t b)
#endif
{
    return (uint32_t)(a / b);
}

// The set's limits, per thread.
struct Limits {
    int n, S, R, Sh, W, Bk;
    uint32_t ccap, mcap;
    int cshift, mshift;
};

KO_HD int ffs64(unsigned long long v)
{
#ifdef __CUDA_ARCH__
    return __ffsll((long long)v) - 1;
#else
    return __builtin_ffsll((long long)v) - 1;
#endif
}
KO_HD int ffs32(uint32_t v)
{
#ifdef __CUDA_ARCH__
    return __ffs((int)v) - 1;
#else
    return __builtin_ffs((int)v) - 1;
#endif
}

// Kernel constants a simulation looks up by kernel id: all of them, and the
// packed record the release and duration steps read (one 16-byte load).
struct KParam {
    int r, s, w, b, c, m;
};
struct KRel {
    uint32_t pk;   // registers | 1 << 19 | warps << 25: one block's share of the usage word
    uint32_t s, c, m;
};

template <int STRIDE, class KLoad, class SH>
struct LaneSim {
    static constexpr int kRuns = SH::kRuns, kPool = SH::kPool, kWords = SH::kWords;
    static constexpr unsigned long long kPoolAll = SH::kPoolAll;
    static constexpr int W_RB = SH::W_RB, W_RU = SH::W_RU, W_RS = SH::W_RS, W_RC = SH::W_RC, W_RM = SH::W_RM,
                         W_RE = SH::W_RE, W_L0 = SH::W_L0, W_L1 = SH::W_L1, W_GE = SH::W_GE, W_GD = SH::W_GD;
    uint32_t *col;            // word f at col[f * STRIDE]
    KLoad kl;                 // kernel constants by id
    Limits L;
    unsigned long long t;      // clock
    unsigned long long freeg;  // free pool slots
    unsigned long long rel;    // slots released at t, free once every run ending at t is released
    unsigned long long pend;   // slots of groups started at t that are not listed yet (burst open)
    unsigned long long placed; // slots event() started and listed in this burst, for the head kernel
    int p;                     // round-robin pointer (an SM index) when the burst began
    int nr;                    // runs
    int run_limit;
    int fail;
    uint32_t fresh, todo;      // runs the burst offers the head kernel; those event() has not taken yet
    int ends;                  // the runs in `fresh` have groups ending at t (0: the kernel's first burst)
    int drain;                 // the burst empties the queue: runs in `todo` are released, not filled
    int pmax, pbest;           // event()'s placements at t: largest capacity, and how far past p its
                               // cyclically last SM lies (what the pointer moves by when t passes)
    uint32_t tail, dburst;     // latest end of the groups listed before t, and of those listed at t, minus t
    // head kernel
    int hk, hr, hs, hw, hc, hm;
    uint32_t hpk;             // registers | 1 << 19 | warps << 25
    float frr, frs, frw, fsb; // reciprocals of registers, shared memory, warps (rounded down)

    KO_HD uint32_t &W(int f) const { return col[f * STRIDE]; }
#ifdef __CUDA_ARCH__
    KO_HD uint32_t gd(int g) const
    {
        return reinterpret_cast<const uint16_t *>(col + (W_GD + (g >> 1)) * STRIDE)[g & 1];
    }
    KO_HD void set_gd(int g, uint32_t v) const
    {
        reinterpret_cast<uint16_t *>(col + (W_GD + (g >> 1)) * STRIDE)[g & 1] = (uint16_t)v;
    }
#else
    KO_HD uint32_t gd(int g) const { return (W(W_GD + (g >> 1)) >> ((g & 1) * 16)) & 0xffffu; }
    KO_HD void set_gd(int g, uint32_t v) const
    {
        uint32_t &x = W(W_GD + (g >> 1));
        const int sh = (g & 1) * 16;
        x = (x & ~(0xffffu << sh)) | (v << sh);
    }
#endif
    KO_HD unsigned long long list(int j) const
    {
        return (unsigned long long)W(W_L0 + j) | ((unsigned long long)W(W_L1 + j) << 32);
    }
    KO_HD void set_list(int j, unsigned long long l) const
    {
        W(W_L0 + j) = (uint32_t)l;
        W(W_L1 + j) = (uint32_t)(l >> 32);
    }
    // the list without its first entry
    KO_HD static unsigned long long pop(unsigned long long l) { return (l >> kListBits) | (0x3full << 58); }

    KO_HD void init()
    {
        W(W_RB) = (uint32_t)L.S << kCntShift;
        W(W_RU) = 0; W(W_RS) = 0; W(W_RC) = 0; W(W_RM) = 0;
        set_list(0, ~0ull);
        nr = 1;
        t = 0;
        p = 0;
        freeg = kPoolAll;
        pend = 0;
        tail = 0;
        settle();
    }

    // No burst in progress beyond the pending groups (a node state's registers).
    KO_HD void settle()
    {
        rel = placed = 0;
        fresh = todo = 0;
        ends = drain = 0;
        pmax = pbest = 0;
        dburst = 0;
        fail = 0;
    }

    KO_HD void set_head(int k)
    {
        const KParam q = kl.full(k);
        hk = k; hr = q.r; hs = q.s; hw = q.w; hc = q.c; hm = q.m;
        hpk = (uint32_t)q.r | (1u << 19) | ((uint32_t)q.w << 25);
        // A quotient of at most 40 estimated with one of these lies within 1 below the true one and
        // never above it: the reciprocal, the conversion and the product each err by less than 2^-21
        // relative, and the factor takes 2^-18 off (cap() corrects the estimate exactly).
        const float down = 1.0f - 1.0f / 262144.0f;
#ifdef __CUDA_ARCH__
        frr = __fdividef(down, (float)q.r);
        frw = __fdividef(down, (float)q.w);
        frs = q.s > 0 ? __fdividef(down, (float)q.s) : 0.0f;
#else
        frr = down / (float)q.r;
        frw = down / (float)q.w;
        frs = q.s > 0 ? down / (float)q.s : 0.0f;
#endif
        fsb = q.s > 0 ? 0.0f : 40.0f;  // no shared memory: that limit never binds
    }

    // Blocks of the head kernel an SM with usage u / us still takes: the least
    // quotient of free resources, estimated in floating point and raised by one
    // where one block more fits all of them.  At most 32 (the block limit).
    KO_HD int cap(uint32_t u, uint32_t us) const
    {
        const int xr = L.R - (int)(u & kRegMask), xw = L.W - (int)(u >> 25), xs = L.Sh - (int)us;
        const int xb = L.Bk - (int)((u >> 19) & 63u);
        float f = (float)xr * frr;
        const float fw = (float)xw * frw, fs = (float)xs * frs + fsb;
        f = fw < f ? fw : f;
        f = fs < f ? fs : f;
        f = f < 40.0f ? f : 40.0f;
        int q = (int)f;
        if ((q + 1) * hr <= xr && (q + 1) * hw <= xw && (q + 1) * hs <= xs) q++;
        return q < xb ? q : xb;
    }

    KO_HD uint32_t duration(uint32_t c, uint32_t m, uint32_t sc, uint32_t sm) const
    {
        // every factor fits 32 bits (c, m <= 2^24; SumC, SumM < 2^30; caps <= 2^30), so each
        // product is one 32 x 32 -> 64-bit multiply; every duration is below 2^31
        const uint32_t scc = sc > L.ccap ? sc : L.ccap, smm = sm > L.mcap ? sm : L.mcap;
        const unsigned long long pc = (unsigned long long)c * scc + (L.ccap - 1u);
        const unsigned long long pm = (unsigned long long)m * smm + (L.mcap - 1u);
        const uint32_t dc = L.cshift >= 0 ? (uint32_t)(pc >> L.cshift) : quotient(pc, L.ccap);
        const uint32_t dm = L.mshift >= 0 ? (uint32_t)(pm >> L.mshift) : quotient(pm, L.mcap);
        return dc > dm ? dc : dm;
    }

    // Insert slot g, which ends at t + dur, into list l in order of end (after
    // equal ends); `first` tells whether it became the earliest.  Ends are read
    // four at a time, so the loads of a turn overlap.
    KO_HD unsigned long long insert(unsigned long long l, int g, uint32_t dur, bool &first)
    {
        const uint32_t t32 = (uint32_t)t;
        if (((l >> (kListBits * (kListLen - 1))) & 63u) != kNoSlot) fail = 1;  // full: the item is handed on
        int pos = 0;
        unsigned long long rest = l;
        for (;;) {
            int in = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
            for (int i = 0; i < 4; i++) {
                const uint32_t s = (uint32_t)(rest >> (kListBits * i)) & 63u;
                const uint32_t e = W(W_GE + (int)(s < (uint32_t)kPool ? s : 0u)) - t32;
                in += (s != kNoSlot && e <= dur) ? 1 : 0;
            }
            pos += in;
            if (in < 4) break;  // at most three turns: entries past the tenth read as none
            rest = (rest >> (4 * kListBits)) | (~0ull << (64 - 4 * kListBits));
        }
        first = pos == 0;
        const unsigned long long below = (1ull << (kListBits * pos)) - 1ull;
        return (l & below) | ((unsigned long long)g << (kListBits * pos)) | ((l & ~below) << kListBits) | (0xfull << 60);
    }

    // A free slot for q blocks per SM of the head kernel on run j (freeg != 0).
    KO_HD int take_slot(int j, int q)
    {
        const int g = ffs64(freeg);
        freeg &= freeg - 1;
        set_gd(g, (uint32_t)hk | ((uint32_t)(q - 1) << 5) | ((uint32_t)j << kDescOwnerShift));
        return g;
    }

    // Start q blocks per SM of the head kernel on run j as a new pending group.
    KO_HD void add_group(int j, int q)
    {
        if (freeg == 0) { fail = 1; return; }
        pend |= 1ull << take_slot(j, q);
        W(W_RU + j) += (uint32_t)q * hpk;
        W(W_RS + j) += (uint32_t)(q * hs);
        W(W_RC + j) += (uint32_t)(q * hc);
        W(W_RM + j) += (uint32_t)(q * hm);
    }

    // Split run j after x SMs (0 < x < its count): run j keeps the first x, the
    // new run `nr` takes the rest.
    KO_HD void split(int j, int x)
    {
        if (nr >= run_limit) { fail = 1; return; }
        const int k = nr++;
        const uint32_t rb = W(W_RB + j);
        W(W_RB + j) = (rb & ~(kSmMask << kCntShift)) | ((uint32_t)x << kCntShift);
        W(W_RB + k) = rb + (uint32_t)x - ((uint32_t)x << kCntShift);
        W(W_RU + k) = W(W_RU + j);
        W(W_RS + k) = W(W_RS + j);
        W(W_RC + k) = W(W_RC + j);
        W(W_RM + k) = W(W_RM + j);
        W(W_RE + k) = W(W_RE + j);
        W(W_L0 + k) = W(W_L0 + j);
        W(W_L1 + k) = W(W_L1 + j);
        // run j's pending groups: the new run gets its own copies
        for (unsigned long long pm = pend; pm; pm &= pm - 1) {
            const uint32_t d = gd(ffs64(pm));
            if ((int)(d >> kDescOwnerShift) == j) {
                if (freeg == 0) fail = 1;
                else {
                    const int g2 = ffs64(freeg);
                    freeg &= freeg - 1;
                    pend |= 1ull << g2;
                    set_gd(g2, (d & ((1u << kDescOwnerShift) - 1u)) | ((uint32_t)k << kDescOwnerShift));
                }
            }
        }
    }

    // How far past p (in SMs, cyclically) the last SM of the run rb lies, 1..S.
    KO_HD int last_past(uint32_t rb) const
    {
        const int b = (int)(rb & kSmMask), d = b + (int)((rb >> kCntShift) & kSmMask) - p;
        if (b < p && d > 0) return L.S;  // p lies inside: its last SM from p on is p - 1
        return d <= 0 ? d + L.S : d;
    }

    KO_HD void move_pointer(int by)
    {
        p += by;
        if (p >= L.S) p -= L.S;
    }

    // A run's state while a step works on it.
    struct RunState {
        uint32_t u, s, c, m, re;
        unsigned long long l;
    };

    // Release the groups of the run that end at t.
    KO_HD void release(RunState &r)
    {
        const uint32_t now = (uint32_t)t;
        for (;;) {
            const uint32_t s0 = (uint32_t)r.l & 63u;
            const int g = (int)(s0 < (uint32_t)kPool ? s0 : 0u);  // a run released here lists a group
            const uint32_t d = gd(g);
            const KRel q = kl.rel((int)(d & kDescKernel));
            r.l = pop(r.l);
            const uint32_t nx = (uint32_t)r.l & 63u;
            const bool more = nx != kNoSlot;
            r.re = W(W_GE + (int)(more ? nx : 0u));
            const uint32_t nb = ((d >> 5) & 63u) + 1u;
            r.u -= nb * q.pk;
            r.s -= nb * q.s;
            r.c -= nb * q.c;
            r.m -= nb * q.m;
            rel |= 1ull << g;
            if (!more || r.re != now) break;
        }
    }

    // Jump to the earliest end of a run.  While blocks are queued and the burst
    // is closed every run lists a group (an empty SM takes a block of any
    // kernel), so every run's earliest end is valid.
    KO_HD void advance()
    {
        const uint32_t t32 = (uint32_t)t;
        uint32_t e[kRuns];
        uint32_t dmin = 0xffffffffu;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int j = 0; j < kRuns; j++) {
            e[j] = 0xffffffffu;
            if (j < nr) e[j] = W(W_RE + j) - t32;
            dmin = e[j] < dmin ? e[j] : dmin;
        }
        fresh = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int j = 0; j < kRuns; j++)
            if (e[j] == dmin) fresh |= 1u << j;
        t += dmin;
        tail = (tail > dburst ? tail : dburst) - dmin;
        dburst = 0;
        todo = fresh;
        ends = 1;
        placed = 0;
        move_pointer(pbest);
        pmax = pbest = 0;
    }

    // Queue all blocks of kernel k behind the current queue: its first burst
    // offers it the runs with room for one block (four compares; every other
    // run is skipped), which event() then takes one by one.  Returns the blocks
    // queued.
    KO_HD int begin_kernel(int k)
    {
        set_head(k);
        uint32_t room = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int j = 0; j < kRuns; j++) {
            if (j < nr) {
                const uint32_t u = W(W_RU + j);
                const bool fits = (int)((u >> 19) & 63u) < L.Bk && (int)(u & kRegMask) + hr <= L.R &&
                                  (int)(u >> 25) + hw <= L.W && (int)W(W_RS + j) + hs <= L.Sh;
                room |= (fits ? 1u : 0u) << j;
            }
        }
        fresh = todo = room;
        ends = 0;
        placed = 0;
        return kl.full(k).b;
    }

    // One step while the head kernel has queued blocks, for one run:
    //   a run of the burst in progress (`todo`): release what ends, place the
    //     head kernel's full capacity and list the new group;
    //   none left: list one group that was pending when the kernel's first
    //     burst began (its run's SumC / SumM are final now);
    //   neither: the next event begins.
    // Returns true when this burst empties the queue; the caller finishes it
    // with place_partial.  `mask`: the threads of the warp that run this step
    // together; they reconverge after each stage.
    KO_HD bool event(int &left, unsigned mask)
    {
        if (todo == 0 && pend == 0) advance();
        KO_RECONVERGE(mask);
        const bool listing = todo == 0;
        int g = 0, j;
        uint32_t kc = (uint32_t)hc, km = (uint32_t)hm;
        if (listing) {
            g = ffs64(pend);
            pend &= pend - 1;
            const uint32_t d = gd(g);
            j = (int)(d >> kDescOwnerShift);
            const KRel q = kl.rel((int)(d & kDescKernel));
            kc = q.c;
            km = q.m;
        } else {
            j = ffs32(todo);
            todo &= todo - 1;
        }
        RunState r{W(W_RU + j), W(W_RS + j), W(W_RC + j), W(W_RM + j), W(W_RE + j), list(j)};
        const uint32_t rb = W(W_RB + j);
        if (!listing && ends) release(r);
        KO_RECONVERGE(mask);
        if (todo == 0) {  // every holder of the slots released at t has let go
            freeg |= rel;
            rel = 0;
        }
        bool put = listing;
        if (!listing) {
            const int q = cap(r.u, r.s);
            const int take = q * (int)((rb >> kCntShift) & kSmMask);
            if (take >= left && take > 0) drain = 1;
            if (q > 0 && !drain) {
                if (freeg == 0) fail = 1;
                else {
                    g = take_slot(j, q);
                    placed |= 1ull << g;
                    r.u += (uint32_t)q * hpk;
                    r.s += (uint32_t)(q * hs);
                    r.c += (uint32_t)(q * hc);
                    r.m += (uint32_t)(q * hm);
                    left -= take;
                    const int pos = last_past(rb);
                    pbest = q > pmax ? pos : (q == pmax && pos > pbest ? pos : pbest);
                    pmax = q > pmax ? q : pmax;
                    put = true;
                }
            }
        }
        KO_RECONVERGE(mask);
        if (put) {
            const uint32_t dur = duration(kc, km, r.c, r.m);
            W(W_GE + g) = (uint32_t)t + dur;
            dburst = dur > dburst ? dur : dburst;
            bool first = false;
            r.l = insert(r.l, g, dur, first);
            if (first) r.re = (uint32_t)t + dur;
        }
        KO_RECONVERGE(mask);
        W(W_RU + j) = r.u; W(W_RS + j) = r.s; W(W_RC + j) = r.c; W(W_RM + j) = r.m;
        W(W_RE + j) = r.re;
        set_list(j, r.l);
        if (!ends && drain) todo = 0;  // nothing ends in a first burst: no run left to release
        return drain && todo == 0 && !fail;
    }

    // The burst that empties the queue: take back what event() placed in it and
    // fill its runs jointly.  Blocks go round-robin over the SMs with room, so
    // every SM ends with min(capacity, L - 1) blocks of this burst and the first
    // ones past p with more room have one more; runs are cut at p and where the
    // last sweep stops.  The burst stays open for the next kernel.
    KO_HD void place_partial(int &left)
    {
        for (; placed; placed &= placed - 1) {
            const int g = ffs64(placed);
            const uint32_t d = gd(g), q = ((d >> 5) & 63u) + 1u;
            const int j = (int)(d >> kDescOwnerShift);
            W(W_RU + j) -= q * hpk;
            W(W_RS + j) -= q * (uint32_t)hs;
            W(W_RC + j) -= q * (uint32_t)hc;
            W(W_RM + j) -= q * (uint32_t)hm;
            left += (int)q * (int)((W(W_RB + j) >> kCntShift) & kSmMask);
            freeg |= 1ull << g;
            // out of the list
            const unsigned long long all = list(j);
            int at = 0;
            while (at < kListLen && ((uint32_t)(all >> (kListBits * at)) & 63u) != (uint32_t)g) at++;
            const unsigned long long keep = (1ull << (kListBits * at)) - 1ull;
            const unsigned long long nl = (all & keep) | (pop(all) & ~keep);
            set_list(j, nl);
            const uint32_t head = (uint32_t)nl & 63u;
            if (head != kNoSlot) W(W_RE + j) = W(W_GE + (int)head);
        }
        drain = 0;
        dburst = 0;
        pmax = pbest = 0;
        // capacities, kept in the runs' words
        uint32_t elig = 0;
        int cmax = 0;
        for (uint32_t e = fresh; e; e &= e - 1) {
            const int j = ffs32(e);
            const int c = cap(W(W_RU + j), W(W_RS + j));
            const uint32_t rb = W(W_RB + j) & kSpanMask;
            W(W_RB + j) = rb | ((uint32_t)c << kCapShift);
            cmax = c > cmax ? c : cmax;
            elig |= (c > 0 ? 1u : 0u) << j;
        }
        // smallest sweep count L with F(L) = sum cnt * min(cap, L) >= left (total >= left)
        int lo = 1, hi = cmax;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            int f = 0;
            for (uint32_t e = elig; e; e &= e - 1) {
                const uint32_t rb = W(W_RB + ffs32(e));
                const int c = (int)(rb >> kCapShift);
                f += (int)((rb >> kCntShift) & kSmMask) * (c < mid ? c : mid);
            }
            if (f >= left) hi = mid; else lo = mid + 1;
        }
        const int Lsw = lo;
        // runs whose SMs can take a block in the last sweep; of those, the one that holds p past its start
        uint32_t last = 0, cut = 0;
        int rem = left;
        for (uint32_t e = elig; e; e &= e - 1) {
            const int j = ffs32(e);
            const uint32_t rb = W(W_RB + j);
            const int c = (int)(rb >> kCapShift), b = (int)(rb & kSmMask), n = (int)((rb >> kCntShift) & kSmMask);
            rem -= n * (c < Lsw - 1 ? c : Lsw - 1);
            if (c >= Lsw) {
                last |= 1u << j;
                if (b < p && p < b + n) cut = 1u << j;
            }
        }
        // rem = 1 .. number of SMs with cap >= L.  Visit those runs cyclically from p, one more block
        // to each of their SMs; a run is split where p or the sweep's end lies inside it.
        uint32_t plus = 0;
        int acc = 0, newp = p;
        bool going = last != 0;
        while (going) {
            int j = 0, x;
            if (cut) {
                j = ffs32(cut);
                x = p - (int)(W(W_RB + j) & kSmMask);
            } else {
                int best = 0x7fffffff;
                for (uint32_t e = last; e; e &= e - 1) {
                    const int i = ffs32(e);
                    int d = (int)(W(W_RB + i) & kSmMask) - p;
                    if (d < 0) d += L.S;
                    if (d < best) { best = d; j = i; }
                }
                last &= ~(1u << j);
                plus |= 1u << j;
                const uint32_t rb = W(W_RB + j);
                const int n = (int)((rb >> kCntShift) & kSmMask);
                x = 0;
                if (acc + n >= rem) {
                    x = rem - acc;
                    newp = (int)(rb & kSmMask) + x;
                    if (x == n) x = 0;
                    last = 0;
                }
                acc += n;
            }
            if (x > 0) {
                split(j, x);
                elig |= 1u << (nr - 1);
                if (cut) last |= 1u << (nr - 1);
            }
            cut = 0;
            going = last != 0 && !fail;
        }
        p = newp >= L.S ? newp - L.S : newp;
        for (uint32_t e = elig; e; e &= e - 1) {
            const int j = ffs32(e);
            const int c = (int)(W(W_RB + j) >> kCapShift);
            const int q = (c < Lsw - 1 ? c : Lsw - 1) + (int)((plus >> j) & 1u);
            if (q > 0) add_group(j, q);
        }
        left = 0;
    }

    // The makespan: the latest end of any group, the pending ones' included
    // (groups that have left ended by t).
    KO_HD long long finish() const
    {
        uint32_t d = tail;
        for (unsigned long long pm = pend; pm; pm &= pm - 1) {
            const uint32_t w = gd(ffs64(pm));
            const int j = (int)(w >> kDescOwnerShift);
            const KRel q = kl.rel((int)(w & kDescKernel));
            const uint32_t e = duration(q.c, q.m, W(W_RC + j), W(W_RM + j));
            d = e > d ? e : d;
        }
        return (long long)(t + d);
    }

    // Registers of a node state (the queue is empty, the burst open).
    KO_HD void regs_out(uint32_t *r) const
    {
        r[0] = (uint32_t)t; r[1] = (uint32_t)(t >> 32);
        r[2] = (uint32_t)freeg; r[3] = (uint32_t)(freeg >> 32);
        r[4] = (uint32_t)pend; r[5] = (uint32_t)(pend >> 32);
        r[6] = (uint32_t)p | ((uint32_t)nr << 16); r[7] = tail;
    }
    KO_HD void regs_in(const uint32_t *r)
    {
        t = (unsigned long long)r[0] | ((unsigned long long)r[1] << 32);
        freeg = (unsigned long long)r[2] | ((unsigned long long)r[3] << 32);
        pend = (unsigned long long)r[4] | ((unsigned long long)r[5] << 32);
        p = (int)(r[6] & 0xffffu); nr = (int)(r[6] >> 16);
        tail = r[7];
        settle();
    }

    // The first burst of kernel k and the close of a burst as whole calls, for
    // callers that do not step event() themselves.
    KO_HD int start_kernel(int k)
    {
        int left = begin_kernel(k);
        while (todo && !fail)
            if (event(left, 0u)) place_partial(left);
        return left;
    }
    KO_HD void close_burst()
    {
        int left = 1;  // listing takes no blocks
        while (pend && !fail) event(left, 0u);
    }
};

}  // namespace kolane

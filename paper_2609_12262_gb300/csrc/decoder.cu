// decoder.cu -- parallel sparse-blossom decoder for sm_103a.
//
// A team of threads decodes one shot end to end, and a persistent grid of
// teams pulls shots from a device work counter.  A team is either one warp
// (the batched path: thousands of shots in flight, the 32 lanes of a warp
// working on one shot) or one whole thread block of NW warps (large windows:
// every step below spread over all of the block's threads, for the latency of
// a single window).
//   1. defect compaction: the shot's syndrome bitmap is read with 16-byte
//      vector loads and compacted by a warp prefix sum (input D of the paper's
//      "Decoding task"; Alg. 1 input).
//   2. neighbourhoods: every pair of events within b_1 is read off the graph's
//      ball table (balls.cu: for each detector the detectors near it with exact
//      distances), by testing the entries of each event's list against the
//      syndrome row; every event's nearest boundary is read off a second table.
//      A growing region keeps an explored radius R_s >= Rad(s) + L (L above the
//      largest weight); when it falls due (EXTEND) the events it can touch until
//      the next time come from the pairs already listed or from the farther
//      entries of its list, so the ball itself stays virtual.  Only a region
//      that outgrows the table's radius (about 1 shot in 1,000 at d = 21,
//      p = 0.003, 1 in 60 at d = 51, p = 0.005) makes its shot explore balls
//      {x : dist(s,x) <= R_s} (hash table keyed by (vertex, event), grown band
//      by band by team-parallel label-correcting relaxation; each new entry is
//      checked against the other events' balls holding the same vertex, and
//      against events sitting on it).  Either way the exact distance of two
//      events is known before their regions touch.  The graph-fill region of s
//      (SI S1) is the ball of radius Rad(s) <= R_s, so two regions are found
//      touching exactly when their pair distance equals Rad(a) + Rad(b) (ARRIVE =
//      an extension, COLLIDE = a tight pair, boundary COLLIDE = Rad(s) reaching
//      the nearest boundary, IMPLODE = an inner blossom's dual reaching 0).
//   3. Algorithm 1, level 1: with every pair within b_1 and every boundary
//      contact, min-label components, the diameter <= d_1 test and the parity
//      condition decide the level-1 processing clusters.
//   4. Algorithm 2: level-1 clusters and islands (components of the level-1
//      graph that it does not accept) are solved in closed form where every
//      event only meets its nearest one, else each by a run of its own from t = 0
//      in shared memory; islands whose regions met something outside are joined
//      with it (a level-1 cluster frozen as it stopped) and run again.  That is
//      the run of every remaining event from t = 0 with the stopped level-1
//      configurations present as frozen regions (hierarchical execution rule),
//      which shots outside the limits of this path, and global mode, take as one
//      run with its state in the slab (the general path).
//   5. Result: the weight is the sum of the duals (every matched edge is tight),
//      the observable mask that of the boundary matches' edges.  Only where
//      detector-detector edges carry observables, and in the sliding-window
//      instantiations (batch_kernel<true, *>), blossoms are expanded into matched
//      event pairs and their canonical paths walked: a window commits the edges
//      that touch its commit region.
//
// Simultaneous events are applied in the canonical order (t, kind, lo, hi) with
// kind EXTEND < IMPLODE < COLLIDE < BOUNDARY and lo, hi the ranks of the events
// in the sorted defect list, which makes the result independent of execution
// order, of the team size and equal to global sparse blossom (Theorem 1).
//
// Every loop is bounded: the event budget, hash probe lengths and list
// capacities end a shot with a status code instead of spinning.  In a team of
// several warps every decision that steers control flow around a team barrier
// is taken from a team reduction or broadcast, or from shot state that no
// thread writes between the barrier before the read and the barrier after it,
// so all threads of a team always take the same path.
//
// The rarely taken steps (blossom, shatter, path walks, the general path) are
// kept out of line (__noinline__), so that the kernel's hot code stays small
// enough for the instruction cache.
//
// What bounds it: dependent loads of per-shot state and of the tables and the
// issue of ~3,000 (d = 11) to ~8,000 (d = 21) warp instructions per shot (no
// contraction; the algorithmic bytes take a hundredth of the time).  What it
// took, on one GB300, million shots of d = 7 .. 21 at p = 0.003 / one d = 51
// window / 1,024 circuit-level d = 13 shots, in ms:
//   hash insertions, contact walks, path enumerations   88.7 / 1.42 / 7.4
//   ball tables (per event ~13 coalesced list entries)  21.5 / 0.92 / 0.16
//   islands in shared memory                            13.7 / 0.115 / 0.33
//   phases in step, islands pooled                      12.0 / 0.096 / 0.24
//   closed forms, 20 warps per SM                        8.9 / 0.064 / 0.20
//   larger islands, wider tables                         9.3 / 0.065 / 0.12
//   one-warp overflow deferred; waits, bounds, records   9.8 / 0.065 / 0.13

#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdint>

#include "qec_internal.h"

#define WS 32   // lanes per warp
#ifndef QEC_HT_FACTOR
#define QEC_HT_FACTOR 64   // explored-table slots per detection event (rounded up to a power of two)
#endif
#ifndef QEC_MAX_WARPS
#define QEC_MAX_WARPS 4   // warps of a block that decode a shot each
#endif
#ifndef QEC_SM_WARPS
#define QEC_SM_WARPS 20   // such warps per SM that the register budget must allow
#endif

namespace qec {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr unsigned long long EMPTY64 = ~0ull;
constexpr int INF32 = INT_MAX;

enum { EV_EXTEND = 0, EV_IMPLODE = 1, EV_COLLIDE = 2, EV_BOUNDARY = 3 };
constexpr int ID_BITS = 18;
constexpr int ID_MAX = (1 << ID_BITS) - 1;
constexpr long long T_MAX = (1LL << 26) - 1;

enum { MATE_NONE = -1, MATE_BOUNDARY = -2 };

// slab counters (C_R0 .. C_NEXT: work-list counters of multi-warp teams)
enum { C_ECOUNT = 0, C_WL = 1, C_NPAIRS = 2, C_CCOUNT = 3, C_NFREE = 4, C_ERR = 5, C_NHI = 7,
       C_TL = 8, C_CHANGED = 9, C_TNP = 10, C_TNX = 11, C_R0 = 12, C_NEXT = 15, C_TOTAL = 16 };
enum { ERR_CAP = 1, ERR_INTERNAL = 2 };

__device__ __forceinline__ unsigned long long ev_key(long long t, int kind, int lo, int hi) {
    t = t < T_MAX ? t : T_MAX;
    return ((unsigned long long)t << 38) | ((unsigned long long)kind << 36) |
           ((unsigned long long)lo << 18) | (unsigned long long)hi;
}

// Loads of per-shot state written by other threads of this team (plain stores
// or atomics): relaxed at CTA scope, so they may hit L1 and still observe every
// write ordered before them by the team's barriers.
__device__ __forceinline__ int ldr(const int *p) {
    int v;
    asm volatile("ld.relaxed.cta.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ldr(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.cta.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// One explored entry: key (vertex << 32 | source) and exact distance in one
// 16-byte slot, read by a single vector load.
struct __align__(16) HEnt {
    unsigned long long key;
    int val;
    int pad;
};
__device__ __forceinline__ void ld_ent(const HEnt *p, unsigned long long &k, int &v) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.cta.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    k = a;
    v = (int)(unsigned)(b & 0xffffffffu);
}
// Claim an empty entry (all 16 bytes ones) for (key, d) with one 16-byte
// compare-and-swap; returns true on success, else the key found there.
__device__ __forceinline__ bool claim_ent(HEnt *p, unsigned long long key, int d, unsigned long long &found) {
    const unsigned long long ek = ~0ull, ev = ~0ull;   // an empty entry is all ones
    const unsigned long long nv = (unsigned long long)(unsigned)d;
    unsigned long long ok, ov;
    asm volatile("{\n\t.reg .b128 cmp, swp, old;\n\t"
                 "mov.b128 cmp, {%2, %3};\n\t"
                 "mov.b128 swp, {%4, %5};\n\t"
                 "atom.relaxed.cta.global.cas.b128 old, [%6], cmp, swp;\n\t"
                 "mov.b128 {%0, %1}, old;\n\t}"
                 : "=l"(ok), "=l"(ov) : "l"(ek), "l"(ev), "l"(key), "l"(nv), "l"(p) : "memory");
    found = ok;
    return ok == ek && ov == ev;
}

// Claim an empty pair entry for (key, d) recording pair record idx in the
// entry's upper word; returns true on success, else the entry found there
// (key, value | record << 32).
__device__ __forceinline__ bool claim_pair(HEnt *p, unsigned long long key, int d, int idx,
                                           unsigned long long &fk, unsigned long long &fv) {
    const unsigned long long ek = ~0ull, ev = ~0ull;
    const unsigned long long nv = ((unsigned long long)(unsigned)idx << 32) | (unsigned)d;
    unsigned long long ok, ov;
    asm volatile("{\n\t.reg .b128 cmp, swp, old;\n\t"
                 "mov.b128 cmp, {%2, %3};\n\t"
                 "mov.b128 swp, {%4, %5};\n\t"
                 "atom.relaxed.cta.global.cas.b128 old, [%6], cmp, swp;\n\t"
                 "mov.b128 {%0, %1}, old;\n\t}"
                 : "=l"(ok), "=l"(ov) : "l"(ek), "l"(ev), "l"(key), "l"(nv), "l"(p) : "memory");
    fk = ok;
    fv = ov;
    return ok == ek && ov == ev;
}

// Warp-aggregated atomicAdd(ctr, 1) over the currently active lanes.
__device__ __forceinline__ int agg_inc(int *ctr, int lane) {
    const unsigned m = __activemask();
    const int leader = __ffs(m) - 1;
    const int rank = __popc(m & ((1u << lane) - 1u));
    int base = 0;
    if (lane == leader) base = atomicAdd(ctr, __popc(m));
    base = __shfl_sync(m, base, leader);
    return base + rank;
}

__device__ __forceinline__ unsigned long long warp_min64(unsigned long long v) {
#pragma unroll
    for (int o = WS / 2; o; o >>= 1) {
        unsigned long long w = __shfl_xor_sync(FULL, v, o);
        v = w < v ? w : v;
    }
    return v;
}

// The same with the 32-bit reduction unit: the smallest high word, then the
// smallest low word among the lanes holding it (faster in a block-wide team,
// measured slower in the one-warp path).
__device__ __forceinline__ unsigned long long warp_min64_redux(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_min_sync(FULL, hi);
    const unsigned ml = __reduce_min_sync(FULL, hi == mh ? (unsigned)v : 0xffffffffu);
    return ((unsigned long long)mh << 32) | ml;
}

// 64-bit sums and XORs with the 32-bit reduction unit (values below 2^51: 26
// low bits and the rest apart, so that 32 of either stay below 2^31).
__device__ __forceinline__ long long warp_sum64(long long v) {
    const long long lo = __reduce_add_sync(FULL, (unsigned)v & 0x3ffffffu);
    return lo + ((long long)(int)__reduce_add_sync(FULL, (unsigned)(v >> 26)) << 26);
}

__device__ __forceinline__ unsigned long long warp_xor64(unsigned long long v) {
    return ((unsigned long long)__reduce_xor_sync(FULL, (unsigned)(v >> 32)) << 32) | __reduce_xor_sync(FULL, (unsigned)v);
}

// ------------------------------------------------------------------ teams --

// Shared scratch of a multi-warp team: one slot per warp for reductions, in
// two alternating buffers (every team operation ends with one barrier, so a
// buffer is reused only after every thread has read it).  Functions kept out
// of line take their Team by value and end with a barrier after their last
// team operation, so the caller may go on with its own buffer parity.
struct __align__(16) TSlot {
    unsigned long long u;
    int a, b;
};
struct TeamShared {
    TSlot s[2][32];
};

// Per-thread identity of a team member: a one-warp team needs only the lane
// (its thread index is the lane, its warp 0, and it has no shared scratch).
template <int NW>
struct TeamId {
    int tid_, lane, warp_, ph;
    TeamShared *sh;
    __device__ __forceinline__ int tid() const { return tid_; }
    __device__ __forceinline__ int warp() const { return warp_; }
};
template <>
struct TeamId<1> {
    int lane;
    __device__ __forceinline__ int tid() const { return lane; }
    __device__ __forceinline__ int warp() const { return 0; }
};

template <int NW>
struct Team : TeamId<NW> {
    static constexpr int NT = WS * NW;
    using TeamId<NW>::lane;
    using TeamId<NW>::tid;
    using TeamId<NW>::warp;

    __device__ __forceinline__ void sync() const {
        if constexpr (NW == 1) __syncwarp(); else __syncthreads();
    }
    // thread 0's value for every thread
    __device__ __forceinline__ int bcast(int v) {
        if constexpr (NW == 1) {
            return __shfl_sync(FULL, v, 0);
        } else {
            if (tid() == 0) this->sh->s[this->ph][0].a = v;
            __syncthreads();
            v = this->sh->s[this->ph][0].a;
            this->ph ^= 1;
            return v;
        }
    }
    __device__ __forceinline__ unsigned long long bcast64(unsigned long long v) {
        if constexpr (NW == 1) {
            return __shfl_sync(FULL, v, 0);
        } else {
            if (tid() == 0) this->sh->s[this->ph][0].u = v;
            __syncthreads();
            v = this->sh->s[this->ph][0].u;
            this->ph ^= 1;
            return v;
        }
    }
    // Cross-warp stage of a block reduction: lane 0 of every warp stores its
    // warp's value in its slot; after the barrier lane w of every warp reads
    // slot w (one 16-byte load), and each warp reduces those NW values itself.
    __device__ __forceinline__ TSlot gather(const TSlot &mine, const TSlot &identity) {
        if (lane == 0) this->sh->s[this->ph][warp()] = mine;
        __syncthreads();
        const TSlot x = lane < NW ? this->sh->s[this->ph][lane] : identity;
        this->ph ^= 1;
        return x;
    }
    __device__ __forceinline__ unsigned long long min64(unsigned long long v) {
        if constexpr (NW == 1) return warp_min64(v);
        else return warp_min64_redux(gather(TSlot{warp_min64_redux(v), 0, 0}, TSlot{EMPTY64, 0, 0}).u);
    }
    __device__ __forceinline__ long long sum64(long long v) {
        v = warp_sum64(v);
        if constexpr (NW == 1) return v;
        else return warp_sum64((long long)gather(TSlot{(unsigned long long)v, 0, 0}, TSlot{0, 0, 0}).u);
    }
    __device__ __forceinline__ unsigned long long xor64(unsigned long long v) {
        v = warp_xor64(v);
        if constexpr (NW == 1) return v;
        else return warp_xor64(gather(TSlot{v, 0, 0}, TSlot{0, 0, 0}).u);
    }
    // op: 0 = add, 1 = max, 2 = or
    template <int OP>
    __device__ __forceinline__ int warp_red32(int v) {
        if constexpr (OP == 0) return (int)__reduce_add_sync(FULL, (unsigned)v);
        else if constexpr (OP == 1) return __reduce_max_sync(FULL, v);
        else return (int)__reduce_or_sync(FULL, (unsigned)v);
    }
    template <int OP>
    __device__ __forceinline__ int red32(int v) {
        v = warp_red32<OP>(v);
        if constexpr (NW == 1) return v;
        else return warp_red32<OP>(gather(TSlot{0, v, 0}, TSlot{0, OP == 1 ? INT_MIN : 0, 0}).a);
    }
    __device__ __forceinline__ int add(int v) { return red32<0>(v); }
    __device__ __forceinline__ int maxi(int v) { return red32<1>(v); }
    __device__ __forceinline__ bool any(bool b) { return red32<2>(b ? 1 : 0) != 0; }
    // The event search's reduction in one barrier: smallest key, OR of flags,
    // smallest m (as unsigned).
    __device__ __forceinline__ void reduce_ev(unsigned long long &key, int &flags, unsigned &m) {
        if constexpr (NW == 1) key = warp_min64(key);
        else key = warp_min64_redux(key);
        flags = (int)__reduce_or_sync(FULL, (unsigned)flags);
        m = __reduce_min_sync(FULL, m);
        if constexpr (NW > 1) {
            const TSlot x = gather(TSlot{key, flags, (int)m}, TSlot{EMPTY64, 0, -1});
            key = warp_min64_redux(x.u);
            flags = (int)__reduce_or_sync(FULL, (unsigned)x.a);
            m = __reduce_min_sync(FULL, (unsigned)x.b);
        }
    }
    // Exclusive prefix sum of v over the team's threads in tid order; `total`
    // receives the sum over all threads.
    __device__ __forceinline__ int excl_scan(int v, int &total) {
        int incl = v;
#pragma unroll
        for (int o = 1; o < WS; o <<= 1) {
            const int t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        const int wtot = __shfl_sync(FULL, incl, WS - 1);
        if constexpr (NW == 1) {
            total = wtot;
            return incl - v;
        } else {
            // lane w holds warp w's total: the warp's offset and the block total
            const int x = gather(TSlot{0, wtot, 0}, TSlot{0, 0, 0}).a;
            const int off = (int)__reduce_add_sync(FULL, (unsigned)(lane < warp() ? x : 0));
            total = (int)__reduce_add_sync(FULL, (unsigned)x);
            return off + incl - v;
        }
    }
};

// Per-source state read together by the event search, the dual update and
// the EXTEND scan: one 16-byte record (a single vector load).
//   stop: top-level matcher node containing the source; srad: Rad(s);
//   sR: explored radius (-1: never explored); inplay: part of the current run;
//   sexh: ball exhausted (no vertex left to explore).
struct __align__(16) SRec {
    int stop, srad, sR;
    unsigned char inplay, sexh, pad0, pad1;
};
__device__ __forceinline__ int4 ld_src(const SRec *p) { return *reinterpret_cast<const int4 *>(p); }
__device__ __forceinline__ int rec_inplay(const int4 &r) { return r.w & 0xff; }
__device__ __forceinline__ int rec_sexh(const int4 &r) { return (r.w >> 8) & 0xff; }

// Matcher node state read together by the node scans (dual update,
// implosions, fix-ups): y = the node's own dual, bpar = parent blossom (-1:
// top level), label = +1 outer / -1 inner / 0 not in a tree, alive.
struct __align__(16) NRec {
    int y, bpar, label, alive;
};
__device__ __forceinline__ int4 ld_nd(const NRec *p) { return *reinterpret_cast<const int4 *>(p); }

// A pair of events and their exact distance: ranks lo < hi (lo = -1: an unused
// record), the distance, and the pair's hash slot (-1 while the pair is only
// listed; set once the shot explores balls, see go_real).
struct __align__(16) PRec {
    int lo, hi;
    unsigned val;
    int slot;
};
__device__ __forceinline__ int4 ld_pr(const PRec *p) { return *reinterpret_cast<const int4 *>(p); }

struct Slab {
    // per detection event (source)
    SRec *src;
    int *svtx, *sbeg, *scnt, *comp, *cst0, *cst1, *cst2;
    unsigned long long *sbnd;
    // explored entries (open addressing, keyed by vertex and source); `ent`
    // holds the table slots of every source's bands (band lists)
    HEnt *ht;
    int *ent;
    unsigned long long *wl0, *wl1, *tl;   // work lists (table slots) / new entries (slot << 32 | position)
    int *xsrc, *xR, *xcnt, *xcur;         // sources being extended, target radii, band counts
    int *xidx;                            // position of a source in xsrc during an extension
    int *wcum;                            // detection events in syndrome words before word w
    // pair records, and once the shot explores balls their hash (key lo << 32
    // | hi, value distance, the record's index in the upper word)
    HEnt *pt;
    PRec *pr;
    // matcher nodes (leaf s = node s, blossoms above K)
    NRec *nd;
    int *tpar, *tps, *tpo, *mate, *ms, *mo, *nroot, *minleaf, *cbeg, *clen, *freel, *tmpa, *tmpb, *stk;
    int *cnode, *cs, *co;
    int *ctr;
};

template <typename T>
__host__ __device__ inline T *bump(char *&p, long long n) {
    uintptr_t q = (reinterpret_cast<uintptr_t>(p) + 15) & ~uintptr_t(15);
    T *r = reinterpret_cast<T *>(q);
    p = reinterpret_cast<char *>(q + sizeof(T) * (size_t)n);
    return r;
}

__host__ __device__ inline long long carve(char *base, const SlabCaps &c, Slab &S) {
    char *p = base;
    S.src = bump<SRec>(p, c.kc);
    S.svtx = bump<int>(p, c.kc); S.sbeg = bump<int>(p, c.kc); S.scnt = bump<int>(p, c.kc);
    S.comp = bump<int>(p, c.kc);
    S.cst0 = bump<int>(p, c.kc); S.cst1 = bump<int>(p, c.kc); S.cst2 = bump<int>(p, c.kc);
    S.sbnd = bump<unsigned long long>(p, c.kc);
    S.ht = bump<HEnt>(p, c.hc);
    S.ent = bump<int>(p, c.ec);
    S.wl0 = bump<unsigned long long>(p, c.wc); S.wl1 = bump<unsigned long long>(p, c.wc);
    S.tl = bump<unsigned long long>(p, c.ec);
    S.xsrc = bump<int>(p, c.kc); S.xR = bump<int>(p, c.kc); S.xcnt = bump<int>(p, c.kc); S.xcur = bump<int>(p, c.kc);
    S.xidx = bump<int>(p, c.kc);
    S.wcum = bump<int>(p, c.wcap);
    S.pt = bump<HEnt>(p, c.phc);
    S.pr = bump<PRec>(p, (c.phc >> 1) + 1);
    S.nd = bump<NRec>(p, c.nc);
    S.tpar = bump<int>(p, c.nc); S.tps = bump<int>(p, c.nc); S.tpo = bump<int>(p, c.nc);
    S.mate = bump<int>(p, c.nc); S.ms = bump<int>(p, c.nc); S.mo = bump<int>(p, c.nc);
    S.nroot = bump<int>(p, c.nc); S.minleaf = bump<int>(p, c.nc); S.cbeg = bump<int>(p, c.nc);
    S.clen = bump<int>(p, c.nc); S.freel = bump<int>(p, c.nc);
    S.tmpa = bump<int>(p, 2 * c.nc + 64); S.tmpb = bump<int>(p, 2 * c.nc + 64);
    S.stk = bump<int>(p, 4 * c.nc + 64);
    S.cnode = bump<int>(p, c.cc); S.cs = bump<int>(p, c.cc); S.co = bump<int>(p, c.cc);
    S.ctr = bump<int>(p, C_TOTAL);
    return (long long)(p - base) + 16;
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

struct Shot {
    unsigned long long deadline;   // globaltimer value after which the shot gives up (0 = none)
    DGraph g;
    int K;            // detection events
    unsigned hmask;   // explored-entry hash mask
    unsigned pmask;   // pair hash mask
    int ec, wc, nc, cc;
    int pcap;         // pair records the slab holds
    int real;         // balls are explored (else every ball is virtual, see extend_due)
    int paths;        // a path was walked through an explored ball
    int band;
    int L;                 // lookahead: explored radius >= Rad + L for every growing region
    const unsigned *row;   // the shot's syndrome row (defect test)
    long long t;
    long long events;
    long long max_events;
    // parallel-event-count bookkeeping of the current run (Methods, "Numerical
    // evaluation"): matcher events applied, those at times <= tcut, the time of
    // the last one, and flooder band extensions
    int nm, ncut, tcut, tlast, nx;
};

// Home slots: the high bits of a multiplicative (Fibonacci) hash, so that
// nearby vertices spread over the whole table; mask + 1 is a power of two.
__device__ __forceinline__ unsigned hslot(int v, unsigned mask) {
    return ((unsigned)v * 2654435761u) >> (32 - __popc(mask));
}

__device__ __forceinline__ unsigned pslot(int lo, int hi, unsigned mask) {
    return (((unsigned)lo * 2654435761u + (unsigned)hi) * 2246822519u) >> (32 - __popc(mask));
}

__device__ __forceinline__ void set_err(const Slab &S, int bit) { atomicOr(&S.ctr[C_ERR], bit); }

// exact distance of (v, s) if explored, else INF32
__device__ int ht_get(const Slab &S, const Shot &C, int v, int s) {
    const unsigned long long key = ((unsigned long long)(unsigned)v << 32) | (unsigned)s;
    unsigned i = hslot(v, C.hmask);
    for (unsigned n = 0; n <= C.hmask; n++) {
        unsigned long long k;
        int v;
        ld_ent(&S.ht[i], k, v);
        if (k == key) return v;
        if (k == EMPTY64) return INF32;
        i = (i + 1) & C.hmask;
    }
    return INF32;
}

// insert-or-decrease; returns 1 inserted, 2 decreased, 0 unchanged, -1 table
// full; `slot` receives the entry's table slot
__device__ int ht_upsert(const Slab &S, const Shot &C, int v, int s, int d, unsigned &slot) {
    const unsigned long long key = ((unsigned long long)(unsigned)v << 32) | (unsigned)s;
    unsigned i = hslot(v, C.hmask);
    for (unsigned n = 0; n <= C.hmask; n++) {
        unsigned long long k;
        int v;
        ld_ent(&S.ht[i], k, v);
        if (k == EMPTY64) {
            if (claim_ent(&S.ht[i], key, d, k)) {
                slot = i;
                return 1;
            }
            v = INF32;
        }
        if (k == key) {
            slot = i;
            if (d >= v) return 0;   // values only decrease: nothing to do
            int old = atomicMin(&S.ht[i].val, d);
            return d < old ? 2 : 0;
        }
        i = (i + 1) & C.hmask;
    }
    set_err(S, ERR_CAP);
    return -1;
}

// Insert-or-decrease the pair (a, b) with distance d (shots that explore
// balls): a new pair reserves the next record, complete but for its slot,
// before claiming its hash slot, and every smaller value goes to the entry and
// to the record, so both hold the minimum after the next barrier.
__device__ void pair_upsert(const Slab &S, const Shot &C, int a, int b, int d) {
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const unsigned long long key = ((unsigned long long)(unsigned)lo << 32) | (unsigned)hi;
    unsigned i = pslot(lo, hi, C.pmask);
    int idx = -1;
    for (unsigned n = 0; n <= C.pmask; n++) {
        unsigned long long k, w;
        asm volatile("ld.relaxed.cta.v2.b64 {%0, %1}, [%2];" : "=l"(k), "=l"(w) : "l"(&S.pt[i]) : "memory");
        if (k == EMPTY64) {
            if (idx < 0) {
                idx = atomicAdd(&S.ctr[C_NPAIRS], 1);
                if ((unsigned)idx * 2u > C.pmask || idx >= C.pcap) { set_err(S, ERR_CAP); return; }
                S.pr[idx] = PRec{lo, hi, (unsigned)d, -1};
                __threadfence_block();
            }
            if (claim_pair(&S.pt[i], key, d, idx, k, w)) {
                S.pr[idx].slot = (int)i;
                return;
            }
        }
        if (k == key) {
            const int v = (int)(unsigned)(w & 0xffffffffu), j = (int)(w >> 32);
            if (d < v) {
                atomicMin(&S.pt[i].val, d);
                atomicMin(&S.pr[j].val, (unsigned)d);
            }
            if (idx >= 0) S.pr[idx].lo = -1;   // reserved, lost the slot to the same pair
            return;
        }
        i = (i + 1) & C.pmask;
    }
    set_err(S, ERR_CAP);
}

struct SlotV {
    int nbr;   // neighbour detector, -1 for the boundary
    int w;     // internal weight
    int eid;   // merged edge id (boundary slots only; -1 otherwise)
};

__device__ __forceinline__ SlotV load_slot(const DGraph &g, int j) {
    const int2 v = __ldg(reinterpret_cast<const int2 *>(g.slot) + j);
    SlotV s;
    s.w = v.y;
    if (v.x < 0) { s.nbr = -1; s.eid = -1 - v.x; }
    else { s.nbr = v.x; s.eid = -1; }
    return s;
}

__device__ __forceinline__ bool is_defect(const Shot &C, int v) {
    return (__ldg(C.row + (v >> 5)) >> (v & 31)) & 1u;
}

// Rank of detection event vertex v in the sorted event list (v must be an
// event): events in earlier words plus set bits below v in its own word.
__device__ __forceinline__ int rank_of(const Slab &S, const Shot &C, int v) {
    const unsigned w = __ldg(C.row + (v >> 5));
    return S.wcum[v >> 5] + __popc(w & ((1u << (v & 31)) - 1u));
}

// Grow the explored balls of the sources xsrc[0 .. nx) from radius sR[s] to
// xR[i] (xR[i] - sR[s] >= largest weight), all at once: the previous band of
// each source is the frontier (its own vertex when never explored),
// label-correcting relaxation runs on work lists of table slots (a slot's key
// names the vertex and source, its value the current distance) until no
// distance changes, with CONTACTS every new entry is checked for contacts with
// the other sources' balls, and each source's new band is stored contiguously
// in `ent` as its next frontier.  Every thread of the team calls with the same
// nx.  Only shots with a region too large for the ball table get here, so it
// stays out of line.
template <bool CONTACTS, int NW>
__device__ __noinline__ void extend_many(const Slab &S, const Shot &C, int nx, Team<NW> T) {
    const DGraph &g = C.g;
    if (nx <= 0) return;
    const int lane = T.lane;
    T.sync();
    if (T.tid() == 0) {
        S.ctr[C_TL] = 0; S.ctr[C_WL] = 0;
        if constexpr (NW > 1) { S.ctr[C_R0] = 0; S.ctr[C_R0 + 1] = 0; }
    }
    for (int i = T.tid(); i < nx; i += T.NT) { S.xcnt[i] = 0; S.xidx[S.xsrc[i]] = i; }
    T.sync();
    unsigned *F = reinterpret_cast<unsigned *>(S.wl0), *Wn = reinterpret_cast<unsigned *>(S.wl1);
    for (int i = T.tid(); i < nx; i += T.NT) {
        const int s = S.xsrc[i];
        if (S.src[s].sR < 0) {
            unsigned hs;
            const int r = ht_upsert(S, C, S.svtx[s], s, 0, hs);
            if (r < 0) continue;
            if (r == 1) {
                const int e = atomicAdd(&S.ctr[C_TL], 1);
                if (e < C.ec) S.tl[e] = ((unsigned long long)hs << 32) | (unsigned)i; else set_err(S, ERR_CAP);
            }
            const int w = atomicAdd(&S.ctr[C_WL], 1);
            if (w < C.wc) F[w] = hs; else set_err(S, ERR_CAP);
            continue;
        }
        const int fb = S.sbeg[s], fc = S.scnt[s];
        const int base = atomicAdd(&S.ctr[C_WL], fc);
        for (int k = 0; k < fc; k++) {
            if (base + k < C.wc) F[base + k] = (unsigned)S.ent[fb + k];
            else set_err(S, ERR_CAP);
        }
    }
    T.sync();
    int nf = min(ldr(&S.ctr[C_WL]), C.wc);
    // a one-warp team keeps the list counters in registers (warp-uniform) and
    // places each round's appends by ballot; several warps reserve their
    // appends with one atomic per warp and round on counters that rotate over
    // three slots (a slot is cleared two rounds before its next use)
    int ntl = ldr(&S.ctr[C_TL]);
    const unsigned lt = (1u << lane) - 1u;
    for (int iter = 0;; iter++) {
        if (iter >= 4096) { if (T.tid() == 0) set_err(S, ERR_INTERNAL); break; }
        int nwl = 0;
        int *const wctr = &S.ctr[C_R0 + iter % 3];
        if constexpr (NW > 1) {
            if (T.tid() == 0) S.ctr[C_R0 + (iter + 1) % 3] = 0;
        }
        // one lane per (work item, adjacency slot): items are taken 32 at a
        // time per warp, their slots numbered by a warp prefix sum of the
        // degrees, and slot t goes to lane t mod 32 (its item found by binary
        // search)
        for (int base = T.warp() * WS; base < nf; base += T.NT) {
            const int i = base + lane;
            unsigned long long key = 0;
            int dx = 0, Rn = -1, r0 = 0, deg = 0, xi = 0;
            if (i < nf) {
                const unsigned hx = F[i];
                ld_ent(&S.ht[hx], key, dx);
                const int x = (int)(key >> 32);
                xi = S.xidx[(int)(unsigned)(key & 0xffffffffu)];
                Rn = S.xR[xi];
                r0 = __ldg(g.row + x);
                deg = __ldg(g.row + x + 1) - r0;
            }
            int incl = deg;
            for (int o = 1; o < WS; o <<= 1) {
                const int v = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(FULL, incl, WS - 1);
            const int excl = incl - deg;
            for (int t0 = 0; t0 < total; t0 += WS) {
                const int t = t0 + lane;
                // owner: the last lane whose first slot number is <= t
                int ow = 0;
                for (int step = WS / 2; step > 0; step >>= 1) {
                    const int e = __shfl_sync(FULL, excl, ow + step);
                    if (e <= t) ow += step;
                }
                const unsigned long long okey = __shfl_sync(FULL, key, ow);
                const int odx = __shfl_sync(FULL, dx, ow);
                const int oRn = __shfl_sync(FULL, Rn, ow);
                const int oj = __shfl_sync(FULL, r0 - excl, ow) + t;
                const int oxi = __shfl_sync(FULL, xi, ow);
                int r = 0;
                unsigned hs = 0;
                if (t < total) {
                    const int s = (int)(unsigned)(okey & 0xffffffffu);
                    const SlotV sl = load_slot(g, oj);
                    const int nd = odx + sl.w;
                    if (sl.nbr >= 0 && nd <= oRn) r = ht_upsert(S, C, sl.nbr, s, nd, hs);
                }
                const unsigned mt = __ballot_sync(FULL, r == 1);
                const unsigned mw = __ballot_sync(FULL, r >= 1);
                int bt, bw;
                if constexpr (NW == 1) {
                    bt = ntl; bw = nwl;
                    ntl += __popc(mt);
                    nwl += __popc(mw);
                } else {
                    bt = 0; bw = 0;
                    if (lane == 0) {
                        if (mt) bt = atomicAdd(&S.ctr[C_TL], __popc(mt));
                        if (mw) bw = atomicAdd(wctr, __popc(mw));
                    }
                    bt = __shfl_sync(FULL, bt, 0);
                    bw = __shfl_sync(FULL, bw, 0);
                }
                if (r == 1) {
                    const int e = bt + __popc(mt & lt);
                    if (e < C.ec) S.tl[e] = ((unsigned long long)hs << 32) | (unsigned)oxi; else set_err(S, ERR_CAP);
                }
                if (r >= 1) {
                    const int w = bw + __popc(mw & lt);
                    if (w < C.wc) Wn[w] = hs; else set_err(S, ERR_CAP);
                }
            }
        }
        T.sync();
        bool stop;
        if constexpr (NW == 1) {
            const int err = ldr(&S.ctr[C_ERR]);
            stop = nwl == 0 || err;
        } else {
            // this round's counter is written by no thread until two rounds
            // on, so every thread reads the same value: a uniform decision
            // without a reduction (a capacity error ends the rounds once no
            // insertion succeeds; the caller reads the error word)
            nwl = ldr(wctr);
            stop = nwl == 0;
        }
        if (stop) break;
        nf = min(nwl, C.wc);
        unsigned *t = F; F = Wn; Wn = t;
    }
    if constexpr (NW == 1) {
        if (lane == 0) S.ctr[C_TL] = ntl;
    }
    T.sync();
    const unsigned long long ne = T.bcast64(((unsigned long long)(unsigned)min(ldr(&S.ctr[C_TL]), C.ec) << 32) |
                                            (unsigned)ldr(&S.ctr[C_ECOUNT]));
    const int nt = (int)(unsigned)(ne >> 32);
    const int e0 = (int)(unsigned)(ne & 0xffffffffu);
    // explored-entry table at most half full, list room left
    if (e0 + nt > C.ec || (unsigned)(e0 + nt) * 2u > C.hmask) {
        if (T.tid() == 0) set_err(S, ERR_CAP);
        T.sync();
        return;
    }
    // bands made contiguous per source (counting sort of the new entries)
    for (int i = T.tid(); i < nt; i += T.NT) atomicAdd(&S.xcnt[(int)(unsigned)(S.tl[i] & 0xffffffffu)], 1);
    T.sync();
    if constexpr (NW == 1) {
        // band starts in list order, by lane 0 (a warp extends only a few
        // sources at a time; measured faster than a warp-wide scan)
        if (lane == 0) {
            int acc = e0;
            for (int i = 0; i < nx; i++) {
                const int s = S.xsrc[i];
                const int c = S.xcnt[i];
                S.xcur[i] = acc;
                S.sbeg[s] = acc;
                S.scnt[s] = c;
                S.src[s].sR = S.xR[i];
                if (c == 0) S.src[s].sexh = 1;
                acc += c;
            }
            S.ctr[C_ECOUNT] = acc;
        }
    } else {
        // band starts: exclusive prefix sum of the counts in list order, each
        // thread one contiguous chunk of the list
        const int per = (nx + T.NT - 1) / T.NT;
        const int i0 = min(nx, T.tid() * per), i1 = min(nx, i0 + per);
        int loc = 0;
        for (int i = i0; i < i1; i++) loc += S.xcnt[i];
        int total = 0;
        int acc = e0 + T.excl_scan(loc, total);
        for (int i = i0; i < i1; i++) {
            const int s = S.xsrc[i];
            const int c = S.xcnt[i];
            S.xcur[i] = acc;
            S.sbeg[s] = acc;
            S.scnt[s] = c;
            S.src[s].sR = S.xR[i];
            if (c == 0) S.src[s].sexh = 1;
            acc += c;
        }
        if (T.tid() == 0) {
            S.ctr[C_ECOUNT] = e0 + total;
            S.ctr[C_NEXT] = 0;
        }
    }
    T.sync();
    for (int i = T.tid(); i < nt; i += T.NT) {
        const unsigned long long it = S.tl[i];
        const int pos = atomicAdd(&S.xcur[(int)(unsigned)(it & 0xffffffffu)], 1);
        S.ent[pos] = (int)(it >> 32);
    }
    T.sync();
    // contacts of every new entry y of source s: other explored balls holding y
    // (same vertex), and y being another detection event's own vertex (reach).
    // With explored radius >= Rad + L for every growing region (L >= largest
    // weight, >= the radius of any never-explored frozen region) these find every
    // pair of regions at the instant they become tight: on a shortest path
    // between them, the first vertex at distance >= Rad(a) from a lies in b's
    // region and within Rad(a) + largest weight of a.
    // Each lane walks the probe chain of one entry, one probe per round; a lane
    // whose walk has ended takes the next unwalked entry, so the lanes stay busy
    // however the chain lengths vary (a warp of a larger team claims entries
    // from a shared counter).
    if constexpr (CONTACTS) {
        int cur = -1, yv = 0, s = 0, dy = 0;
        unsigned pos = 0, nprobe = 0;
        int next = 0;
        for (long long round = 0; round < (long long)nt * (C.hmask + 2) + 1; round++) {
            const unsigned idle = __ballot_sync(FULL, cur < 0);
            int kb;
            if constexpr (NW == 1) {
                kb = next;
                next += __popc(idle);
            } else {
                kb = 0;
                if (lane == 0 && idle) kb = atomicAdd(&S.ctr[C_NEXT], __popc(idle));
                kb = __shfl_sync(FULL, kb, 0);
            }
            if (cur < 0) {
                const int k = kb + __popc(idle & lt);
                if (k < nt) {
                    cur = k;
                    const unsigned hy = (unsigned)(S.tl[k] >> 32);
                    unsigned long long key;
                    ld_ent(&S.ht[hy], key, dy);
                    yv = (int)(key >> 32);
                    s = (int)(unsigned)(key & 0xffffffffu);
                    pos = hslot(yv, C.hmask);
                    nprobe = 0;
                    if (yv != S.svtx[s] && is_defect(C, yv)) {
                        const int f = rank_of(S, C, yv);
                        if (f >= 0 && f != s) pair_upsert(S, C, s, f, dy);
                    }
                }
            }
            if (!__any_sync(FULL, cur >= 0)) break;
            if (cur >= 0) {
                unsigned long long k;
                int v;
                ld_ent(&S.ht[pos], k, v);
                if (k == EMPTY64 || ++nprobe > C.hmask) {
                    cur = -1;
                } else {
                    if ((int)(k >> 32) == yv) {
                        const int s2 = (int)(unsigned)(k & 0xffffffffu);
                        if (s2 != s) pair_upsert(S, C, s, s2, dy + v);
                    }
                    pos = (pos + 1) & C.hmask;
                }
            }
        }
    }
    T.sync();
}

// Grow one source's ball by one band, without contacts (path tracing).  Every
// thread of the team calls.
template <int NW>
__device__ void extend_one(const Slab &S, const Shot &C, int s, Team<NW> &T) {
    if (T.tid() == 0) { S.xsrc[0] = s; S.xR[0] = max(S.src[s].sR, 0) + C.band; }
    T.sync();
    extend_many<false>(S, C, 1, T);
}

// From here on the shot explores balls: the listed pairs enter the pair hash,
// and every source with a virtual ball gets the ball of that radius.  Every
// thread of the team calls.
template <int NW>
__device__ __noinline__ void go_real(const Slab &S, Shot &C, Team<NW> T) {
    C.real = 1;
    const int np = T.bcast(ldr(&S.ctr[C_NPAIRS]));
    if (np > C.pcap || (unsigned)np * 2u > C.pmask) {
        if (T.tid() == 0) set_err(S, ERR_CAP);
        T.sync();
        return;
    }
    T.sync();
    if (T.tid() == 0) S.ctr[C_WL] = 0;
    for (int i = T.tid(); i < np; i += T.NT) {
        const int4 q = ld_pr(&S.pr[i]);
        const unsigned long long key = ((unsigned long long)(unsigned)q.x << 32) | (unsigned)q.y;
        unsigned h = pslot(q.x, q.y, C.pmask);
        for (unsigned n = 0; n <= C.pmask; n++) {
            unsigned long long k, w;
            if (claim_pair(&S.pt[h], key, q.z, i, k, w)) { S.pr[i].slot = (int)h; break; }
            if (k == key) { S.pr[i].lo = -1; break; }   // listed from both ends, at the same distance
            h = (h + 1) & C.pmask;
        }
    }
    T.sync();
    for (int s = T.tid(); s < C.K; s += T.NT) {
        const int r = S.src[s].sR;
        if (r < 0) continue;
        const int k = atomicAdd(&S.ctr[C_WL], 1);
        S.xsrc[k] = s;
        S.xR[k] = r;
        S.src[s].sR = -1;
    }
    T.sync();
    const int nx = T.bcast(ldr(&S.ctr[C_WL]));
    T.sync();
    extend_many<true>(S, C, nx, T);
}

// Radius within which every other detection event of source s has to be known
// once its ball has radius R: no region with a smaller ball can be touched
// farther away (Rad <= R - L for explored regions, Rad <= b1 / 2 for level-1
// configurations never explored).
__device__ __forceinline__ int reach_of(const Shot &C, int R) {
    const int r = R - C.L;
    return r + max(r, (C.g.b1 + 1) >> 1);
}

// EXTEND: every growing region whose radius has come within L of its explored
// radius gets a larger ball.  While the ball table covers the radius that
// matters (reach_of) the ball stays virtual: the events within that radius
// are read off the table's list of the source's vertex (nothing at all when
// the pairs within b1, listed at the start of the shot, already cover it).
// Otherwise the shot goes over to explored balls.  The table's radius (balls.cu:
// six largest weights) lets a region's radius grow to three edges before that;
// a shot gains a band each time exactly when it would with explored balls, so
// the diagnostics do not depend on which is used.  Returns the number of due
// regions.  Every thread of the team calls; ends with a barrier.
template <int NW>
__device__ int extend_due(const Slab &S, Shot &C, Team<NW> &T) {
    const DGraph &g = C.g;
    for (;;) {
        // the list counter is zero on entry (cleared ahead of the event
        // search's barrier)
        int any = 0;   // bit 0: a region is due, bit 1: one is beyond the table
        for (int s = T.tid(); s < C.K; s += T.NT) {
            const int4 r = ld_src(&S.src[s]);
            const int rad = r.y, sR = r.z;
            if (!rec_inplay(r) || rec_sexh(r) || sR - C.L + 1 - rad > 0 || S.nd[r.x].label != 1) continue;
            const int R = max(sR + C.band, rad + C.L + C.band);
            any |= 1;
            if (!C.real) {
                const int q = reach_of(C, R);
                if (sR < 0 && q <= g.b1) { S.src[s].sR = R; continue; }
                if (q > g.brad || sR > g.brad - g.wmax || __ldg(g.bhdr + S.svtx[s]).w < 0) { any |= 2; continue; }
            }
            const int k = atomicAdd(&S.ctr[C_WL], 1);
            S.xsrc[k] = s;
            S.xR[k] = R;
        }
        any = T.template red32<2>(any);
        if constexpr (NW == 1) T.sync();
        if (any & 2) {
            go_real(S, C, T);
            if (T.tid() == 0) S.ctr[C_WL] = 0;
            T.sync();
            if (T.bcast(ldr(&S.ctr[C_ERR]))) return any;
            continue;
        }
        const int nx = T.bcast(ldr(&S.ctr[C_WL]));
        if (C.real) {
            T.sync();
            extend_many<true>(S, C, nx, T);
            return any;
        }
        for (int i = T.warp(); i < nx; i += NW) {
            const int s = S.xsrc[i], R = S.xR[i], sR = S.src[s].sR;
            const int v = S.svtx[s];
            const int4 h = __ldg(g.bhdr + v);
            const int q = reach_of(C, R), q0 = sR < 0 ? g.b1 : max(g.b1, reach_of(C, sR));
            const int n = h.z + h.w;
            bool more = false;
            for (int k = 0; k < n; k += WS) {
                bool hit = false;
                int2 e = make_int2(0, 0);
                if (k + T.lane < n) {
                    e = __ldg(g.ball + (unsigned)h.x + k + T.lane);
                    more |= e.y > sR;
                    hit = e.y > q0 && e.y <= q && is_defect(C, e.x);
                }
                const unsigned m = __ballot_sync(FULL, hit);
                if (!m) continue;
                int b = 0;
                if (T.lane == 0) b = atomicAdd(&S.ctr[C_NPAIRS], __popc(m));
                b = __shfl_sync(FULL, b, 0);
                if (hit) {
                    const int j = b + __popc(m & ((1u << T.lane) - 1u));
                    const int f = rank_of(S, C, e.x);
                    if (j < C.pcap) S.pr[j] = PRec{min(s, f), max(s, f), (unsigned)e.y, -1};
                    else set_err(S, ERR_CAP);
                }
            }
            // a ball that gains no vertex has covered its component
            more = __any_sync(FULL, more);
            if (T.lane == 0) {
                S.src[s].sR = R;
                if (sR >= 0 && !more) S.src[s].sexh = 1;
            }
        }
        T.sync();
        return any;
    }
}

// ---------------------------------------------------------------- matcher --

// Child of blossom B that contains `leaf` (-1 if B is not an ancestor).
__device__ __forceinline__ int child_of(const Slab &S, int B, int leaf) {
    int v = leaf;
    for (int n = 0; n < 1 << 20 && v >= 0 && S.nd[v].bpar != B; n++) v = S.nd[v].bpar;
    return v;
}

// flip matches along the tree path from outer A to its root (thread 0)
__device__ void flip_to_root(const Slab &S, int A) {
    int v = A;
    for (int n = 0; n < 1 << 22 && S.tpar[v] >= 0; n++) {
        const int I = S.tpar[v];
        const int O = S.tpar[I];
        if (O < 0) { S.ctr[C_ERR] |= ERR_INTERNAL; return; }
        S.mate[I] = O; S.ms[I] = S.tps[I]; S.mo[I] = S.tpo[I];
        S.mate[O] = I; S.ms[O] = S.tpo[I]; S.mo[O] = S.tps[I];
        v = O;
    }
}

// Events (b), (f), (g).  B < 0: boundary.  Every thread of the team calls.
template <int NW>
__device__ __noinline__ void ev_augment(const Slab &S, Shot &C, int A, int a, int B, int b, Team<NW> T, int nhi) {
    int rA = 0, rB = -3;
    bool bout = false;
    // flip the matches along both tree paths and match A with B (thread 0)
    auto rematch = [&]() {
        flip_to_root(S, A);
        if (bout) flip_to_root(S, B);
        if (B >= 0) {
            S.mate[A] = B; S.ms[A] = a; S.mo[A] = b;
            S.mate[B] = A; S.ms[B] = b; S.mo[B] = a;
        } else {
            S.mate[A] = MATE_BOUNDARY; S.ms[A] = a; S.mo[A] = -1;
        }
    };
    if (T.tid() == 0) {
        rA = S.nroot[A];
        bout = B >= 0 && S.nd[B].label == 1;
        rB = bout ? S.nroot[B] : -3;
        if constexpr (NW == 1) rematch();
    }
    {
        // both roots in one broadcast (a block's broadcast is also its barrier)
        const unsigned long long pr = T.bcast64(((unsigned long long)(unsigned)rA << 32) | (unsigned)rB);
        rA = (int)(unsigned)(pr >> 32);
        rB = (int)(unsigned)(pr & 0xffffffffu);
    }
    if constexpr (NW == 1) {
        T.sync();
        for (int v = T.tid(); v < nhi; v += T.NT) {
            const int4 q = ld_nd(&S.nd[v]);
            if (q.w && q.y < 0 && q.z != 0 && (S.nroot[v] == rA || S.nroot[v] == rB)) {
                S.nd[v].label = 0; S.tpar[v] = -1; S.nroot[v] = -1;
            }
        }
    } else {
        // The two trees' nodes leave them (label and root cleared; a node's
        // tree parent is only read while it is in a tree, and is set again when
        // it joins one), while thread 0 rewrites the matches along the tree
        // paths, which reads tree parents and writes only mates: the two
        // overlap.  Independent loads first (one round trip per node).
        for (int v = T.tid(); v < nhi; v += T.NT) {
            const int4 q = ld_nd(&S.nd[v]);
            const int nr = S.nroot[v];
            if (q.w && q.y < 0 && q.z != 0 && (nr == rA || nr == rB)) { S.nd[v].label = 0; S.nroot[v] = -1; }
        }
        if (T.tid() == 0) rematch();
    }
    T.sync();
}

// Event (a): outer A touches frozen B (matched to C).  Thread 0 only.
__device__ void ev_grow(const Slab &S, int A, int a, int B, int b) {
    const int Cn = S.mate[B];
    S.nd[B].label = -1; S.tpar[B] = A; S.tps[B] = b; S.tpo[B] = a; S.nroot[B] = S.nroot[A];
    S.nd[Cn].label = 1; S.tpar[Cn] = B; S.tps[Cn] = S.ms[Cn]; S.tpo[Cn] = S.mo[Cn]; S.nroot[Cn] = S.nroot[A];
}

// Event (c): outer A, B in one tree form a blossom.  Every thread of the team calls.
template <int NW>
__device__ __noinline__ void ev_blossom(const Slab &S, Shot &C, int A, int a, int B, int b, Team<NW> T, int &nhi) {
    int N = -1, L = -1, Lroot = 0;
    if (T.tid() == 0) {
        int na = 0, nb = 0;
        for (int v = A; v >= 0 && na < 2 * C.nc; v = S.tpar[v]) S.tmpa[na++] = v;
        for (int v = B; v >= 0 && nb < 2 * C.nc; v = S.tpar[v]) S.tmpb[nb++] = v;
        while (na > 1 && nb > 1 && S.tmpa[na - 2] == S.tmpb[nb - 2]) { na--; nb--; }
        L = S.tmpa[na - 1];
        const int m = na + nb - 1;
        const int nf = S.ctr[C_NFREE];
        const int cb = S.ctr[C_CCOUNT];
        if (L != S.tmpb[nb - 1] || nf <= 0 || cb + m > C.cc) {
            S.ctr[C_ERR] |= (L != S.tmpb[nb - 1]) ? ERR_INTERNAL : ERR_CAP;
        } else {
            N = S.freel[nf - 1];
            S.ctr[C_NFREE] = nf - 1;
            S.ctr[C_CCOUNT] = cb + m;
            int i = 0;
            S.cnode[cb + i++] = L;
            for (int j = na - 2; j >= 0; j--) S.cnode[cb + i++] = S.tmpa[j];
            for (int j = 0; j <= nb - 2; j++) S.cnode[cb + i++] = S.tmpb[j];
            const int ia = na - 1;
            int ml = INT_MAX;
            for (int j = 0; j < m; j++) {
                const int x = S.cnode[cb + j], z = S.cnode[cb + (j + 1) % m];
                if (j < ia) { S.cs[cb + j] = S.tpo[z]; S.co[cb + j] = S.tps[z]; }
                else if (j == ia) { S.cs[cb + j] = a; S.co[cb + j] = b; }
                else { S.cs[cb + j] = S.tps[x]; S.co[cb + j] = S.tpo[x]; }
                ml = min(ml, S.minleaf[x]);
            }
            S.nd[N] = NRec{0, -1, 1, 1};
            S.tpar[N] = S.tpar[L]; S.tps[N] = S.tps[L]; S.tpo[N] = S.tpo[L];
            S.mate[N] = S.mate[L]; S.ms[N] = S.ms[L]; S.mo[N] = S.mo[L];
            Lroot = (S.nroot[L] == L);
            S.nroot[N] = Lroot ? N : S.nroot[L];
            S.minleaf[N] = ml; S.cbeg[N] = cb; S.clen[N] = m;
            for (int j = 0; j < m; j++) S.nd[S.cnode[cb + j]].bpar = N;
        }
    }
    {
        // N, L and whether L was its tree's root in one broadcast (ids < 2^18)
        const unsigned hi = L >= 0 ? ((unsigned)L | ((unsigned)Lroot << 30)) : 0xffffffffu;
        const unsigned long long pk = T.bcast64(((unsigned long long)hi << 32) | (unsigned)N);
        N = (int)(unsigned)(pk & 0xffffffffu);
        const unsigned h = (unsigned)(pk >> 32);
        L = h == 0xffffffffu ? -1 : (int)(h & 0x3fffffffu);
        Lroot = h == 0xffffffffu ? 0 : (int)((h >> 30) & 1u);
    }
    if constexpr (NW == 1) T.sync();
    if (N < 0) return;
    nhi = max(nhi, N + 1);
    for (int v = T.tid(); v < nhi; v += T.NT) {
        if constexpr (NW == 1) {
            const int4 q = ld_nd(&S.nd[v]);
            if (!q.w || q.y >= 0 || v == N) continue;
            const int tp = S.tpar[v];
            if (tp >= 0 && S.nd[tp].bpar == N) S.tpar[v] = N;
            const int mt = S.mate[v];
            if (mt >= 0 && S.nd[mt].bpar == N) S.mate[v] = N;
            if (Lroot && S.nroot[v] == L) S.nroot[v] = N;
        } else {
            // independent loads first, the parents' blossom pointers after
            const int4 q = ld_nd(&S.nd[v]);
            const int al = q.w, bp = q.y, tp = S.tpar[v], mt = S.mate[v], nr = S.nroot[v];
            if (!al || bp >= 0 || v == N) continue;
            const int btp = tp >= 0 ? S.nd[tp].bpar : -1, bmt = mt >= 0 ? S.nd[mt].bpar : -1;
            if (btp == N) S.tpar[v] = N;
            if (bmt == N) S.mate[v] = N;
            if (Lroot && nr == L) S.nroot[v] = N;
        }
    }
    for (int s = T.tid(); s < C.K; s += T.NT) {
        const int tp = S.src[s].stop;
        if (tp != N && S.nd[tp].bpar == N) S.src[s].stop = N;
    }
    T.sync();
}

// Event (d): inner blossom B with zero dual shatters.  Every thread of the team calls.
template <int NW>
__device__ __noinline__ void ev_shatter(const Slab &S, Shot &C, int B, Team<NW> T) {
    for (int s = T.tid(); s < C.K; s += T.NT)
        if (S.src[s].stop == B) {
            const int c = child_of(S, B, s);
            if (c >= 0) S.src[s].stop = c; else atomicOr(&S.ctr[C_ERR], ERR_INTERNAL);
        }
    T.sync();
    if (T.tid() == 0) {
        const int m = S.clen[B], cb = S.cbeg[B];
        const int P = S.tpar[B], Cn = S.mate[B];
        const int xp = S.tps[B] >= 0 ? child_of(S, B, S.tps[B]) : -1;
        const int xc = S.ms[B] >= 0 ? child_of(S, B, S.ms[B]) : -1;
        int ip = -1, ic = -1;
        for (int j = 0; j < m; j++) {
            if (S.cnode[cb + j] == xp) ip = j;
            if (S.cnode[cb + j] == xc) ic = j;
        }
        if (ip < 0 || ic < 0 || Cn < 0) {
            S.ctr[C_ERR] |= ERR_INTERNAL;
        } else {
            const int rootB = S.nroot[B];
            for (int j = 0; j < m; j++) S.nd[S.cnode[cb + j]].bpar = -1;
            const int fwd = ((ic - ip) % m + m) % m;
            const int dir = (fwd % 2 == 0) ? 1 : -1;
            const int L = dir > 0 ? fwd : m - fwd;
            int prev = -1;
            for (int j = 0; j <= L; j++) {
                const int idx = ((ip + dir * j) % m + m) % m;
                const int q = S.cnode[cb + idx];
                S.nd[q].label = (j % 2 == 0) ? -1 : 1;
                S.nroot[q] = rootB;
                if (j == 0) {
                    S.tpar[q] = P; S.tps[q] = S.tps[B]; S.tpo[q] = S.tpo[B];
                } else {
                    const int pidx = ((ip + dir * (j - 1)) % m + m) % m;
                    int self, other;
                    if (dir > 0) { self = S.co[cb + pidx]; other = S.cs[cb + pidx]; }
                    else { self = S.cs[cb + idx]; other = S.co[cb + idx]; }
                    S.tpar[q] = prev; S.tps[q] = self; S.tpo[q] = other;
                    if (j % 2 == 1) {
                        S.mate[q] = prev; S.ms[q] = self; S.mo[q] = other;
                        S.mate[prev] = q; S.ms[prev] = other; S.mo[prev] = self;
                    }
                }
                prev = q;
            }
            const int qL = prev;
            S.mate[qL] = Cn; S.ms[qL] = S.ms[B]; S.mo[qL] = S.mo[B];
            S.mate[Cn] = qL; S.tpar[Cn] = qL;
            const int rem = m - 1 - L;
            for (int j = 1; j <= rem; j += 2) {
                const int i1 = ((ic + dir * j) % m + m) % m;
                const int i2 = ((ic + dir * (j + 1)) % m + m) % m;
                const int x = S.cnode[cb + i1], z = S.cnode[cb + i2];
                int lx, lz;
                if (dir > 0) { lx = S.cs[cb + i1]; lz = S.co[cb + i1]; }
                else { lx = S.co[cb + i2]; lz = S.cs[cb + i2]; }
                S.nd[x].label = 0; S.nd[z].label = 0;
                S.tpar[x] = -1; S.tpar[z] = -1;
                S.nroot[x] = -1; S.nroot[z] = -1;
                S.mate[x] = z; S.ms[x] = lx; S.mo[x] = lz;
                S.mate[z] = x; S.ms[z] = lz; S.mo[z] = lx;
            }
            S.nd[B].alive = 0; S.tpar[B] = -1; S.mate[B] = MATE_NONE; S.nd[B].y = 0; S.clen[B] = 0;
            const int nf = S.ctr[C_NFREE];
            S.freel[nf] = B;
            S.ctr[C_NFREE] = nf + 1;
        }
    }
    T.sync();
}

// Fresh growing root for source s.
__device__ __forceinline__ void make_root(const Slab &S, int s) {
    S.nd[s] = NRec{0, -1, 1, 1}; S.src[s].srad = 0;
    S.tpar[s] = -1; S.mate[s] = MATE_NONE; S.nroot[s] = s; S.src[s].stop = s; S.src[s].inplay = 1;
}

enum { RUN_OK = 0, RUN_NOSOL = 1, RUN_BUDGET = 2, RUN_CAP = 3, RUN_INTERNAL = 4 };

// Event loop over the sources with inplay[s] = 1, from t = 0 (SI S1).
template <int NW>
__device__ int run_matcher(const Slab &S, Shot &C, Team<NW> &T, int &nhi) {
    C.t = 0;
    for (;;) {
        if (++C.events > C.max_events) return RUN_BUDGET;
        if (C.deadline && (C.events & 63) == 0) {
            int late = 0;
            if (T.tid() == 0) late = now_ns() > C.deadline;
            if (T.bcast(late)) return RUN_BUDGET;
        }
        unsigned long long best = EMPTY64;
        int flags = 0;   // bit 0: a growing region exists, bit 1: inconsistent state
        unsigned inner_leaf_min = INT_MAX;
        auto src_item = [&](int s) {
            // independent loads first, one dependent load (the label) after
            const int4 r = ld_src(&S.src[s]);
            const int ip = rec_inplay(r), A = r.x, rad = r.y, exh = rec_sexh(r), sR = r.z;
            const unsigned long long bb = ldr(&S.sbnd[s]);
            if (!ip) return;
            const int lab = S.nd[A].label;
            if (lab == 1) {
                flags |= 1;
                if (!exh) {
                    // due when Rad(s) + L would pass the explored radius; a region that
                    // just started growing (or was never explored) is due at once
                    const int ahead = sR - C.L + 1 - rad;
                    best = min(best, ev_key(C.t + (ahead > 0 ? ahead : 0), EV_EXTEND, s, 0));
                }
                if (bb != EMPTY64) {
                    const int bd = (int)(bb >> 32);
                    if (bd < rad) flags |= 2;
                    else best = min(best, ev_key(C.t + (bd - rad), EV_BOUNDARY, s, ID_MAX));
                }
            } else if (lab == -1 && A == s) {
                inner_leaf_min = min(inner_leaf_min, (unsigned)S.nd[s].y);
            }
        };
        auto pair_item = [&](int i) {
            const int4 pq = ld_pr(&S.pr[i]);
            const int a = pq.x, b = pq.y, pv = pq.z;
            if (a < 0) return;
            const int4 qa = ld_src(&S.src[a]), qb = ld_src(&S.src[b]);
            const int ia = rec_inplay(qa), ib = rec_inplay(qb), A = qa.x, B = qb.x;
            const int ra = qa.y, rb = qb.y;
            if (!ia || !ib || A == B) return;
            const int r = S.nd[A].label + S.nd[B].label;
            if (r <= 0) return;
            const int gap = pv - ra - rb;
            if (gap < 0 || gap % r) { flags |= 2; return; }
            best = min(best, ev_key(C.t + gap / r, EV_COLLIDE, a, b));
        };
        auto node_item = [&](int v) {
            const int4 q = ld_nd(&S.nd[v]);
            if constexpr (NW == 1) {
                if (q.w && q.y < 0 && q.z == -1) best = min(best, ev_key(C.t + q.x, EV_IMPLODE, S.minleaf[v], 0));
            } else {
                const int ml = S.minleaf[v];
                if (q.w && q.y < 0 && q.z == -1) best = min(best, ev_key(C.t + q.x, EV_IMPLODE, ml, 0));
            }
        };
        const int np = ldr(&S.ctr[C_NPAIRS]);
        if constexpr (NW == 1) {
            for (int s = T.tid(); s < C.K; s += T.NT) src_item(s);
            for (int i = T.tid(); i < np; i += T.NT) pair_item(i);
            for (int v = C.K + T.tid(); v < nhi; v += T.NT) node_item(v);
        } else {
            // one strided pass over sources, pairs and blossoms together, so
            // every thread of the block gets the same number of items
            const int n1 = C.K, n2 = C.K + np, n3 = np + nhi;
            for (int j = T.tid(); j < n3; j += T.NT) {
                if (j < n1) src_item(j);
                else if (j < n2) pair_item(j - n1);
                else node_item(j - np);
            }
        }
        // the EXTEND list counter is reset ahead of the reduction's barrier
        // (nothing uses it between ball extensions)
        if (T.tid() == 0) S.ctr[C_WL] = 0;
        T.reduce_ev(best, flags, inner_leaf_min);
        if (flags & 2) return RUN_INTERNAL;
        if (!(flags & 1)) return RUN_OK;
        if (best == EMPTY64) return RUN_NOSOL;
        const long long tn = (long long)(best >> 38);
        const int kind = (int)((best >> 36) & 3);
        const int lo = (int)((best >> 18) & ID_MAX);
        const int hi = (int)(best & ID_MAX);
        if (tn >= T_MAX) return RUN_CAP;
        const int dt = (int)(tn - C.t);
        if ((unsigned)dt > inner_leaf_min) return RUN_INTERNAL;
        if (dt > 0) {
            for (int v = T.tid(); v < nhi; v += T.NT) {
                if constexpr (NW == 1) {
                    const int4 q = ld_nd(&S.nd[v]);
                    if (q.w && q.y < 0 && q.z != 0) S.nd[v].y = q.x + q.z * dt;
                } else {
                    const int4 q = ld_nd(&S.nd[v]);
                    if (q.w && q.y < 0 && q.z != 0) S.nd[v].y = q.x + q.z * dt;
                }
            }
            for (int s = T.tid(); s < C.K; s += T.NT) {
                const int4 r = ld_src(&S.src[s]);
                if (rec_inplay(r)) S.src[s].srad = r.y + S.nd[r.x].label * dt;
            }
        }
        C.t = tn;
        if (kind == EV_EXTEND) {
            C.nx++;
        } else {
            C.nm++;
            if (tn <= C.tcut) C.ncut++;
            C.tlast = (int)tn;
        }
        // The dual update above writes y and srad only.  In a block, the next
        // barrier is the one each step below starts with (EXTEND reads the radii
        // after it; the matcher steps read or write no radius before theirs);
        // one warp keeps its barrier here.
        if constexpr (NW == 1) T.sync();
        if (kind == EV_EXTEND) {
            extend_due(S, C, T);
        } else if (kind == EV_IMPLODE) {
            // the blossom is read by every thread before any thread's shatter
            // loop rewrites the stop pointers
            const int B = S.src[lo].stop;
            T.sync();
            ev_shatter(S, C, B, T);
        } else if (kind == EV_BOUNDARY) {
            ev_augment(S, C, S.src[lo].stop, lo, -1, -1, T, nhi);
        } else {
            int a = lo, b = hi;
            int A = S.src[a].stop, B = S.src[b].stop;
            if (S.nd[A].label != 1) { int t = A; A = B; B = t; t = a; a = b; b = t; }
            const int lb = S.nd[B].label;
            // 0 blossom, 1 augment, 2 grow, 3 inconsistent
            int act = 3;
            if (lb == 1) act = S.nroot[A] == S.nroot[B] ? 0 : 1;
            else if (lb == 0 && S.mate[B] == MATE_BOUNDARY) act = 1;
            else if (lb == 0 && S.mate[B] >= 0) act = 2;
            // every thread has read the state it dispatches on before any
            // thread changes it
            T.sync();
            if (act == 0) ev_blossom(S, C, A, a, B, b, T, nhi);
            else if (act == 1) ev_augment(S, C, A, a, B, b, T, nhi);
            else if (act == 2) {
                if (T.tid() == 0) ev_grow(S, A, a, B, b);
                T.sync();
            } else {
                return RUN_INTERNAL;
            }
        }
        // the error word is written only before the barrier that ends each
        // step above and after the next event search's barrier, so every
        // thread reads the same value here
        const int err = ldr(&S.ctr[C_ERR]);
        if (err) return (err & ERR_INTERNAL) ? RUN_INTERNAL : RUN_CAP;
    }
}

__device__ __forceinline__ bool in_commit(const DGraph &g, int v) {
    return (__ldg(g.commit + (v >> 5)) >> (v & 31)) & 1u;
}

// One edge (cur, nxt, id e) of a path: its observables (COMMIT: only when the
// edge touches the commit region, and an endpoint outside the region is
// flipped in `carry`, by the calling thread).
template <bool COMMIT>
__device__ __forceinline__ unsigned long long path_edge(const DGraph &g, int cur, int nxt, int e, bool writer,
                                                        unsigned *carry) {
    if constexpr (COMMIT) {
        const bool ci = in_commit(g, cur), ni = in_commit(g, nxt);
        if (!ci && !ni) return 0;
        if (ci != ni && writer) {
            const int out = ci ? nxt : cur;
            atomicXor(&carry[out >> 5], 1u << (out & 31));
        }
    }
    return __ldg(g.eobs + e);
}

// Canonical path from vertex src (its Dijkstra tree) to vertex x at distance
// dx: predecessor = lowest edge id among tight edges.  Distances come from
// src's list in the ball table, which must cover dx.  One warp; every lane
// returns the XOR of the path's observables (path_edge).
template <bool COMMIT>
__device__ unsigned long long walk_table(const Slab &S, const DGraph &g, int src, int4 h, int x, int dx, int lane,
                                         unsigned *carry) {
    unsigned long long o = 0;
    const int n = dx <= g.b1 ? h.z : h.z + max(h.w, 0);   // (nothing on the path is farther than dx)
    int cur = x, dcur = dx;
    for (int step = 0; step < 1 << 22 && cur != src; step++) {
        const int r0 = __ldg(g.row + cur), deg = __ldg(g.row + cur + 1) - r0;
        unsigned long long best = EMPTY64;
        int dbest = INF32;
        for (int j0 = 0; j0 < deg; j0 += WS) {
            const int j = j0 + lane, nq = min(WS, deg - j0);
            SlotV sl;
            sl.nbr = -1; sl.w = 0; sl.eid = -1;
            if (j < deg) sl = load_slot(g, r0 + j);
            int dy = sl.nbr == src ? 0 : INF32;
            for (int k = 0; k < n; k += WS) {
                int2 e = make_int2(-2, 0);
                if (k + lane < n) e = __ldg(g.ball + (unsigned)h.x + k + lane);
                for (int q = 0; q < nq; q++) {
                    const int y = __shfl_sync(FULL, sl.nbr, q);
                    const unsigned m = __ballot_sync(FULL, e.x == y);
                    if (!m) continue;
                    const int d = __shfl_sync(FULL, e.y, __ffs(m) - 1);
                    if (lane == q) dy = d;
                }
            }
            unsigned long long key = EMPTY64;
            if (sl.nbr >= 0 && dy != INF32 && dy + sl.w == dcur)
                key = ((unsigned long long)(unsigned)__ldg(g.seid + r0 + j) << 32) | (unsigned)sl.nbr;
            const unsigned long long kb = warp_min64(key);
            if (kb < best) {
                best = kb;
                dbest = __shfl_sync(FULL, dy, __ffs(__ballot_sync(FULL, key == kb)) - 1);
            }
        }
        if (best == EMPTY64) { if (lane == 0) set_err(S, ERR_INTERNAL); break; }
        const int nxt = (int)(unsigned)(best & 0xffffffffu);
        o ^= path_edge<COMMIT>(g, cur, nxt, (int)(best >> 32), lane == 0, carry);
        cur = nxt;
        dcur = dbest;
    }
    return o;
}

// The same from source s through its explored ball, which grows until it holds
// dx.  Every thread of the team calls.
template <bool COMMIT, int NW>
__device__ unsigned long long walk_ball(const Slab &S, Shot &C, int s, int x, int dx, Team<NW> &T, unsigned *carry) {
    const DGraph &g = C.g;
    C.paths = 1;
    for (int n = 0; n < 1 << 16; n++) {
        const int more = S.src[s].sR < dx && !S.src[s].sexh && !ldr(&S.ctr[C_ERR]);
        if (!T.bcast(more)) break;
        extend_one(S, C, s, T);
    }
    // a ball that outgrew the tables: the attempt is retried with larger ones
    if (T.bcast(ldr(&S.ctr[C_ERR]))) return 0;
    unsigned long long o = 0;
    const int src = S.svtx[s];
    int cur = x, dcur = dx;
    for (int n = 0; n < 1 << 22 && cur != src; n++) {
        const int r0 = __ldg(g.row + cur), r1 = __ldg(g.row + cur + 1);
        unsigned long long best = EMPTY64;
        for (int j = r0 + T.tid(); j < r1; j += T.NT) {
            SlotV sl = load_slot(g, j);
            if (sl.nbr < 0) continue;
            const int dy = ht_get(S, C, sl.nbr, s);
            if (dy != INF32 && dy + sl.w == dcur)
                best = min(best, ((unsigned long long)(unsigned)__ldg(g.seid + j) << 32) | (unsigned)sl.nbr);
        }
        best = T.min64(best);
        if (best == EMPTY64) { if (T.tid() == 0) S.ctr[C_ERR] |= ERR_INTERNAL; break; }
        const int nxt = (int)(unsigned)(best & 0xffffffffu);
        o ^= path_edge<COMMIT>(g, cur, nxt, (int)(best >> 32), T.tid() == 0, carry);
        cur = nxt;
        dcur = ht_get(S, C, cur, s);
    }
    T.sync();
    return o;
}

// Distance of two matched events: their edge is tight, so it is the sum of
// their radii less twice the duals of the blossoms that hold both.
__device__ int tight_dist(const Slab &S, int a, int b) {
    int d = S.src[a].srad + S.src[b].srad;
    for (int B = S.nd[a].bpar; B >= 0; B = S.nd[B].bpar) {
        int x = S.nd[b].bpar;
        while (x >= 0 && x != B) x = S.nd[x].bpar;
        if (x == B) {
            for (; B >= 0; B = S.nd[B].bpar) d -= 2 * S.nd[B].y;
            break;
        }
    }
    return d;
}

// Weight (internal units) and observable of the final matching.  Every matched
// edge is tight and every set with a dual has exactly one matched edge leaving
// it, so the weight is the sum of all duals; the observable is that of the
// boundary matches' edges, which the matched top-level nodes name.
template <int NW>
__device__ __forceinline__ void total(const Slab &S, const Shot &C, Team<NW> &T, int nhi, long long &wint,
                                      unsigned long long &obs) {
    long long w = 0;
    unsigned long long o = 0;
    for (int v = T.tid(); v < nhi; v += T.NT) {
        const int4 q = ld_nd(&S.nd[v]);
        if (!q.w) continue;
        w += q.x;
        if (q.y < 0 && S.mate[v] == MATE_BOUNDARY) {
            const unsigned long long bb = S.sbnd[S.ms[v]];
            if (bb == EMPTY64) set_err(S, ERR_INTERNAL);
            else o ^= __ldg(C.g.eobs + (int)(unsigned)(bb & 0xffffffffu));
        }
    }
    wint = T.sum64(w);
    obs = T.xor64(o);
}

// Expand the final matching into leaf-level pairs (tmpa[i], tmpb[i] at distance
// cst2[i]; tmpb = -1 for a boundary match); returns their number.
template <int NW>
__device__ int expand(const Slab &S, Shot &C, Team<NW> &T, int nhi) {
    // matched top-level nodes, team-parallel: each match appends its leaf pair
    // and queues the blossoms on either side for expansion (stack seeds)
    if (T.tid() == 0) { S.ctr[C_TNP] = 0; S.ctr[C_TNX] = 0; }
    T.sync();
    int *stk = S.stk;
    for (int v = T.tid(); v < nhi; v += T.NT) {
        if (!S.nd[v].alive || S.nd[v].bpar >= 0) continue;
        const int mt = S.mate[v];
        if (mt == MATE_BOUNDARY) {
            const int k = agg_inc(&S.ctr[C_TNP], T.lane);
            S.tmpa[k] = S.ms[v]; S.tmpb[k] = -1;
            if (v >= C.K) { const int x = atomicAdd(&S.ctr[C_TNX], 1); stk[2 * x] = v; stk[2 * x + 1] = S.ms[v]; }
        } else if (mt >= 0 && v < mt) {
            const int k = agg_inc(&S.ctr[C_TNP], T.lane);
            S.tmpa[k] = S.ms[v]; S.tmpb[k] = S.mo[v];
            if (v >= C.K) { const int x = atomicAdd(&S.ctr[C_TNX], 1); stk[2 * x] = v; stk[2 * x + 1] = S.ms[v]; }
            if (mt >= C.K) { const int x = atomicAdd(&S.ctr[C_TNX], 1); stk[2 * x] = mt; stk[2 * x + 1] = S.mo[v]; }
        }
    }
    T.sync();
    int np = ldr(&S.ctr[C_TNP]);
    if (T.tid() == 0) {
        // blossoms: the child holding the externally matched leaf keeps that
        // match, the other children pair up along the cycle
        const int stk_cap = 4 * C.nc + 60;
        int sp = 2 * ldr(&S.ctr[C_TNX]);
        while (sp > 0) {
            const int ext = stk[--sp];
            const int node = stk[--sp];
            if (node < C.K) continue;
            const int m = S.clen[node], cb = S.cbeg[node];
            const int c0 = ext >= 0 ? child_of(S, node, ext) : -1;
            if (c0 < 0 || m <= 0) { S.ctr[C_ERR] |= ERR_INTERNAL; break; }
            int i0 = 0;
            for (int j = 0; j < m; j++) if (S.cnode[cb + j] == c0) i0 = j;
            if (sp + 2 * m + 2 > stk_cap || np + m > 2 * C.nc) { S.ctr[C_ERR] |= ERR_CAP; break; }
            stk[sp++] = c0; stk[sp++] = ext;
            for (int j = 1; j < m; j += 2) {
                const int i1 = (i0 + j) % m, i2 = (i0 + j + 1) % m;
                const int lx = S.cs[cb + i1], lz = S.co[cb + i1];
                S.tmpa[np] = lx; S.tmpb[np] = lz; np++;
                stk[sp++] = S.cnode[cb + i1]; stk[sp++] = lx;
                stk[sp++] = S.cnode[cb + i2]; stk[sp++] = lz;
            }
        }
    }
    np = T.bcast(np);
    T.sync();
    for (int i = T.tid(); i < np; i += T.NT)   // boundary matches: the boundary distance
        S.cst2[i] = S.tmpb[i] < 0 ? (int)(S.sbnd[S.tmpa[i]] >> 32) : tight_dist(S, S.tmpa[i], S.tmpb[i]);
    T.sync();
    return np;
}

// Hash table sizes of a shot with C.K events: about 8 (rarely ~15) explored
// entries and 1 (at most ~2) pair per event at the design point; the tables
// stay at most half full or the shot is retried with larger ones.
__device__ __forceinline__ unsigned next_pow2(unsigned x) {
    x--; x |= x >> 1; x |= x >> 2; x |= x >> 4; x |= x >> 8; x |= x >> 16;
    return x + 1;
}
__device__ __forceinline__ void set_tables(const BatchArgs &A, Shot &C, unsigned scale) {
    C.ec = A.caps.ec; C.wc = A.caps.wc; C.cc = A.caps.cc;
    C.pcap = A.caps.phc >> 1;
    C.hmask = min(next_pow2(max(128u, (unsigned)QEC_HT_FACTOR * (unsigned)C.K * scale)), (unsigned)A.caps.hc) - 1;
    C.pmask = min(next_pow2(max(64u, 4u * (unsigned)C.K * scale)), (unsigned)A.caps.phc) - 1;
}

// Walk the canonical paths of a matching: np pairs of events tmpa[i], tmpb[i]
// (-1: boundary) at distance cst2[i].  COMMIT (sliding windows): the correction
// is the union of those paths and of the boundary edges; every edge that
// touches the graph's commit region is committed, and the shot's carry row
// receives the detectors outside the region flipped by committed edges.
// Otherwise the result is the observables of the paths' edges.  A path within
// the ball table's reach is walked by one warp; one that cannot leave its side
// of the region's border (g.seam) commits nothing but its observables, and is
// not walked when those edges carry none.  Farther paths are walked through
// explored balls, for which a fast-path shot (scale > 0) sets up its tables
// first.  svtx: the events' vertices.  Every thread of the team calls.
template <bool COMMIT, int NW>
__device__ __noinline__ unsigned long long walk_paths(const BatchArgs &A, const Slab &S, Shot &C, Team<NW> T,
                                                      const int *svtx, int np, unsigned scale, unsigned *carry) {
    const DGraph &g = C.g;
    if constexpr (COMMIT)
        for (int w = T.tid(); w < g.words; w += T.NT) carry[w] = 0u;
    if (T.tid() == 0) {
        S.ctr[C_TNX] = 0;
        if (scale) S.ctr[C_ERR] = 0;
    }
    T.sync();
    unsigned long long mine = 0, whole = 0;   // found by this lane / by this warp together
    for (int base = T.warp() * WS; base < np; base += T.NT) {
        const int i = base + T.lane;
        int v = 0, x = 0, dx = 0;
        int4 h = make_int4(0, 0, 0, 0);
        bool walk = false;
        if (i < np) {
            const int a = S.tmpa[i], b = S.tmpb[i];
            int s = a;
            dx = S.cst2[i];
            if (b < 0) {
                const int e = (int)(unsigned)(__ldg(g.vbnd + svtx[a]) & 0xffffffffu);
                const int2 ue = __ldg(g.eend + e);
                x = ue.x;
                dx -= ue.y;
                if constexpr (COMMIT) if (in_commit(g, x)) mine ^= __ldg(g.eobs + e);   // the boundary edge itself
            } else {
                s = min(a, b);
                x = svtx[max(a, b)];
            }
            v = svtx[s];
            bool skip = false;
            if constexpr (COMMIT) skip = dx < __ldg(g.seam + v) && (!g.internal_obs || !in_commit(g, v));
            h = __ldg(g.bhdr + v);
            const int cover = h.w >= 0 ? g.brad : (h.z >= 0 ? g.b1 : -1);
            if (!skip && dx > 0) {
                walk = dx <= cover;
                if (!walk) S.stk[atomicAdd(&S.ctr[C_TNX], 1)] = i;
            }
        }
        for (unsigned m = __ballot_sync(FULL, walk); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const int4 hl = make_int4(__shfl_sync(FULL, h.x, l), 0, __shfl_sync(FULL, h.z, l), __shfl_sync(FULL, h.w, l));
            whole ^= walk_table<COMMIT>(S, g, __shfl_sync(FULL, v, l), hl, __shfl_sync(FULL, x, l),
                                        __shfl_sync(FULL, dx, l), T.lane, carry);
        }
    }
    T.sync();
    unsigned long long o = T.xor64(mine ^ (T.lane == 0 ? whole : 0));
    const int nfar = T.bcast(ldr(&S.ctr[C_TNX]));
    if (nfar == 0 || T.bcast(ldr(&S.ctr[C_ERR]))) return o;
    C.paths = 1;
    if (!C.real) {   // no ball is explored yet
        if (scale) {
            set_tables(A, C, scale);
            for (int i = T.tid(); i < C_TOTAL; i += T.NT) S.ctr[i] = 0;
        }
        for (int s = T.tid(); s < C.K; s += T.NT) {
            S.src[s].sR = -1; S.src[s].sexh = 0;
            S.scnt[s] = 0; S.sbeg[s] = 0;
            S.svtx[s] = svtx[s];
        }
        T.sync();
    }
    for (int k = 0; k < nfar; k++) {
        if (T.bcast(ldr(&S.ctr[C_ERR]))) break;
        const int i = S.stk[k];
        const int a = S.tmpa[i], b = S.tmpb[i], d = S.cst2[i];
        if (b < 0) {
            const int2 ue = __ldg(g.eend + (unsigned)(__ldg(g.vbnd + S.svtx[a]) & 0xffffffffu));
            o ^= walk_ball<COMMIT>(S, C, a, ue.x, d - ue.y, T, carry);
        } else {
            o ^= walk_ball<COMMIT>(S, C, min(a, b), S.svtx[max(a, b)], d, T, carry);
        }
    }
    T.sync();
    return o;
}

// Per-shot counters; the tables themselves are already empty (release_tables).
template <int NW>
__device__ void clear_tables(const Slab &S, const Shot &C, Team<NW> &T) {
    for (int i = T.tid(); i < C_TOTAL; i += T.NT) S.ctr[i] = 0;
    T.sync();
}

// Return the explored and pair tables to empty: the slots recorded in the band
// lists (every explored entry) and the pair list (every pair), or with `all`
// the whole region of this attempt's table sizes.
template <int NW>
__device__ __noinline__ void release_tables(const Slab &S, const Shot &C, Team<NW> T, bool all) {
    T.sync();
    const HEnt e = HEnt{EMPTY64, -1, -1};
    if (all) {
        for (unsigned i = T.tid(); i <= C.hmask; i += T.NT) S.ht[i] = e;
        for (unsigned i = T.tid(); i <= C.pmask; i += T.NT) S.pt[i] = e;
    } else {
        const int ne = ldr(&S.ctr[C_ECOUNT]), np = min(ldr(&S.ctr[C_NPAIRS]), C.pcap);
        for (int i = T.tid(); i < ne; i += T.NT) S.ht[S.ent[i] & C.hmask] = e;
        for (int i = T.tid(); i < np; i += T.NT) {
            const int sl = S.pr[i].slot;
            if (sl >= 0) S.pt[sl & C.pmask] = e;
        }
    }
    T.sync();
}

// Compact the set bits of the shot's syndrome row into S.svtx; returns K
// (or -1 when K exceeds kcap).  One warp.
__device__ int load_defects(const Slab &S, const DGraph &g, const unsigned *row, int kcap, int wcap, int lane) {
    int K = 0;
    const int nvec = g.words >> 2;
    const uint4 *rv = reinterpret_cast<const uint4 *>(row);
    for (int base = 0; base < nvec; base += WS) {
        const int i = base + lane;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (i < nvec) v = __ldg(rv + i);
        unsigned wv[4] = {v.x, v.y, v.z, v.w};
        // drop padding bits beyond n
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int bit0 = (i * 4 + q) * 32;
            if (bit0 >= g.n) wv[q] = 0;
            else if (bit0 + 32 > g.n) wv[q] &= (1u << (g.n - bit0)) - 1u;
        }
        int c = __popc(wv[0]) + __popc(wv[1]) + __popc(wv[2]) + __popc(wv[3]);
        int incl = c;
#pragma unroll
        for (int o = 1; o < WS; o <<= 1) {
            int t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(FULL, incl, WS - 1);
        int pos = K + incl - c;
        if (i < nvec && i * 4 + 3 < wcap) {
            S.wcum[i * 4 + 0] = pos;
            S.wcum[i * 4 + 1] = pos + __popc(wv[0]);
            S.wcum[i * 4 + 2] = pos + __popc(wv[0]) + __popc(wv[1]);
            S.wcum[i * 4 + 3] = pos + __popc(wv[0]) + __popc(wv[1]) + __popc(wv[2]);
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
            unsigned bits = wv[q];
            while (bits) {
                const int b = __ffs(bits) - 1;
                bits &= bits - 1;
                if (pos < kcap) S.svtx[pos] = (i * 4 + q) * 32 + b;
                pos++;
            }
        }
        K += total;
    }
    __syncwarp();
    return K > kcap ? -1 : K;
}

// Pairs of events within b_1, each once (from its lower-ranked end), read off
// the ball table: one lane per (event, entry of its vertex's list of higher
// vertices within b_1), numbered by a warp prefix sum of the list lengths; the
// warps of a team take 32 events each in turn.  Numbering the entries keeps
// every lane busy although the lists differ in length (12 on average, fewer at
// the code's sides), and half of each neighbourhood is enough since a pair is
// found from its lower end.  Also the events' boundary distances (canonical
// boundary edge in the low word).  Returns (per thread) bit 0: an event's list
// is not complete, bit 1: an event has more than LB_CAP vertices within b_1 on
// a graph where b_1 spans more than two edges.  Every thread of the team
// calls; ends with a barrier.
constexpr int LB_CAP = 64;
template <int NW>
__device__ __forceinline__ int near_pairs(const Slab &S, const Shot &C, Team<NW> &T) {
    const DGraph &g = C.g;
    const int lane = T.lane;
    int flags = 0, np = 0;
    for (int base = T.warp() * WS; base < C.K; base += T.NT) {
        const int s = base + lane;
        int beg = 0, len = 0;
        if (s < C.K) {
            const int v = S.svtx[s];
            const int4 h = __ldg(g.bhdr + v);
            S.sbnd[s] = __ldg(g.vbnd + v);
            if (h.z < 0) {
                flags |= 1;
            } else {
                beg = h.x;
                len = h.y;
                if (!g.hop2 && h.z >= LB_CAP) flags |= 2;
            }
        }
        int incl = len;
#pragma unroll
        for (int o = 1; o < WS; o <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(FULL, incl, WS - 1);
        const int excl = incl - len;
        for (int t0 = 0; t0 < total; t0 += WS) {
            const int t = t0 + lane;
            int ow = 0;   // owner: the last lane whose first entry number is <= t
#pragma unroll
            for (int step = WS / 2; step > 0; step >>= 1) {
                const int e = __shfl_sync(FULL, excl, ow + step);
                if (e <= t) ow += step;
            }
            const unsigned oj = (unsigned)__shfl_sync(FULL, beg - excl, ow) + (unsigned)t;
            bool hit = false;
            int2 e = make_int2(0, 0);
            unsigned word = 0;
            if (t < total) {
                e = __ldg(g.ball + oj);
                word = __ldg(C.row + (e.x >> 5));
                hit = (word >> (e.x & 31)) & 1u;
            }
            const unsigned m = __ballot_sync(FULL, hit);
            if (!m) continue;
            int b;
            if constexpr (NW == 1) {
                b = np;
                np += __popc(m);
            } else {
                b = 0;
                if (lane == 0) b = atomicAdd(&S.ctr[C_NPAIRS], __popc(m));
                b = __shfl_sync(FULL, b, 0);
            }
            if (hit) {
                const int j = b + __popc(m & ((1u << lane) - 1u));
                const int f = S.wcum[e.x >> 5] + __popc(word & ((1u << (e.x & 31)) - 1u));
                if (j < C.pcap) S.pr[j] = PRec{base + ow, f, (unsigned)e.y, -1};
                else set_err(S, ERR_CAP);
            }
        }
    }
    if constexpr (NW == 1)
        if (lane == 0) S.ctr[C_NPAIRS] = np;
    T.sync();
    return flags;
}

constexpr int LEVEL1_OVERLAP = -6;

// Decode one shot with hash tables scaled by `scale`; returns QEC_SHOT_*, -1
// when the working set overflowed (retry with a larger scale), or
// LEVEL1_OVERLAP when two accepted level-1 clusters have grown into each other.
// (A cluster of odd size stops as late as its nearest boundary contact plus its
// diameter, which can pass the b_1 / 2 that keeps clusters apart.  Their duals
// together are then no solution, and the shot is decoded without level 1.)
// WIN: sliding-window mode (BatchArgs::carry set), compiled as its own kernel so
// that the ordinary kernel carries none of its code.
template <bool WIN, int NW>
__device__ int decode_attempt_body(const BatchArgs &A, int mode, const Slab &S, const DGraph &g, const unsigned *row,
                                   Team<NW> &T, unsigned scale, unsigned long long deadline, long long &w_out,
                                   unsigned long long &o_out, int *dg, Shot &C) {
    C.g = g;
    C.band = max(g.wmax, 1) * max(A.band_factor, 1);
    C.events = 0;
    C.t = 0;
    C.deadline = deadline;
    C.row = row;
    C.L = max(g.wmax, (g.b1 + 1) / 2) + 1;
    C.nm = 0; C.ncut = 0; C.tcut = 0; C.tlast = 0; C.nx = 0;
    C.real = 0;
    if (g.words > A.caps.wcap) return -2;
    int K = 0;
    if (T.warp() == 0) K = load_defects(S, g, row, A.caps.kc, A.caps.wcap, T.lane);
    K = T.bcast(K);
    T.sync();
    if (K < 0) return -2;
    C.K = K;
    C.max_events = min(A.max_events, 256LL * K + 4096);
    if (K == 0) {
        w_out = 0; o_out = 0;
        if (dg && T.tid() < QEC_DIAG_FIELDS) dg[T.tid()] = 0;   // no detection event: E_ideal = 0
        if constexpr (WIN)
            for (int w = T.tid(); w < g.words; w += T.NT) A.carry[(row - A.syn) + w] = 0u;
        return QEC_SHOT_OK;
    }
    if (K > ID_MAX - 1 || 2 * K + 8 > A.caps.nc) return -2;
    C.nc = min(A.caps.nc, 2 * K + 16);   // leaves + at most K blossoms alive at once
    set_tables(A, C, scale);
    clear_tables(S, C, T);
    // sources, leaf nodes, free list
    int nhi = K;
    for (int s = T.tid(); s < K; s += T.NT) {
        S.src[s] = SRec{s, 0, -1, 0, 0, 0, 0}; S.scnt[s] = 0; S.sbeg[s] = 0;
        S.nd[s] = NRec{0, -1, 0, 0}; S.tpar[s] = -1;
        S.mate[s] = MATE_NONE; S.nroot[s] = -1; S.minleaf[s] = s; S.clen[s] = 0;
    }
    const int nfree = C.nc - K;
    for (int i = T.tid(); i < nfree; i += T.NT) {
        const int v = C.nc - 1 - i;   // pop order: K, K+1, ...
        S.freel[i] = v;
        S.nd[v] = NRec{0, -1, 0, 0}; S.clen[v] = 0;
    }
    if (T.tid() == 0) { S.ctr[C_ECOUNT] = 0; S.ctr[C_NFREE] = nfree; }
    T.sync();
    // level-1 critical path (stopping time, event count), clusters, events
    // resolved at level 1, events of all level-1 runs
    int t1 = 0, e1 = 0, ncl1 = 0, nres1 = 0, ntot = 0;
    int gr = K;   // next level-1 cluster (its lowest event) that needs the event loop
    // every pair within b_1 and every boundary distance.  An event whose list
    // is not complete needs explored balls from the start.
    const int odd = T.template red32<2>(near_pairs(S, C, T));
    const int Rbig = max(g.b1, C.band);   // level-1 ball of an event with many vertices within b_1
    if ((odd & 1) || ((odd & 2) && reach_of(C, Rbig) > g.b1)) go_real(S, C, T);
    if (mode == QEC_MODE_HIERARCHICAL) {
        // ---- Algorithm 1, level 1.  An event with more than LB_CAP vertices
        // within b_1 gets its first ball here
        if (odd) {
            if (T.tid() == 0) S.ctr[C_WL] = 0;
            T.sync();
            for (int s = T.tid(); s < K; s += T.NT) {
                const int nb = __ldg(g.bhdr + S.svtx[s]).z;
                if (nb >= 0 && (nb < LB_CAP || g.hop2)) continue;
                if (!C.real) { S.src[s].sR = Rbig; continue; }
                const int k = atomicAdd(&S.ctr[C_WL], 1);
                S.xsrc[k] = s;
                S.xR[k] = Rbig;
            }
            T.sync();
            const int nx = T.bcast(ldr(&S.ctr[C_WL]));
            T.sync();
            extend_many<true>(S, C, nx, T);
        }
    }
    {
        const int err = T.bcast(ldr(&S.ctr[C_ERR]));
        if (err) return (err & ERR_INTERNAL) ? QEC_SHOT_INTERNAL : -1;
    }
    if (mode == QEC_MODE_HIERARCHICAL) {
        const int npairs = T.bcast(ldr(&S.ctr[C_NPAIRS]));
        // connected components of pairs within b_1: min-label propagation
        for (int s = T.tid(); s < K; s += T.NT) { S.comp[s] = s; S.cst0[s] = 0; S.cst1[s] = 0; S.cst2[s] = 0; }
        T.sync();
        for (int round = 0; round <= K; round++) {
            bool changed = false;
            for (int i = T.tid(); i < npairs; i += T.NT) {
                const int4 pq = ld_pr(&S.pr[i]);
                const int a = pq.x, b = pq.y;
                if (a < 0 || pq.z > g.b1) continue;
                const int la = ldr(&S.comp[a]), lb = ldr(&S.comp[b]);
                if (la != lb) {
                    const int m = min(la, lb);
                    atomicMin(&S.comp[a], m);
                    atomicMin(&S.comp[b], m);
                    changed = true;
                }
            }
            T.sync();
            if (!T.any(changed)) break;
        }
        for (int s = T.tid(); s < K; s += T.NT) {
            const int r = S.comp[s];
            atomicAdd(&S.cst0[r], 1);
            const unsigned long long bb = S.sbnd[s];
            if (bb != EMPTY64 && 2LL * (long long)(bb >> 32) <= (long long)g.b1) atomicOr(&S.cst1[r], 1);
        }
        T.sync();
        // pairs within d_1 inside a component; each such pair is also noted at
        // its two events (xcur is free until the flooder runs): the pair of an
        // accepted two-event cluster
        for (int i = T.tid(); i < npairs; i += T.NT) {
            const int4 pq = ld_pr(&S.pr[i]);
            const int a = pq.x, b = pq.y;
            if (a < 0 || pq.z > g.d1) continue;
            if (S.comp[a] == S.comp[b]) {
                atomicAdd(&S.cst2[S.comp[a]], 1);
                S.xcur[a] = i;
                S.xcur[b] = i;
            }
        }
        T.sync();
        // ---- level-1 clusters: closed forms for isolated pairs / boundary singletons
        bool need_general = false;
        for (int s = T.tid(); s < K; s += T.NT) {
            const int r = S.comp[s];
            const int size = S.cst0[r];
            const bool ok = (long long)S.cst2[r] == (long long)size * (size - 1) / 2 &&
                            ((S.cst1[r] & 1) || size % 2 == 0);
            if (!ok) continue;
            if (size == 1) {
                const int bd = (int)(S.sbnd[s] >> 32);
                S.nd[s] = NRec{bd, -1, 0, 1}; S.src[s].srad = bd;
                S.mate[s] = MATE_BOUNDARY; S.ms[s] = s; S.mo[s] = -1; S.src[s].stop = s; S.nroot[s] = -1;
                t1 = max(t1, bd); ncl1++; nres1++;   // one boundary event at time bd
            } else if (size == 2) {
                // the cluster's one pair within d_1
                const int4 pq = ld_pr(&S.pr[S.xcur[s]]);
                const int other = pq.x == s ? pq.y : pq.x, d = pq.z;
                const long long ba = (long long)(S.sbnd[s] >> 32), bo = (long long)(S.sbnd[other] >> 32);
                if (d / 2 <= ba && d / 2 <= bo) {
                    S.nd[s] = NRec{d / 2, -1, 0, 1}; S.src[s].srad = d / 2;
                    S.mate[s] = other; S.ms[s] = s; S.mo[s] = other; S.src[s].stop = s; S.nroot[s] = -1;
                    t1 = max(t1, d / 2); nres1++;   // one collision at time d/2
                    if (s < other) ncl1++;
                } else {
                    need_general = true;
                    atomicOr(&S.cst1[r], 2);   // solve with the event loop
                }
            } else {
                need_general = true;
                atomicOr(&S.cst1[r], 2);
            }
        }
        T.sync();
        t1 = T.maxi(t1);
        ncl1 = T.add(ncl1);
        nres1 = T.add(nres1);
        e1 = ncl1 > 0 ? 1 : 0;
        ntot = ncl1;
        need_general = T.any(need_general);
        gr = need_general ? 0 : K;
    }
    // ---- level-1 clusters without a closed form, one run each (from an empty
    // state apart from themselves), then the top level: every remaining event
    // from t = 0 with the stopped level-1 configurations present as frozen
    // regions (global mode: every event, from an empty state).  One call site
    // of the event loop serves both, which keeps the kernel's hot code small.
    bool ran = false;
    for (int guard = 0; guard <= K + 1; guard++) {
        while (gr < K && (S.comp[gr] != gr || !(S.cst1[gr] & 2))) gr++;
        const bool top = gr >= K;
        if (top && ran) {
            // (the larger of two regions has recorded the pair, see reach_of)
            const int np = T.bcast(ldr(&S.ctr[C_NPAIRS]));
            bool overlap = false;
            for (int i = T.tid(); i < np; i += T.NT) {
                const int4 pq = ld_pr(&S.pr[i]);
                const int a = pq.x, b = pq.y;
                if (a >= 0 && S.comp[a] != S.comp[b]) overlap |= S.src[a].srad + S.src[b].srad > pq.z;
            }
            if (T.any(overlap)) return LEVEL1_OVERLAP;
        }
        if (top) {
            for (int s = T.tid(); s < K; s += T.NT) {
                if (S.nd[s].alive || S.src[s].stop != s) S.src[s].inplay = 1;   // stopped level-1 configuration
                else make_root(S, s);
            }
            C.ncut = 0;
            C.tcut = t1;
        } else {
            for (int s = T.tid(); s < K; s += T.NT)
                if (S.comp[s] == gr) make_root(S, s);
        }
        T.sync();
        C.nm = 0;
        C.tlast = 0;
        const int st = run_matcher(S, C, T, nhi);
        if (st != RUN_OK) {
            if (st == RUN_CAP) return -1;
            return st == RUN_NOSOL ? QEC_SHOT_NO_SOLUTION
                   : st == RUN_BUDGET ? QEC_SHOT_BUDGET_EXCEEDED : QEC_SHOT_INTERNAL;
        }
        if (top) break;
        ran = true;
        for (int s = T.tid(); s < K; s += T.NT)
            if (S.comp[s] == gr) S.src[s].inplay = 0;
        T.sync();
        e1 = max(e1, C.nm); t1 = max(t1, C.tlast); ntot += C.nm; ncl1++; nres1 += S.cst0[gr];
        gr++;
    }
    long long wint = 0;
    unsigned long long ob = 0;
    total(S, C, T, nhi, wint, ob);
    if (WIN || g.internal_obs) {
        // sliding window: the committed part; else the observables of
        // detector-detector edges
        const int npath = expand(S, C, T, nhi);
        if (T.bcast(ldr(&S.ctr[C_ERR])) == 0) {
            const unsigned long long po = walk_paths<WIN>(A, S, C, T, S.svtx, npath, 0,
                                                          WIN ? A.carry + (row - A.syn) : nullptr);
            ob = WIN ? po : ob ^ po;
        }
    }
    const int err = T.bcast(ldr(&S.ctr[C_ERR]));
    if (err) return (err & ERR_INTERNAL) ? QEC_SHOT_INTERNAL : -1;
    w_out = wint / 2;
    o_out = ob;
    if (dg && T.tid() == 0) {
        // parallel event count over level 1 and the top level (Methods,
        // "Numerical evaluation"): the top run's events up to the level-1
        // critical-path time t1 overlap level 1, the rest extend it
        const int ntop = C.nm;
        dg[QEC_DIAG_E_IDEAL] = ntop > 0 ? max(e1, C.ncut) + ntop - C.ncut : e1;
        dg[QEC_DIAG_T_IDEAL] = ntop > 0 ? max(t1, C.tlast) : t1;
        dg[QEC_DIAG_EVENTS] = ntot + ntop;
        dg[QEC_DIAG_L1_CLUSTERS] = ncl1;
        dg[QEC_DIAG_L1_DEFECTS] = nres1;
        dg[QEC_DIAG_TOP_EVENTS] = ntop;
        dg[QEC_DIAG_BANDS] = C.nx;
        dg[QEC_DIAG_DEFECTS] = K;
    }
    return QEC_SHOT_OK;
}

// One decode attempt.  The explored and pair tables are empty (all-ones) on
// entry and are returned empty: after a successful shot only the slots listed
// in the band lists and the pair list are reset, after anything else the
// whole region the attempt could have used.
template <bool WIN, int NW>
__device__ int decode_attempt(const BatchArgs &A, int mode, const Slab &S, const DGraph &g, const unsigned *row, Team<NW> &T,
                              unsigned scale, unsigned long long deadline, long long &w_out,
                              unsigned long long &o_out, int *dg) {
    Shot C;
    C.real = 0;
    C.paths = 0;
    const int st = decode_attempt_body<WIN, NW>(A, mode, S, g, row, T, scale, deadline, w_out, o_out, dg, C);
    // (the tables are used by explored balls only)
    if (C.real || C.paths) release_tables(S, C, T, st != QEC_SHOT_OK);
    return st;
}

// ---------------------------------------------------------------- islands --
//
// The events left after level 1 fall into islands: the components of Algorithm
// 1's level-1 graph (pairs within b_1) that were not accepted.  Two islands,
// or an island and a stopped level-1 cluster, are more than b_1 apart, so they
// hardly ever touch, and what touches only in its own island runs the same
// events in the same order alone as inside one run over everything: the state
// changes are disjoint and the canonical order restricted to an island is the
// order of its own events.  So each island is run by itself, one warp each with
// the whole state in shared memory, and afterwards every recorded pair that
// joins two of them is checked: where the largest radii reach its distance, the
// two are joined (an accepted cluster's events frozen as level 1 left them) and
// run again.  A pair whose regions meet is always recorded: within b_1 it is
// listed from the start, beyond it the extensions of the larger of the two
// regions reach the other's event (Fast::reach) unless both are past
// Fast::cap, which wide_apart checks.  Since the smaller region need not have it,
// a record is kept for as long as the island that made it stands.
//
// A run over everything costs a scan of all events and pairs per event: a d =
// 51 window at p = 0.003 (1,170 events, 250 matcher events in 88 islands of at
// most ~12 events) spent 87 % of its time there, a d = 21 shot (6 islands) 67 %.
// Something is joined in 0.5 % of d = 21 shots and 11 % of those windows.
//
// Shots outside the limits below take the run over everything (the general
// path).  The phases are separate functions whose loops are not unrolled, and
// what they share lies in shared memory: unrolled, the million-shot batch was 40 %
// slower (15.6 against 11.0 ms), waiting for instructions.
constexpr int TOP_BITS = 7, TOP_MASK = (1 << TOP_BITS) - 1, RAD_SHIFT = TOP_BITS + 2;

// What one island, or several, add to the shot (w: internal units).
struct __align__(16) IslRec {
    unsigned long long o;
    int w, size;
    int nm, ncut, tlast, nx;   // matcher events, those at times <= tcut, time of the last, bands counted here
};

// An island: E events per lane.  E = 1 lies in shared memory; E = 2, for the few
// islands that need it (0.1 % of circuit-level d = 13 shots, 1 % of d = 51
// windows at p = 0.005), in the slab.
template <int E>
struct __align__(16) Isl {
    static constexpr int IN = 32 * E;    // events; blossoms are nodes IN .. 2 IN - 1
    static constexpr int IP = E == 1 ? 64 : 256;   // pairs
    static constexpr int IC = 96 * E;    // blossom cycle entries
    static constexpr int LB = 4 + E;     // bits of an event in a key
    int2 pair[IP];        // distance, lower event | higher event << 8
    int pk[IN];           // per event: radius << 9 | (label of its top node + 1) << 7 | top node
    int y[2 * IN];        // duals of the blossoms
    int ev[IN], bd[IN];   // event of the shot, boundary distance
    int xt[IN];           // radius at which the explored radius falls due (NEVER: ball exhausted)
    int meet[IN];         // radius at which the region touches what stands outside (NEVER: nothing so far)
    IslRec rec;           // result
    signed char lab[2 * IN], bpar[2 * IN], tpar[2 * IN], tps[2 * IN], tpo[2 * IN];
    signed char mate[2 * IN], ms[2 * IN], mo[2 * IN], root[2 * IN], minl[2 * IN];
    unsigned char cn[IC], cs[IC], co[IC], cb[IN], cl[IN];   // cycles: child, its leaf, the next child's leaf
    signed char ta[2 * IN], tb[2 * IN];                     // tree paths / expansion stack
    int nc, err;
    __device__ __forceinline__ int top(int e) const { return pk[e] & TOP_MASK; }
    __device__ __forceinline__ int rad(int e) const { return pk[e] >> RAD_SHIFT; }
    __device__ __forceinline__ void set_top(int e, int v) { pk[e] = (pk[e] & ~TOP_MASK) | v; }
};

enum { ST_RUN = -3, ST_ONE = -4, ST_TWO = -5 };
constexpr unsigned CW_OPEN = 1u << 30, CW_SIDE = 1u << 31;
// frozen at the start of the top level
__device__ __forceinline__ bool st_frozen(int st) { return st >= 0 || st == MATE_BOUNDARY || st == ST_RUN; }
constexpr int NEVER = 1 << 30;   // past every radius
enum { ISL_FAIL = 0, ISL_OK = 1, ISL_STOP = 2, ISL_BIG = 3 };
constexpr unsigned ISL_ALONE = 1u << 31;
constexpr unsigned long long MET = 1ull << 27;   // in a pair: its events' regions meet
enum { F_NP = 0, F_N1 = 1, F_N2 = 2, F_AGED = 3, F_NPATH = 4, F_STOP = 5, F_NALL = 6, F_FAIL = 7, F_WIDE = 8, F_TOTAL = 12 };   // Fast::cnt

// The shot being decoded by a team.  Per-event arrays, `stride` ints each, in
// shared memory or, for shots with more events than it holds, in the slab:
//   svtx  vertex                      bd  boundary distance (INT_MAX: none)
//   comp  lowest event of the component
//   px    nearest event: distance << 12 | event (all ones: none within b_1),
//         later the largest radius
//   st    level-1 state: the partner or MATE_BOUNDARY in a closed form,
//         ST_RUN: in a level-1 cluster of more events; a growing root of the
//         top level: MATE_NONE, or ST_ONE / ST_TWO in an island solved in
//         closed form (ST_TWO: the higher event of a pair)
//   cw    at a component's lowest event: size | pairs within d_1 << 12 | not
//         in closed form << 30 | boundary contact << 31; in an island, the
//         event's lane
// and the pairs, lo << 46 | hi << 28 | distance.
struct __align__(16) Fast {
    const DGraph *g;
    const unsigned *row;
    const int *wcum;
    int *ev;
    unsigned long long *pr;
    IslRec *recs;                      // of the islands, by their lowest event
    int *list, *all;                   // clusters and islands to run; all islands once some were joined
    int *aged_t, *aged_c, *aged_n;     // bands of regions that came of age: time, island, its size
    int *pa, *pb, *pd;                 // matched pairs for the path walks
    int *was;                          // after a join: radii of what stands, -1: what runs again
    char *spare;                       // room for larger islands, nspare bytes
    int nspare, nlist;                 // nlist: room in the lists above
    int path0, path1;                  // matched pairs of the level-1 clusters run
    int late;                          // every island has run once, see `was`
    int stride, pcap, K, np0, tcut, L, band, cap, paths;
    int cnt[F_TOTAL];
    __device__ __forceinline__ int *svtx() const { return ev; }
    __device__ __forceinline__ int *bd() const { return ev + stride; }
    __device__ __forceinline__ int *comp() const { return ev + 2 * stride; }
    __device__ __forceinline__ int *px() const { return ev + 3 * stride; }
    __device__ __forceinline__ int *st() const { return ev + 4 * stride; }
    __device__ __forceinline__ unsigned *cw() const { return reinterpret_cast<unsigned *>(ev + 5 * stride); }
    __device__ __forceinline__ bool defect(int v) const { return (__ldg(row + (v >> 5)) >> (v & 31)) & 1u; }
    __device__ __forceinline__ int rank(int v) const {
        return wcum[v >> 5] + __popc(__ldg(row + (v >> 5)) & ((1u << (v & 31)) - 1u));
    }
    // Radius within which the other events have to be known once a ball has
    // radius R, as reach_of, but taking no other region to be larger than `cap`;
    // pairs of regions that are both larger are checked at the end (wide_apart).
    // No region grows past its event's boundary distance.
    __device__ __forceinline__ int reach(int b1, int R, int bd) const {
        const int r = min(R - L, bd);
        return r + min(max(r, (b1 + 1) >> 1), cap);
    }
};

// Shared memory of a team: the shot, per-event arrays of shots with at most KS
// events, and one island per warp.
template <int NW>
struct __align__(16) FastShared {
    static constexpr int KS = NW == 1 ? 128 : (NW == TEAM_MID ? 1280 : 2048), PS = KS + KS / 4;
    Fast f;
    unsigned long long pr[PS];
    int ev[6 * KS];
    Isl<1> isl[NW];
};

__device__ __forceinline__ unsigned long long pk_pair(int a, int b, int d) {
    return ((unsigned long long)(unsigned)a << 46) | ((unsigned long long)(unsigned)b << 28) | (unsigned)d;
}
__device__ __forceinline__ int pr_lo(unsigned long long p) { return (int)(p >> 46); }
__device__ __forceinline__ int pr_hi(unsigned long long p) { return (int)(p >> 28) & 0x3ffff; }
__device__ __forceinline__ int pr_val(unsigned long long p) { return (int)(p & (MET - 1)); }

template <int E>
__device__ __forceinline__ int isl_child_of(const Isl<E> &I, int B, int leaf) {
    int v = leaf;
#pragma unroll 1
    for (int k = 0; k < I.IN && v >= 0 && I.bpar[v] != B; k++) v = I.bpar[v];
    return v;
}

// flip matches along the tree path from outer A to its root (lane 0; I.err when
// the path is no tree path)
template <int E>
__device__ __forceinline__ void isl_flip(Isl<E> &I, int A) {
    int v = A;
#pragma unroll 1
    for (int k = 0; I.tpar[v] >= 0; k++) {
        const int i = I.tpar[v], o = I.tpar[i];
        if (o < 0 || k >= I.IN) { I.err = 1; return; }
        I.mate[i] = (signed char)o; I.ms[i] = I.tps[i]; I.mo[i] = I.tpo[i];
        I.mate[o] = (signed char)i; I.ms[o] = I.tpo[i]; I.mo[o] = I.tps[i];
        v = o;
    }
}

// Event (c): the new blossom N over outer A, B of one tree.  `bal`: blossoms
// alive before.  Returns false when the cycle pool is full or the paths do not
// meet.  One warp.
template <int E>
__device__ __noinline__ bool isl_blossom(Isl<E> &I, int N, int A, int a, int B, int b, int n, unsigned long long bal,
                                         int lane) {
    constexpr int IN = Isl<E>::IN, IC = Isl<E>::IC;
    int ok = 1;
    if (lane == 0) {
        int na = 0, nb = 0;
#pragma unroll 1
        for (int v = A; v >= 0 && na < 2 * IN; v = I.tpar[v]) I.ta[na++] = (signed char)v;
#pragma unroll 1
        for (int v = B; v >= 0 && nb < 2 * IN; v = I.tpar[v]) I.tb[nb++] = (signed char)v;
#pragma unroll 1
        while (na > 1 && nb > 1 && I.ta[na - 2] == I.tb[nb - 2]) { na--; nb--; }
        const int Lc = I.ta[na - 1], m = na + nb - 1, cb = I.nc;
        if (cb + m > IC || Lc != I.tb[nb - 1]) {
            ok = 0;
        } else {
            I.nc = cb + m;
            int i = 0;
            I.cn[cb + i++] = (unsigned char)Lc;
#pragma unroll 1
            for (int j = na - 2; j >= 0; j--) I.cn[cb + i++] = (unsigned char)I.ta[j];
#pragma unroll 1
            for (int j = 0; j <= nb - 2; j++) I.cn[cb + i++] = (unsigned char)I.tb[j];
            const int ia = na - 1;
            int ml = IN;
#pragma unroll 1
            for (int j = 0; j < m; j++) {
                const int x = I.cn[cb + j], z = I.cn[cb + (j + 1 < m ? j + 1 : 0)];
                if (j < ia) { I.cs[cb + j] = I.tpo[z]; I.co[cb + j] = I.tps[z]; }
                else if (j == ia) { I.cs[cb + j] = (unsigned char)a; I.co[cb + j] = (unsigned char)b; }
                else { I.cs[cb + j] = I.tps[x]; I.co[cb + j] = I.tpo[x]; }
                ml = min(ml, (int)I.minl[x]);
                I.bpar[x] = (signed char)N;
            }
            I.y[N] = 0; I.lab[N] = 1; I.bpar[N] = -1;
            I.tpar[N] = I.tpar[Lc]; I.tps[N] = I.tps[Lc]; I.tpo[N] = I.tpo[Lc];
            I.mate[N] = I.mate[Lc]; I.ms[N] = I.ms[Lc]; I.mo[N] = I.mo[Lc];
            I.root[N] = I.root[Lc] == Lc ? (signed char)N : I.root[Lc];
            I.minl[N] = (signed char)ml;
            I.cb[N - IN] = (unsigned char)cb; I.cl[N - IN] = (unsigned char)m;
        }
    }
    if (!__shfl_sync(FULL, ok, 0)) return false;
    __syncwarp();
    const int L0 = I.cn[I.cb[N - IN]];   // if it was its tree's root, N is now
#pragma unroll 1
    for (int h = 0; h < 2 * E; h++) {
        const int v = lane + h * WS;
        if (h < E ? v >= n : !((bal >> (v - IN)) & 1ull)) continue;
        if (I.bpar[v] >= 0) continue;
        const int tp = I.tpar[v], mt = I.mate[v];
        if (tp >= 0 && I.bpar[tp] == N) I.tpar[v] = (signed char)N;
        if (mt >= 0 && I.bpar[mt] == N) I.mate[v] = (signed char)N;
        if (I.root[v] == L0) I.root[v] = (signed char)N;
    }
#pragma unroll 1
    for (int e = lane; e < n; e += WS)
        if (I.bpar[I.top(e)] == N) I.set_top(e, N);
    __syncwarp();
    return true;
}

// Event (d): inner blossom B shatters (I.err on an inconsistent state).  One warp.
template <int E>
__device__ __noinline__ void isl_shatter(Isl<E> &I, int B, int n, int lane) {
    constexpr int IN = Isl<E>::IN;
#pragma unroll 1
    for (int e = lane; e < n; e += WS)
        if (I.top(e) == B) I.set_top(e, max(0, isl_child_of(I, B, e)));
    __syncwarp();
    if (lane == 0) {
        const int m = I.cl[B - IN], cb = I.cb[B - IN];
        const int P = I.tpar[B], Cn = I.mate[B];
        const int xp = isl_child_of(I, B, I.tps[B]), xc = isl_child_of(I, B, I.ms[B]);
        int ip = -1, ic = -1;
#pragma unroll 1
        for (int j = 0; j < m; j++) {
            if (I.cn[cb + j] == xp) ip = j;
            if (I.cn[cb + j] == xc) ic = j;
        }
        if (ip < 0 || ic < 0 || Cn < 0) {
            I.err = 1;
        } else {
#pragma unroll 1
            for (int j = 0; j < m; j++) I.bpar[I.cn[cb + j]] = -1;
            auto wrap = [&](int j) { j %= m; return j < 0 ? j + m : j; };
            const int fwd = wrap(ic - ip), dir = (fwd % 2 == 0) ? 1 : -1, Ln = dir > 0 ? fwd : m - fwd;
            int prev = -1;
#pragma unroll 1
            for (int j = 0; j <= Ln; j++) {
                const int idx = wrap(ip + dir * j), q = I.cn[cb + idx];
                I.lab[q] = (j % 2 == 0) ? -1 : 1;
                I.root[q] = I.root[B];
                if (j == 0) {
                    I.tpar[q] = (signed char)P; I.tps[q] = I.tps[B]; I.tpo[q] = I.tpo[B];
                } else {
                    const int pidx = wrap(ip + dir * (j - 1));
                    const int self = dir > 0 ? I.co[cb + pidx] : I.cs[cb + idx];
                    const int other = dir > 0 ? I.cs[cb + pidx] : I.co[cb + idx];
                    I.tpar[q] = (signed char)prev; I.tps[q] = (signed char)self; I.tpo[q] = (signed char)other;
                    if (j % 2 == 1) {
                        I.mate[q] = (signed char)prev; I.ms[q] = (signed char)self; I.mo[q] = (signed char)other;
                        I.mate[prev] = (signed char)q; I.ms[prev] = (signed char)other; I.mo[prev] = (signed char)self;
                    }
                }
                prev = q;
            }
            I.mate[prev] = (signed char)Cn; I.ms[prev] = I.ms[B]; I.mo[prev] = I.mo[B];
            I.mate[Cn] = (signed char)prev; I.tpar[Cn] = (signed char)prev;
#pragma unroll 1
            for (int j = 1; j <= m - 1 - Ln; j += 2) {
                const int i1 = wrap(ic + dir * j), i2 = wrap(ic + dir * (j + 1));
                const int x = I.cn[cb + i1], z = I.cn[cb + i2];
                const int lx = dir > 0 ? I.cs[cb + i1] : I.co[cb + i2], lz = dir > 0 ? I.co[cb + i1] : I.cs[cb + i2];
                I.lab[x] = 0; I.lab[z] = 0;
                I.tpar[x] = -1; I.tpar[z] = -1;
                I.root[x] = -1; I.root[z] = -1;
                I.mate[x] = (signed char)z; I.ms[x] = (signed char)lx; I.mo[x] = (signed char)lz;
                I.mate[z] = (signed char)x; I.ms[z] = (signed char)lz; I.mo[z] = (signed char)lx;
            }
            I.lab[B] = 0; I.y[B] = 0;
        }
    }
    __syncwarp();
}

// Distance of two matched events of an island (as tight_dist).
template <int E>
__device__ __forceinline__ int isl_dist(const Isl<E> &I, int a, int b) {
    int d = I.rad(a) + I.rad(b);
    int B = I.bpar[a];
#pragma unroll 1
    for (int k = 0; k < I.IN && B >= 0; k++, B = I.bpar[B])   // at most IN blossoms hold an event
        if (isl_child_of(I, B, b) >= 0) break;
#pragma unroll 1
    for (int k = 0; k < I.IN && B >= 0; k++, B = I.bpar[B]) d -= 2 * I.y[B];
    return d;
}

// A matched pair of the shot (b = -1: boundary) at distance d, for the path walks.
__device__ __forceinline__ void put_path(Fast &X, int a, int b, int d) {
    const int k = atomicAdd(&X.cnt[F_NPATH], 1);   // at most one per event
    X.pa[k] = a; X.pb[k] = b; X.pd[k] = d;
}

// The matched pairs of a finished island.  One warp.
template <int E>
__device__ __noinline__ void isl_paths(Fast &X, Isl<E> &I, int n, unsigned long long bal, int lane) {
    constexpr int IN = Isl<E>::IN;
#pragma unroll 1
    for (int h = 0; h < 2 * E; h++) {
        const int v = lane + h * WS;
        if (h < E ? v >= n : !((bal >> (v - IN)) & 1ull)) continue;
        if (I.bpar[v] >= 0) continue;
        const int mt = I.mate[v], s = I.ms[v];
        if (mt == MATE_BOUNDARY) put_path(X, I.ev[s], -1, I.bd[s]);
        else if (v < mt) put_path(X, I.ev[s], I.ev[I.mo[v]], isl_dist(I, s, I.mo[v]));
    }
    if (lane != 0) return;
    // inside blossoms: the child holding the externally matched leaf keeps that
    // match, the other children pair up along the cycle
#pragma unroll 1
    for (int b = IN; b < 2 * IN; b++) {
        int sp = 0;
        if (!((bal >> (b - IN)) & 1ull) || I.bpar[b] >= 0) continue;
        I.ta[sp] = (signed char)b; I.tb[sp++] = I.ms[b];
#pragma unroll 1
        for (int k = 0; k < 2 * IN && sp > 0; k++) {   // each node of the blossom once
            const int v = I.ta[--sp], e = I.tb[sp];
            if (v < IN) continue;
            const int len = I.cl[v - IN], cb = I.cb[v - IN], c0 = isl_child_of(I, v, e);
            if (sp + len > 2 * IN) break;
            int i0 = 0;
#pragma unroll 1
            for (int j = 0; j < len; j++) if (I.cn[cb + j] == c0) i0 = j;
            I.ta[sp] = (signed char)c0; I.tb[sp++] = (signed char)e;
#pragma unroll 1
            for (int j = 1; j < len; j += 2) {
                const int i1 = (i0 + j) % len, i2 = (i0 + j + 1) % len;
                const int lx = I.cs[cb + i1], lz = I.co[cb + i1];
                put_path(X, I.ev[lx], I.ev[lz], isl_dist(I, lx, lz));
                I.ta[sp] = (signed char)I.cn[cb + i1]; I.tb[sp++] = (signed char)lx;
                I.ta[sp] = (signed char)I.cn[cb + i2]; I.tb[sp++] = (signed char)lz;
            }
        }
    }
}

// Events farther from vertex v than the ball table's radius, up to q <= 2 brad -
// 2 wmax: the shortest path to such an event passes a detector y at a distance
// in (r - wmax, r] from v, r = q - brad + wmax <= brad, and the rest of it is
// shorter than brad, so the event is in the list of one of those y.  Lane j gets
// the j-th event found (rank f, exact distance d); returns their number, or -1
// when a list is not complete or more than 32 are found.  One warp.
__device__ __noinline__ int far_events(const Fast &X, int v, int q, int lane, int &f, int &d) {
    const DGraph &g = *X.g;
    const int4 h = __ldg(g.bhdr + v);
    const int n = h.z + max(h.w, 0), r = q - g.brad + g.wmax, brad = g.brad, wmax = g.wmax;
    int found = 0;
    f = -1;
    d = INT_MAX;
#pragma unroll 1
    for (int k = 0; k < n; k += WS) {
        int2 e = make_int2(0, 0);
        int4 he = make_int4(0, 0, 0, 0);
        bool use = false;
        if (k + lane < n) {
            e = __ldg(g.ball + (unsigned)h.x + k + lane);
            use = e.y > r - wmax && e.y <= r;
            if (use) he = __ldg(g.bhdr + e.x);
        }
        if (__any_sync(FULL, he.w < 0)) return -1;
        const int beg = he.x, len = he.z + he.w;
#pragma unroll 1
        for (unsigned m = __ballot_sync(FULL, use); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const int dy = __shfl_sync(FULL, e.y, l), ly = __shfl_sync(FULL, len, l);
            const int2 *const list = g.ball + (unsigned)__shfl_sync(FULL, beg, l);
#pragma unroll 1
            for (int j = 0; j < ly; j += 4 * WS) {   // four loads in flight
                int2 x[4];
                unsigned hit = 0;
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    x[u] = make_int2(v, 0);
                    if (j + u * WS + lane < ly) x[u] = __ldg(list + j + u * WS + lane);
                }
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (dy + x[u].y > brad && dy + x[u].y <= q && x[u].x != v && X.defect(x[u].x)) hit |= 1u << u;
                if (!__any_sync(FULL, hit)) continue;
#pragma unroll
                for (int u = 0; u < 4; u++) {
#pragma unroll 1
                    for (unsigned mh = __ballot_sync(FULL, (hit >> u) & 1u); mh; mh &= mh - 1) {
                        const int o = __ffs(mh) - 1;
                        const int ro = X.rank(__shfl_sync(FULL, x[u].x, o)), dr = dy + __shfl_sync(FULL, x[u].y, o);
                        const unsigned same = __ballot_sync(FULL, f == ro);
                        if (!same) {
                            if (found == WS) return -1;
                            if (lane == found) { f = ro; d = dr; }
                            found++;
                        } else if (f == ro) {
                            d = min(d, dr);
                        }
                    }
                }
            }
        }
    }
    return found;
}

// EXTEND in the island of c (as extend_due): the events that its due regions
// can touch until they fall due again are read off the ball table and recorded
// among the shot's pairs, those of the island itself also in I.pair.  Returns
// the island's pairs, -1 outside the limits, -2 beyond the table.  One warp.
template <int E>
__device__ __noinline__ int isl_extend(Fast &X, Isl<E> &I, int c, int n, int np, bool level1, int lane) {
    constexpr int IP = Isl<E>::IP;
    const DGraph &g = *X.g;
    const int b1 = g.b1, brad = g.brad, wmax = g.wmax;
    const int *const comp = X.comp(), *const st = X.st(), *const px = X.px();
    unsigned scan[E];
    bool far = false;
#pragma unroll
    for (int h = 0; h < E; h++) {
        const int e = lane + h * WS;
        bool sc = false;
        if (e < n) {
            const int p = I.pk[e], rad = p >> RAD_SHIFT, xt = I.xt[e];
            if (((p >> TOP_BITS) & 3) == 2 && xt <= rad) {
                const int sR = xt + X.L - 1;   // explored radius, -1: never
                const int R = max(sR + X.band, rad + X.L + X.band), bd = I.bd[e], q = X.reach(b1, R, bd);
                sc = sR >= 0 || q > b1;
                if (min(R - X.L, bd) > X.cap) X.cnt[F_WIDE] = 1;
                if (!sc) I.xt[e] = R - X.L + 1;
                far |= sc && (q > max(brad, min(2 * brad - 2 * wmax, 6 * wmax + 8)) ||
                              (sR > brad - wmax && R - X.L < bd) ||   // (else it never falls due again)
                              __ldg(g.bhdr + X.svtx()[I.ev[e]]).w < 0);
            }
        }
        scan[h] = __ballot_sync(FULL, sc);
    }
    if (__any_sync(FULL, far)) return -2;
#pragma unroll 1
    for (int i = 0; i < Isl<E>::IN; i++) {
        if (!((scan[i >> 5] >> (i & 31)) & 1u)) continue;
        const int s = I.ev[i], sRl = I.xt[i] + X.L - 1;
        const int R = max(sRl + X.band, I.rad(i) + X.L + X.band), ql = X.reach(b1, R, I.bd[i]);
        const int q0 = sRl < 0 ? b1 : max(b1, X.reach(b1, sRl, I.bd[i]));
        const int v = X.svtx()[s];
        const int4 h = __ldg(g.bhdr + v);
        const int len = h.z + h.w;
        bool more = false;
        // the list's own events, then those beyond it
        int nfar = 0, ff = 0, fd = 0;
        if (ql > brad) nfar = far_events(X, v, ql, lane, ff, fd);
        if (nfar < 0) return -1;
#pragma unroll 1
        for (int k = 0; k < len + (nfar ? WS : 0); k += WS) {
            bool hit = false;
            int f = 0, d = 0;
            if (k < len) {
                if (k + lane < len) {
                    const int2 e = __ldg(g.ball + (unsigned)h.x + k + lane);
                    more |= e.y > sRl;
                    hit = e.y > q0 && e.y <= ql && X.defect(e.x);
                    d = e.y;
                    if (hit) f = X.rank(e.x);
                }
            } else {
                hit = lane < nfar && fd > q0;
                f = ff;
                d = fd;
            }
            const unsigned mh = __ballot_sync(FULL, hit);
            if (!mh) continue;
            const bool in = hit && comp[f] == c;
            // a level-1 cluster stands still unless it is touched, and so does,
            // once every island has run, one that does not run again.  (Others'
            // radii are being written now: they would stop this island, or not, as
            // the warps happen to be timed.)
            int rf = -1;
            if (hit && !in) {
                if (X.late) rf = X.was[f];
                else if (st_frozen(st[f]) && !(level1 && st[f] == ST_RUN)) rf = px[f];
            }
            const int mt = __reduce_min_sync(FULL, rf >= 0 ? d - rf : INT_MAX);
            if (lane == 0) I.meet[i] = min(I.meet[i], mt);
            int b = 0;
            if (lane == 0) b = atomicAdd(&X.cnt[F_NP], __popc(mh));
            b = __shfl_sync(FULL, b, 0) + __popc(mh & ((1u << lane) - 1u));
            if (hit && b < X.pcap) X.pr[b] = pk_pair(min(s, f), max(s, f), d);
            // inside the island: unless the other event has it recorded
            const int k2 = in ? (int)X.cw()[f] : 0;
            const bool add = in && (I.xt[k2] != NEVER && d > max(b1, X.reach(b1, I.xt[k2] + X.L - 1, I.bd[k2])));
            const unsigned mi = __ballot_sync(FULL, add);
            const int j = np + __popc(mi & ((1u << lane) - 1u));
            if (add && j < IP) I.pair[j] = make_int2(d, min(i, k2) | max(i, k2) << 8);
            np += __popc(mi);
            if (np > IP || __any_sync(FULL, hit && b >= X.pcap)) return -1;
        }
        more = __any_sync(FULL, more);
        if (lane == 0) I.xt[i] = sRl >= 0 && !more && sRl <= brad - wmax ? NEVER : R - X.L + 1;
        __syncwarp();
    }
    __syncwarp();
    return np;
}

// Run the island of the component with lowest event c and `size` events from t
// = 0 (SI S1, events as in run_matcher): growing roots and, in an island that
// was joined with level-1 clusters, their events frozen as level 1 left them.
// level1: a level-1 cluster (its bands are counted here; the top level's aged
// bands are collected, since regions due at the same time share one).  One
// warp.  The result is left in I.rec.  Returns ISL_FAIL when the island is
// outside the limits, ISL_BIG when a larger E has room, ISL_STOP when a region
// touched a level-1 cluster outside or outgrew the ball table (the radii so far
// are in px, cw[c] is ISL_ALONE).
template <int E>
__device__ __forceinline__ int run_island(Fast &X, Isl<E> &I, int c, int size, bool level1, int lane) {
    constexpr int IN = Isl<E>::IN, IP = Isl<E>::IP, LB = Isl<E>::LB;
    constexpr unsigned DT_END = (1u << (30 - 2 * LB)) - 1u;
    if (size > IN) return ISL_BIG;
    const int n = size;
    {
        // members in rank order: the first is c, the others are near it
        const int *const comp = X.comp();
        unsigned *const cw = X.cw();
        const int K = X.K;
        int k = 0;
#pragma unroll 1
        for (int base = c; base < K && k < n; base += WS) {
            const int s = base + lane;
            const bool in = s < K && comp[s] == c;
            const unsigned m = __ballot_sync(FULL, in);
            if (in) {
                const int j = k + __popc(m & ((1u << lane) - 1u));
                I.ev[j] = s;
                cw[s] = (unsigned)j;   // its place
            }
            k += __popc(m);
        }
    }
    __syncwarp();
    int rad[E], top[E];
    bool bad = false;
#pragma unroll
    for (int h = 0; h < E; h++) {
        const int e = lane + h * WS;
        rad[h] = 0;
        top[h] = e;
        if (e < n) {
            const int ev = I.ev[e], bd = X.bd()[ev];
            const int st = level1 ? (int)MATE_NONE : X.st()[ev];
            const bool frozen = st_frozen(st);
            bad |= st == ST_RUN;
            if (st == MATE_BOUNDARY) rad[h] = bd;   // (a frozen pair's radius: with its pair below)
            I.bd[e] = bd;
            // explored radius after the first extension, due at t = 0, which the listed pairs cover
            I.xt[e] = frozen ? -X.L : X.band + 1;
            I.meet[e] = NEVER;
            I.pk[e] = rad[h] << RAD_SHIFT | e;
            I.lab[e] = frozen ? 0 : 1; I.bpar[e] = -1; I.tpar[e] = -1;
            I.mate[e] = frozen ? MATE_BOUNDARY : MATE_NONE; I.ms[e] = (signed char)e; I.mo[e] = -1;
            I.root[e] = frozen ? -1 : (signed char)e; I.minl[e] = (signed char)e;
        }
    }
    if (lane == 0) { I.nc = 0; I.err = 0; }
    if (__any_sync(FULL, bad)) return ISL_FAIL;
    __syncwarp();
    int np = 0;
    {
        const unsigned long long *const pr = X.pr;
        const int *const comp = X.comp(), np0 = X.np0;
#pragma unroll 1
        for (int base = 0; base < np0; base += WS) {
            const int i = base + lane;
            unsigned long long p = 0;
            bool in = false;
            if (i < np0) {
                p = pr[i];
                in = comp[pr_lo(p)] == c;
            }
            const unsigned m = __ballot_sync(FULL, in);
            if (!m) continue;
            const int k = np + __popc(m & ((1u << lane) - 1u));
            if (in && k < IP) {
                const int a = (int)X.cw()[pr_lo(p)], b = (int)X.cw()[pr_hi(p)], d = pr_val(p);
                I.pair[k] = make_int2(d, a | b << 8);
                if (!level1 && X.st()[pr_lo(p)] == pr_hi(p)) {   // a level-1 pair: frozen, matched at d / 2
                    I.pk[a] = d / 2 << RAD_SHIFT | a;
                    I.pk[b] = d / 2 << RAD_SHIFT | b;
                    I.mate[a] = (signed char)b; I.mo[a] = (signed char)b;
                    I.mate[b] = (signed char)a; I.mo[b] = (signed char)a;
                }
            }
            np += __popc(m);
        }
    }
    if (np > IP) return ISL_BIG;
    __syncwarp();
    int yl[E], mrad[E], lab[E];   // the leaf's dual, the largest radius so far, the label of its top node
    unsigned bal[E];              // blossoms alive
#pragma unroll
    for (int h = 0; h < E; h++) {
        if (lane + h * WS < n) rad[h] = I.rad(lane + h * WS);
        yl[h] = mrad[h] = rad[h];
        bal[h] = 0;
    }
    // (by value to the functions out of line: a reference would put it in memory)
    auto alive = [&]() { return E == 1 ? (unsigned long long)bal[0] : bal[0] | (unsigned long long)bal[E - 1] << 32; };
    int t = 0, nm = 0, ncut = 0, tlast = 0, nx = level1 ? 1 : 0;
#pragma unroll 1
    for (int it = 0;; it++) {
        if (it > 200 * n || t >= (1 << 21)) return ISL_FAIL;   // far below the shot's event budget
        bool grows = false;
#pragma unroll
        for (int h = 0; h < E; h++) {
            const int e = lane + h * WS;
            lab[h] = 0;
            if (e < n) {
                lab[h] = I.lab[top[h]];
                I.pk[e] = rad[h] << RAD_SHIFT | (lab[h] + 1) << TOP_BITS | top[h];
            }
            grows |= lab[h] == 1;
        }
        if (!__any_sync(FULL, grows)) break;
        __syncwarp();
        // next event: key dt | kind | lo | hi; touching a level-1 cluster
        // outside is kind EXTEND with hi = 1
        unsigned key = ~0u;
        auto cand = [&](int dt, int kind, int lo, int hi) {
            if ((unsigned)dt < DT_END) key = min(key, ((unsigned)dt << (2 + 2 * LB)) | (unsigned)(kind << (2 * LB) | lo << LB | hi));
        };
#pragma unroll
        for (int h = 0; h < E; h++) {
            const int e = lane + h * WS;
            bad |= rad[h] < 0;   // two regions past Fast::cap have met without knowing each other
            if (lab[h] == 1) {
                const int bd = I.bd[e];
                bad |= bd < rad[h];
                cand(max(0, I.xt[e] - rad[h]), EV_EXTEND, e, 0);
                cand(max(0, I.meet[e] - rad[h]), EV_EXTEND, e, 1);
                cand(bd - rad[h], EV_BOUNDARY, e, 0);
            }
        }
#pragma unroll 1
        for (int p = lane; p < np; p += WS) {
            const int2 pq = I.pair[p];
            const int a = pq.y & 255, b = pq.y >> 8;
            const int ka = I.pk[a], kb = I.pk[b];
            const int r = ((ka >> TOP_BITS) & 3) + ((kb >> TOP_BITS) & 3) - 2;
            if (((ka ^ kb) & TOP_MASK) == 0 || r <= 0) continue;
            const int gap = pq.x - (ka >> RAD_SHIFT) - (kb >> RAD_SHIFT);
            bad |= gap < 0 || (gap & (r - 1)) != 0;
            cand(gap >> (r - 1), EV_COLLIDE, a, b);
        }
#pragma unroll
        for (int h = 0; h < E; h++)
            if ((bal[h] >> lane) & 1u) {
                const int v = IN + lane + h * WS;
                if (I.bpar[v] < 0 && I.lab[v] == -1) cand(I.y[v], EV_IMPLODE, I.minl[v], 0);
            }
        if (__any_sync(FULL, bad)) return ISL_FAIL;
        key = __reduce_min_sync(FULL, key);
        if (key == ~0u) return ISL_FAIL;   // no event left (no solution), or far away
        const int dt = (int)(key >> (2 + 2 * LB)), kind = (int)(key >> (2 * LB)) & 3;
        const int lo = (int)(key >> LB) & (IN - 1), hi = (int)key & (IN - 1);
        t += dt;
        if (dt > 0) {
#pragma unroll
            for (int h = 0; h < E; h++) {
                rad[h] += lab[h] * dt;
                mrad[h] = max(mrad[h], rad[h]);
                if (top[h] == lane + h * WS) yl[h] += lab[h] * dt;
                if ((bal[h] >> lane) & 1u) {
                    const int v = IN + lane + h * WS;
                    if (I.bpar[v] < 0) I.y[v] += I.lab[v] * dt;
                }
            }
        }
        if (kind == EV_EXTEND) {
            int r = -2;
            if (!hi) {
#pragma unroll
                for (int h = 0; h < E; h++)
                    if (lane + h * WS < n) I.pk[lane + h * WS] = rad[h] << RAD_SHIFT | (lab[h] + 1) << TOP_BITS | top[h];
                __syncwarp();
                r = isl_extend(X, I, c, n, np, level1, lane);
                if (r == -1) return ISL_BIG;
            }
            if (r == -2) {
#pragma unroll
                for (int h = 0; h < E; h++)
                    if (lane + h * WS < n) X.px()[I.ev[lane + h * WS]] = mrad[h];
                if (lane == 0) { X.cw()[c] = ISL_ALONE; atomicAdd(&X.cnt[F_STOP], 1); }
                __syncwarp();
                return ISL_STOP;
            }
            np = r;
            // a band: counted at once, except that at the top level regions of
            // several islands coming of age at one time share it
            if (level1 || dt == 0) {
                nx++;
            } else if (lane == 0) {
                const int k = atomicAdd(&X.cnt[F_AGED], 1);
                if (k < X.nlist) { X.aged_t[k] = t; X.aged_c[k] = c; X.aged_n[k] = n; }
            }
            continue;
        }
        nm++;
        if (t <= X.tcut) ncut++;
        tlast = t;
        bool tops = false;   // the events' top nodes changed
        if (kind == EV_IMPLODE) {
            const int B = I.top(lo);
            __syncwarp();   // every lane has read it before the shatter moves the event to another node
            isl_shatter(I, B, n, lane);
#pragma unroll
            for (int h = 0; h < E; h++)
                if (((B - IN) >> 5) == h) bal[h] &= ~(1u << (B & 31));
            tops = true;
        } else {
            int a = lo, b = hi, A = I.top(a), B = -1;
            if (kind == EV_COLLIDE) {
                B = I.top(b);
                if (I.lab[A] != 1) { int x = A; A = B; B = x; x = a; a = b; b = x; }
            }
            const int lb = B >= 0 ? I.lab[B] : 0, mb = B >= 0 ? (int)I.mate[B] : (int)MATE_BOUNDARY;
            const int rA = I.root[A], rB = lb == 1 ? I.root[B] : -3;
            __syncwarp();
            if (lb == 1 && rA == rB) {
                int N = -1;
#pragma unroll
                for (int h = 0; h < E; h++)
                    if (N < 0 && bal[h] != ~0u) N = IN + h * WS + __ffs(~bal[h]) - 1;
                if (N < 0 || !isl_blossom(I, N, A, a, B, b, n, alive(), lane)) return ISL_BIG;
#pragma unroll
                for (int h = 0; h < E; h++)
                    if (((N - IN) >> 5) == h) bal[h] |= 1u << (N & 31);
                tops = true;
            } else if (lb == 1 || mb == MATE_BOUNDARY) {
                // augment: the trees' nodes leave them while lane 0 rematches
                // along the tree paths
#pragma unroll
                for (int h = 0; h < 2 * E; h++) {
                    const int v = lane + h * WS;
                    if (h < E ? v >= n : !((bal[h < E ? 0 : h - E] >> lane) & 1u)) continue;
                    if (I.bpar[v] < 0 && I.lab[v] != 0 && (I.root[v] == rA || I.root[v] == rB)) { I.lab[v] = 0; I.root[v] = -1; }
                }
                if (lane == 0) {
                    isl_flip(I, A);
                    if (B >= 0) {
                        if (lb == 1) isl_flip(I, B);
                        I.mate[A] = (signed char)B; I.ms[A] = (signed char)a; I.mo[A] = (signed char)b;
                        I.mate[B] = (signed char)A; I.ms[B] = (signed char)b; I.mo[B] = (signed char)a;
                    } else {
                        I.mate[A] = MATE_BOUNDARY; I.ms[A] = (signed char)a; I.mo[A] = -1;
                    }
                }
            } else if (lb == 0 && mb >= 0) {
                if (lane == 0) {   // grow
                    I.lab[B] = -1; I.tpar[B] = (signed char)A; I.tps[B] = (signed char)b; I.tpo[B] = (signed char)a;
                    I.root[B] = (signed char)rA;
                    I.lab[mb] = 1; I.tpar[mb] = (signed char)B; I.tps[mb] = I.ms[mb]; I.tpo[mb] = I.mo[mb];
                    I.root[mb] = (signed char)rA;
                }
            } else {
                return ISL_FAIL;
            }
        }
        __syncwarp();
        if (I.err) return ISL_FAIL;
        if (tops) {
#pragma unroll
            for (int h = 0; h < E; h++)
                if (lane + h * WS < n) top[h] = I.top(lane + h * WS);
        }
    }
    // result: the duals' sum, the boundary matches' observables, largest radii
    int w = 0;
    unsigned long long o = 0;
#pragma unroll
    for (int h = 0; h < E; h++) {
        const int e = lane + h * WS, v = IN + e;
        if (e < n) {
            w += yl[h];
            X.px()[I.ev[e]] = mrad[h];
            if (I.bpar[e] < 0 && I.mate[e] == MATE_BOUNDARY) o ^= __ldg(X.g->vobs + X.svtx()[I.ev[I.ms[e]]]);
        }
        if ((bal[h] >> lane) & 1u) {
            w += I.y[v];
            if (I.bpar[v] < 0 && I.mate[v] == MATE_BOUNDARY) o ^= __ldg(X.g->vobs + X.svtx()[I.ev[I.ms[v]]]);
        }
    }
    if (X.paths) {
        __syncwarp();
        isl_paths(X, I, n, alive(), lane);
    }
    w = (int)__reduce_add_sync(FULL, (unsigned)w);
    o = ((unsigned long long)__reduce_xor_sync(FULL, (unsigned)(o >> 32)) << 32) | __reduce_xor_sync(FULL, (unsigned)o);
    if (lane == 0) I.rec = IslRec{o, w, n, nm, ncut, tlast, nx};
    __syncwarp();
    return ISL_OK;
}

__device__ __noinline__ int run_island_big(Fast &X, Isl<2> &I, int c, int size, bool level1, int lane) {
    return run_island<2>(X, I, c, size, level1, lane);
}

// Detection events of the row into svtx (those past cap dropped) and their
// counts before each word into S.wcum; returns their number.  Every thread of
// the team calls; ends with a barrier.
template <int NW>
__device__ __forceinline__ int load_events(int *wcum, const DGraph &g, const unsigned *row, int *svtx, int cap, Team<NW> &T) {
    int K = 0;
    const int nvec = g.words >> 2, n = g.n;
    const uint4 *rv = reinterpret_cast<const uint4 *>(row);
#pragma unroll 1
    for (int base = 0; base < nvec; base += T.NT) {
        const int i = base + T.tid();
        uint4 v = make_uint4(0, 0, 0, 0);
        if (i < nvec) v = __ldg(rv + i);
        unsigned wv[4] = {v.x, v.y, v.z, v.w};
        if (i * 128 + 128 > n) {   // drop padding bits beyond n
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int bit0 = (i * 4 + q) * 32;
                if (bit0 >= n) wv[q] = 0;
                else if (bit0 + 32 > n) wv[q] &= (1u << (n - bit0)) - 1u;
            }
        }
        const int c0 = __popc(wv[0]), c1 = c0 + __popc(wv[1]), c2 = c1 + __popc(wv[2]), c = c2 + __popc(wv[3]);
        int total;
        int pos = K + T.excl_scan(c, total);
        if (i < nvec) reinterpret_cast<int4 *>(wcum)[i] = make_int4(pos, pos + c0, pos + c1, pos + c2);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            unsigned bits = wv[q];
#pragma unroll 1
            while (bits) {
                const int b = __ffs(bits) - 1;
                bits &= bits - 1;
                if (pos < cap) svtx[pos] = (i * 4 + q) * 32 + b;
                pos++;
            }
        }
        K += total;
    }
    T.sync();
    return K;
}

// Per-event arrays of the shot and its pairs within b_1 (as near_pairs: from
// their lower ends, off the ball table; eight lanes per event and two entries
// per lane, since most lists have 12 entries).  Pairs are first noted with the
// other event's vertex and get its rank afterwards, every lane busy.  Returns
// false when an event's list is not complete or longer than level 1 takes.
// Every thread of the team calls; ends with a barrier.
template <int NW>
__device__ __forceinline__ bool fast_pairs(Fast &X, Team<NW> &T) {
    const DGraph &g = *X.g;
    const int lane = T.lane, K = X.K, sub = 2 * (lane & 7);
    int *const svtx = X.svtx(), *const bd = X.bd(), *const comp = X.comp(), *const px = X.px();
    unsigned *const cw = X.cw();
    const unsigned *const row = X.row;
    unsigned long long *const pr = X.pr;
    const int pcap = X.pcap;
    const int2 *const ball = g.ball;
    const int most = g.hop2 ? INT_MAX : LB_CAP - 1;
    const unsigned lt = (1u << lane) - 1u;
    bool odd = false;
    int np = 0;
#pragma unroll 1
    for (int base = T.warp() * WS; base < K; base += T.NT) {
        const int s = base + lane;
        int beg = 0, len = 0;
        if (s < K) {
            const int v = svtx[s];
            const int4 h = __ldg(g.bhdr + v);
            const unsigned long long vb = __ldg(g.vbnd + v);
            bd[s] = vb == EMPTY64 ? INT_MAX : (int)(vb >> 32);
            comp[s] = s;
            cw[s] = 0;
            px[s] = -1;
            odd |= h.z < 0 || h.z > most;
            beg = h.x;
            len = h.z < 0 ? 0 : h.y;
        }
        const int longest = __reduce_max_sync(FULL, len);
#pragma unroll 1
        for (int e0 = lane >> 3; __any_sync(FULL, e0 < WS && base + e0 < K); e0 += 4) {
            const unsigned eb = (unsigned)__shfl_sync(FULL, beg, e0);
            const int el = __shfl_sync(FULL, len, e0);
#pragma unroll 1
            for (int k = sub; __any_sync(FULL, k - sub < longest); k += 16) {
                bool h0 = false, h1 = false;
                int4 e = make_int4(0, 0, 0, 0);
                if (k < el) {
                    e = __ldg(reinterpret_cast<const int4 *>(ball + eb + k));   // lists start on 128-byte lines
                    h0 = (__ldg(row + (e.x >> 5)) >> (e.x & 31)) & 1u;
                    h1 = k + 1 < el && ((__ldg(row + (e.z >> 5)) >> (e.z & 31)) & 1u);
                }
                const unsigned m0 = __ballot_sync(FULL, h0), m1 = __ballot_sync(FULL, h1);
                if (!(m0 | m1)) continue;
                const int c0 = __popc(m0), c = c0 + __popc(m1);
                int b;
                if constexpr (NW == 1) {
                    b = np;
                    np += c;
                } else {
                    b = 0;
                    if (lane == 0) b = atomicAdd(&X.cnt[F_NP], c);
                    b = __shfl_sync(FULL, b, 0);
                }
                const unsigned long long self = (unsigned long long)(unsigned)(base + e0) << 52;
                const int j0 = b + __popc(m0 & lt), j1 = b + c0 + __popc(m1 & lt);
                if (h0 && j0 < pcap) pr[j0] = self | ((unsigned long long)(unsigned)e.x << 26) | (unsigned)e.y;
                if (h1 && j1 < pcap) pr[j1] = self | ((unsigned long long)(unsigned)e.z << 26) | (unsigned)e.w;
            }
        }
    }
    if constexpr (NW == 1)
        if (lane == 0) X.cnt[F_NP] = np;
    odd = T.any(odd);
    if constexpr (NW == 1) T.sync();
    const int n = min(X.cnt[F_NP], pcap);
#pragma unroll 1
    for (int i = T.tid(); i < n; i += T.NT) {
        const unsigned long long p = pr[i];
        pr[i] = pk_pair((int)(p >> 52), X.rank((int)(p >> 26) & 0x3ffffff), (int)p & 0x3ffffff);
    }
    T.sync();
    return !odd;
}

// Components of the events by min-label propagation with shortcuts over the
// pairs within b_1, [0, np0), and those marked MET in [np0, np1); labels start
// as they are.  Every thread of the team calls; ends with a barrier.
template <int NW>
__device__ __forceinline__ void fast_components(Fast &X, int np1, Team<NW> &T) {
    int *const compw = X.comp();
    volatile int *const comp = compw;
    const unsigned long long *const pr = X.pr;
    const int np0 = X.np0, K = X.K;
    // after an earlier join the pairs that joined events may be gone, and their
    // labels alone hold them together: those have to settle too
    const bool joined = X.late;
    bool again = false;
#pragma unroll 1
    for (int round = 0; round <= 2 * K; round++) {
        bool changed = again;
        again = false;
#pragma unroll 1
        for (int i = T.tid(); i < np1; i += T.NT) {
            const unsigned long long p = pr[i];
            if (i >= np0 && !(p & MET)) continue;
            const int a = pr_lo(p), b = pr_hi(p), la = comp[a], lb = comp[b];
            if (la != lb) {
                const int m = min(la, lb), h = max(la, lb);
                atomicMin(&compw[a], m);
                atomicMin(&compw[b], m);
                atomicMin(&compw[h], m);
                changed = true;
            }
        }
        T.sync();
        if (!T.any(changed)) break;
#pragma unroll 1
        for (int s = T.tid(); s < K; s += T.NT) {
            const int r = comp[s], rr = comp[r];
            if (rr < r) { comp[s] = rr; again = joined; }
        }
        T.sync();
    }
    T.sync();
}

// Level 1 of the shot: sizes, contacts and pairs within d_1 of the components,
// then what has a closed form (its weight and observable added to w and o):
// level-1 clusters of one or two events, and with `quick` every cluster or
// island in which each event either meets the event nearest to it, which
// has no nearer one itself (at half their distance), or the boundary first, and
// no other pair can touch before both its events have stopped.  Those are 60 %
// of the islands (two or three pairs near each other).  A pair that could be
// tight at the very time its events stop leaves the island open: the order of
// simultaneous events decides there.  Without `quick` (diagnostics are wanted)
// islands still take the closed form, level-1 clusters of more events run.
// The other clusters (from the front of X.list) and the islands (from its back)
// are listed by their lowest event.  Per-thread: t1 the last stopping time, ncl
// the clusters, nres their events.  Every thread of the team calls; ends with a
// barrier.
struct Level1 {
    long long w, wr;   // wr, ro: of clusters that nothing reopens
    unsigned long long o, ro;
    int t1, ncl, nres;
};
__device__ __forceinline__ void add_closed(Fast &X, int s, int partner, int d, long long &w, unsigned long long &o) {
    if (partner < 0) {
        const int bd = X.bd()[s];
        w += bd;
        o ^= __ldg(X.g->vobs + X.svtx()[s]);
        if (X.paths) put_path(X, s, -1, bd);
    } else {
        w += d / 2;
        if (X.paths && s < partner) put_path(X, s, partner, d);
    }
}
template <int NW>
__device__ __forceinline__ void fast_level1(Fast &X, Level1 &out, bool quick, Team<NW> &T) {
    const DGraph &g = *X.g;
    const int K = X.K, np0 = X.np0, b1 = g.b1, d1 = g.d1, band = X.band;
    const int *const comp = X.comp(), *const bdv = X.bd();
    int *const px = X.px(), *const stv = X.st();
    unsigned *const cwv = X.cw();
    const unsigned long long *const pr = X.pr;
    int *const list = X.list;
    const bool pack = b1 < (1 << 19);   // distances fit beside the event
#pragma unroll 1
    for (int s = T.tid(); s < K; s += T.NT) {
        const int r = comp[s];
        atomicAdd(&cwv[r], 1u);
        if (2LL * bdv[s] <= (long long)b1) atomicOr(&cwv[r], CW_SIDE);
    }
#pragma unroll 1
    for (int i = T.tid(); i < np0; i += T.NT) {
        const unsigned long long p = pr[i];
        const int a = pr_lo(p), b = pr_hi(p), d = pr_val(p);
        if (d <= d1) atomicAdd(&cwv[comp[a]], 1u << 12);
        atomicMin(reinterpret_cast<unsigned *>(px) + a, (unsigned)d << 12 | (unsigned)b);
        atomicMin(reinterpret_cast<unsigned *>(px) + b, (unsigned)d << 12 | (unsigned)a);
    }
    T.sync();
    // when each event would stop (st: 2 x time, + 1 at the boundary)
#pragma unroll 1
    for (int s = T.tid(); s < K; s += T.NT) {
        const unsigned near = (unsigned)px[s];
        const int bd = bdv[s], d = near == ~0u ? INT_MAX : (int)(near >> 12);
        bool ok = pack;
        int t = d >> 1;
        if (bd < t) {
            t = bd;
            stv[s] = 2 * min(t, 1 << 29) + 1;
        } else {
            const unsigned back = near == ~0u ? 0u : (unsigned)px[near & 4095u];
            ok &= near != ~0u && (back & 4095u) == (unsigned)s && bdv[near & 4095u] >= t;
            stv[s] = 2 * min(t, 1 << 29);
        }
        if (!ok || t > band) atomicOr(&cwv[comp[s]], CW_OPEN);
    }
    T.sync();
#pragma unroll 1
    for (int i = T.tid(); i < np0; i += T.NT) {
        const unsigned long long p = pr[i];
        const int a = pr_lo(p), b = pr_hi(p), d = pr_val(p), sa = stv[a], sb = stv[b];
        const bool matched = (px[a] & 4095) == b && !(sa & 1) && (px[b] & 4095) == a;
        if (!matched && d <= (sa >> 1) + (sb >> 1)) atomicOr(&cwv[comp[a]], CW_OPEN);
    }
    T.sync();
    Level1 L{0, 0, 0, 0, 0, 0, 0};
    const bool whole = quick && !X.paths;   // clusters of more events too
#pragma unroll 1
    for (int s = T.tid(); s < K; s += T.NT) {
        const int r = comp[s];
        const unsigned cw = cwv[r];
        const int size = (int)(cw & 4095u), prs = (int)(cw >> 12) & 0x3ffff;
        const bool ok = prs == size * (size - 1) / 2 && ((cw & CW_SIDE) || size % 2 == 0);
        const int near = (int)((unsigned)px[s] >> 12), other = px[s] & 4095;
        // a cluster of one or two events: one boundary event, or one collision
        // when no boundary is nearer
        const bool small = ok && pack && (size == 1 || (size == 2 && near / 2 <= bdv[s] && near / 2 <= bdv[other]));
        if (small || (!(cw & CW_OPEN) && (!ok || whole))) {
            const bool side = small ? size == 1 : (stv[s] & 1) != 0;
            const int rad = side ? bdv[s] : near / 2;
            stv[s] = small ? (side ? (int)MATE_BOUNDARY : other)
                           : (ok ? (int)ST_RUN : (side || s < other ? (int)ST_ONE : (int)ST_TWO));
            if (ok && !small) add_closed(X, s, side ? -1 : other, near, L.wr, L.ro);
            else add_closed(X, s, side ? -1 : other, near, L.w, L.o);
            px[s] = rad;
            if (ok) {
                L.t1 = max(L.t1, rad);
                L.nres++;
                if (s == r) L.ncl++;
            }
            continue;
        }
        stv[s] = ok ? (int)ST_RUN : (int)MATE_NONE;
        if (s == r) {
            if (ok) { list[atomicAdd(&X.cnt[F_N1], 1)] = s; L.nres += size; L.ncl++; }
            else list[K - 1 - atomicAdd(&X.cnt[F_N2], 1)] = s;
        }
    }
    T.sync();
    out = L;
}

// What islands met, after they have run: marks the pairs in [np0, np1) whose
// regions meet, joins their components and lists what has to run (in X.list,
// from its back) and all islands (in X.all); of the pairs those that what has to
// run would not record again are kept.  w, o: what is left of the closed forms.
// Returns 0 when nothing met, 1 when something was joined, 2 when the shot is
// outside the limits.  Every thread of the team calls; ends with a barrier.
template <int NW>
__device__ __noinline__ int fast_join(Fast &X, int np1, int n2, int round, Team<NW> T, long long &w,
                                      unsigned long long &o) {
    int *const list = X.list, *const all = X.all;
    const int K = X.K, np0 = X.np0, nstop = X.cnt[F_STOP];
    int *const comp = X.comp(), *const px = X.px(), *const st = X.st();
    unsigned *const cw = X.cw();
    int flags = 0;   // 1: something met, 2: outside the limits
#pragma unroll 1
    for (int i = np0 + T.tid(); i < np1; i += T.NT) {
        const unsigned long long p = X.pr[i];
        const int a = pr_lo(p), b = pr_hi(p);
        if (comp[a] != comp[b] && px[a] + px[b] >= pr_val(p)) {
            flags |= 1;
            if (st[a] == ST_RUN || st[b] == ST_RUN) flags |= 2;
            X.pr[i] = p | MET;
            cw[comp[a]] = 0;
            cw[comp[b]] = 0;
        }
    }
    T.sync();
    // an island that stopped but met nothing needs explored balls
#pragma unroll 1
    for (int i = nstop ? T.tid() : n2; i < n2; i += T.NT)
        if (cw[list[K - 1 - i]] == ISL_ALONE) flags |= 2;
    flags = T.template red32<2>(flags);
    if ((flags & 2) || ((flags & 1) && round >= 32)) {
        T.sync();
        return 2;
    }
    if (!(flags & 1)) {
        T.sync();
        return 0;
    }
    // run what was joined (with paths: everything, since their list starts over)
    T.sync();
    fast_components(X, np1, T);
#pragma unroll 1
    for (int s = T.tid(); s < K; s += T.NT) {
        cw[s] = 0;
        if (round == 0 && st[s] != MATE_NONE) X.recs[s].size = 0;   // not run so far
        if (st[s] == ST_ONE || st[s] == ST_TWO) st[s] = MATE_NONE;   // run from now on
    }
    if (T.tid() == 0) {
        X.cnt[F_N2] = 0; X.cnt[F_NALL] = 0; X.cnt[F_STOP] = 0;
        X.late = 1;
        // the path list keeps the pairs of the level-1 clusters run
        int k = 0;
#pragma unroll 1
        for (int i = X.path0; i < X.path1; i++, k++) { X.pa[k] = X.pa[i]; X.pb[k] = X.pb[i]; X.pd[k] = X.pd[i]; }
        X.path0 = 0;
        X.path1 = X.cnt[F_NPATH] = k;
    }
    T.sync();
#pragma unroll 1
    for (int s = T.tid(); s < K; s += T.NT) atomicAdd(&cw[comp[s]], 1u);
    T.sync();
    w = 0;
    o = 0;
    // what an event is part of: 0 a level-1 cluster on its own, 1 an island that
    // stands as it ran, 2 an island to run
    auto part = [&](int s) {
        const int c = comp[s], size = (int)cw[c];
        if ((st[s] == MATE_BOUNDARY && size == 1) || (st[s] >= 0 && size == 2) || st[s] == ST_RUN) return 0;
        return X.paths || X.recs[c].size != size ? 2 : 1;
    };
#pragma unroll 1
    for (int s = T.tid(); s < K; s += T.NT) {
        const int p = part(s);
        X.was[s] = p == 2 ? -1 : px[s];
        if (p == 0) {
            if (st[s] != ST_RUN) add_closed(X, s, st[s], 2 * px[s], w, o);   // (MATE_BOUNDARY is negative)
        } else if (s == comp[s]) {
            all[atomicAdd(&X.cnt[F_NALL], 1)] = s;
            if (p == 2) list[K - 1 - atomicAdd(&X.cnt[F_N2], 1)] = s;
        }
    }
    // pairs recorded by what stands stay: the region that recorded one does not
    // come back to it, and the other, the smaller of the two, may not reach as far.
    // What runs records its own again.
    if (T.warp() == 0) {
        int np = np0;
#pragma unroll 1
        for (int base = np0; base < np1; base += WS) {
            unsigned long long p = 0;
            bool keep = false;
            if (base + T.lane < np1) {
                p = X.pr[base + T.lane];
                keep = part(pr_lo(p)) != 2 || part(pr_hi(p)) != 2;
            }
            const unsigned m = __ballot_sync(FULL, keep);   // (read before any is moved)
            if (keep) X.pr[np + __popc(m & ((1u << T.lane) - 1u))] = p;
            np += __popc(m);
            __syncwarp();
        }
        if (T.lane == 0) X.cnt[F_NP] = np;
    }
    T.sync();
    return 1;
}

// Whether every two regions past the cap of Fast::reach knew each other when they
// met, or stayed apart: they are at most two caps apart (where they meet, the
// larger one has half the distance, and its reach holds the rest; farther ones may
// be recorded too late), or their distance (in the ball table of one of them, or
// beyond it) exceeds the sum of their radii.  One warp.
__device__ __noinline__ bool wide_apart(Fast &X, int lane) {
    const DGraph &g = *X.g;
    const int K = X.K, cap = X.cap, brad = g.brad;
    const int *const px = X.px(), *const svtx = X.svtx();
    int mine = -1, n = 0;   // lane j: the j-th wide event
#pragma unroll 1
    for (int base = 0; base < K; base += WS) {
        const bool wide = base + lane < K && px[base + lane] > cap;
#pragma unroll 1
        for (unsigned m = __ballot_sync(FULL, wide); m; m &= m - 1, n++)
            if (lane == n) mine = base + __ffs(m) - 1;
    }
    if (n > WS) return false;
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i + 1 < n; i++) {
        const int a = __shfl_sync(FULL, mine, i), ra = px[a];
        const int4 h = __ldg(g.bhdr + svtx[a]);
        const int v = lane > i && lane < n ? svtx[mine] : -1, rb = v < 0 ? 0 : px[mine];
        if (h.w < 0 || __any_sync(FULL, v >= 0 && ra + rb > brad)) return false;
#pragma unroll 1
        for (int k = 0; k < h.z + h.w; k++) {   // one entry for all lanes
            const int2 e = __ldg(g.ball + (unsigned)h.x + k);
            if (e.x == v && e.y <= ra + rb && e.y > 2 * cap) ok = false;
        }
    }
    return !__any_sync(FULL, !ok);
}

constexpr int USE_GENERAL = -3;   // the shot is outside the fast path's limits
constexpr int HAS_ISLANDS = -4;   // begun: its islands are listed
constexpr int NOT_FAST = -5;      // the fast path takes no shot of this graph and mode

// What the warps of a block that decode a shot each share: the islands of all
// their shots, taken by whichever warp is free.
struct Pool {
    int n[32], next;
};

// The fields of a team's Fast that stay the same from shot to shot.  One thread.
template <int NW>
__device__ __forceinline__ void fast_small(FastShared<NW> &M) {
    M.f.ev = M.ev;
    M.f.pr = M.pr;
    M.f.stride = M.KS;
    M.f.pcap = M.PS;
}
template <int NW>
__device__ __forceinline__ void fast_setup(const Slab &S, const SlabCaps &caps, FastShared<NW> &M) {
    Fast &X = M.f;
    X.wcum = S.wcum;
    X.recs = reinterpret_cast<IslRec *>(S.wl0);
    X.spare = reinterpret_cast<char *>(X.recs + caps.kc);
    X.nspare = caps.wc * 8 - caps.kc * (int)sizeof(IslRec);
    X.nlist = caps.kc;
    X.list = S.xsrc; X.all = S.xcnt;
    X.aged_t = S.xR; X.aged_c = S.sbeg; X.aged_n = S.scnt;
    X.pa = S.tmpa; X.pb = S.tmpb; X.pd = S.cst2;
    X.was = S.xcur;
    fast_small(M);
}

// A shot between the phases of the fast path (per thread).
struct FastShot {
    Level1 L;
    IslRec lev;   // level-1 clusters run (lane 0 of each warp)
    int lmax, K, np0, n1, n2;
};

// First phase: events, pairs, level 1.  Returns QEC_SHOT_OK for a shot without
// events (everything written), HAS_ISLANDS, USE_GENERAL or NOT_FAST.
template <bool WIN, int NW>
__device__ __forceinline__ int fast_begin(const BatchArgs &A, const Slab &S, const DGraph &g, const unsigned *row,
                                          Team<NW> &T, FastShared<NW> &M, FastShot &Q, int *dg) {
    if (!fast_path_takes(g, A.mode, A.band_factor)) return NOT_FAST;
    if (g.words > A.caps.wcap) return USE_GENERAL;
    const int band = max(g.wmax, 1) * max(A.band_factor, 1);
    Fast &X = M.f;
    bool small = true;
    int K = 0;
#pragma unroll 1
    for (;;) {
        if (T.tid() == 0) {
            X.g = &g;
            X.row = row;
            X.L = max(g.wmax, (g.b1 + 1) / 2) + 1;
            X.band = band;
            X.cap = max(2 * g.wmax + 1, (g.b1 + 1) >> 1);
            X.paths = WIN || g.internal_obs;
            X.tcut = 0;
            X.late = X.path0 = X.path1 = 0;
            if (!small) {
                X.ev = reinterpret_cast<int *>(S.wl1);   // 48 K words of 8 bytes
                X.pr = S.tl;
                X.stride = A.caps.kc;
                X.pcap = A.caps.ec;
            } else if (X.stride != M.KS) {
                fast_small(M);
            }
        }
        if (T.tid() < F_TOTAL) X.cnt[T.tid()] = 0;
        T.sync();
        K = load_events(S.wcum, g, row, X.ev, X.stride, T);
        if (K == 0) {
            if (dg && T.tid() < QEC_DIAG_FIELDS) dg[T.tid()] = 0;   // no detection event: E_ideal = 0
            if constexpr (WIN)
                for (int w = T.tid(); w < g.words; w += T.NT) A.carry[(row - A.syn) + w] = 0u;
            return QEC_SHOT_OK;
        }
        if (K > A.caps.kc || K > 4000) return USE_GENERAL;
        if (K <= X.stride) {
            if (T.tid() == 0) X.K = K;
            T.sync();
            if (!fast_pairs(X, T)) return USE_GENERAL;
            Q.np0 = X.cnt[F_NP];
            if (Q.np0 <= X.pcap && Q.np0 < (1 << 18)) break;
            if (!small) return USE_GENERAL;
        }
        T.sync();
        small = false;
    }
    if (T.tid() == 0) X.np0 = Q.np0;
    T.sync();
    fast_components(X, Q.np0, T);
    fast_level1(X, Q.L, !dg, T);
    Q.K = K;
    Q.n1 = X.cnt[F_N1];
    Q.n2 = X.cnt[F_N2];
    Q.lev = IslRec{0, 0, 0, 0, 0, 0, 0};
    Q.lmax = 0;
    if (WIN || g.internal_obs) {
        if (T.tid() == 0) X.path0 = X.path1 = X.cnt[F_NPATH];
        T.sync();
    }
    if (dg) {
        Q.L.t1 = T.maxi(Q.L.t1);
        T.sync();
        if (T.tid() == 0) X.tcut = Q.L.t1;
        T.sync();
    }
    return HAS_ISLANDS;
}

// Second phase: the islands, and what remains of level 1 before them.  POOL: the
// warps of the block have a shot each and share their islands (phases of the
// warps in step keep the instruction cache warm, and no warp waits for the
// largest shot alone); `busy`: this warp has one.  Then the shot's own pairs
// recorded by extensions, which join different islands or clusters when the
// radii reach their distance.  Returns QEC_SHOT_OK or USE_GENERAL.
template <bool WIN, int NW, bool POOL>
__device__ __forceinline__ int fast_islands(Team<NW> &T, FastShared<NW> &M, Pool &P, FastShot &Q, bool busy, int *dg) {
    Isl<1> &I = M.isl[T.warp()];
    const int lane = T.lane, K = Q.K;
    // stage 0: level-1 clusters; 1: islands; 2: islands joined since
    int stage = busy && Q.n1 > 0 ? 0 : 1, round = 0, i = T.warp(), status = QEC_SHOT_OK, pooled = 0;
    int incl = 0;   // islands of the block's shots up to this lane's
#pragma unroll 1
    for (;;) {
        // the next cluster or island
        int c = -1;
        Fast *X = &M.f;
        if (stage == 1 && POOL) {
            if (!pooled) {
                if (lane == 0) P.n[threadIdx.x >> 5] = busy && status == QEC_SHOT_OK ? Q.n2 : 0;
                __syncthreads();
                incl = lane < (int)(blockDim.x >> 5) ? P.n[lane] : 0;
#pragma unroll
                for (int o = 1; o < WS; o <<= 1) {
                    const int v = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += v;
                }
                pooled = __shfl_sync(FULL, incl, WS - 1) + 1;
            }
            int k = 0;
            if (lane == 0) k = atomicAdd(&P.next, 1);
            k = __shfl_sync(FULL, k, 0);
            if (k < pooled - 1) {
                const int w = __popc(__ballot_sync(FULL, incl <= k));   // whose island it is
                const int before = __shfl_sync(FULL, incl, max(w - 1, 0));
                X = &(&M - (threadIdx.x >> 5) + w)->f;
                c = X->list[X->K - 1 - (k - (w ? before : 0))];
            }
        } else if (i < (stage ? Q.n2 : Q.n1) && status == QEC_SHOT_OK) {
            c = M.f.list[stage ? K - 1 - i : i];
            i += NW;
        }
        if (c >= 0) {
            const int size = (int)(X->cw()[c] & 4095u);
            int r = run_island<1>(*X, I, c, size, stage == 0, lane);
            const IslRec *rec = &I.rec;
            if (r == ISL_BIG) {
                r = ISL_FAIL;
                // spare list room of this team's slab, which holds one per warp
                // in all but the smallest slabs of block-wide teams
                Isl<2> *const big = reinterpret_cast<Isl<2> *>(M.f.spare) + T.warp();
                if (reinterpret_cast<char *>(big + 1) <= M.f.spare + M.f.nspare) {
                    r = run_island_big(*X, *big, c, size, stage == 0, lane);
                    if (r == ISL_BIG) r = ISL_FAIL;
                    rec = &big->rec;
                }
            }
            if (lane == 0) {
                if (r == ISL_OK && stage == 0) {
                    Q.lev.w += rec->w; Q.lev.o ^= rec->o; Q.lev.nm += rec->nm; Q.lev.nx += rec->nx;
                    Q.lev.tlast = max(Q.lev.tlast, rec->tlast);
                    Q.lmax = max(Q.lmax, rec->nm);
                } else if (r == ISL_OK) {
                    X->recs[c] = *rec;
                } else {
                    if (r == ISL_FAIL || stage == 0) X->cnt[F_FAIL] = 1;
                    X->recs[c].size = -1;
                }
            }
            __syncwarp();
            continue;
        }
        // the end of a stage
        if (stage == 1 && POOL) {
            __syncthreads();
            if (threadIdx.x == 0) P.next = 0;
            if (!busy) return QEC_SHOT_OK;
        }
        T.sync();
        i = T.warp();
        if (M.f.cnt[F_FAIL] || M.f.cnt[F_AGED] > M.f.nlist) status = USE_GENERAL;
        if (stage == 0) {
            if (T.tid() == 0) M.f.path1 = M.f.cnt[F_NPATH];
            T.sync();
            stage = 1;
            if (dg) {
                Q.L.t1 = max(Q.L.t1, T.maxi(Q.lev.tlast));
                T.sync();
                if (T.tid() == 0) M.f.tcut = Q.L.t1;
                T.sync();
            }
            continue;
        }
        if (status != QEC_SHOT_OK) return status;
        const int np1 = M.f.cnt[F_NP];
        if (np1 > M.f.pcap) return USE_GENERAL;
        auto stands = [&]() -> int {
            if (!M.f.cnt[F_WIDE]) return QEC_SHOT_OK;
            bool ok = true;
            if (T.warp() == 0) ok = wide_apart(M.f, lane);
            return T.any(!ok) ? USE_GENERAL : QEC_SHOT_OK;
        };
        if (np1 == Q.np0) return M.f.cnt[F_STOP] ? USE_GENERAL : stands();   // (stopped, having met nothing)
        const int j = fast_join(M.f, np1, Q.n2, round++, T, Q.L.w, Q.L.o);
        if (j != 1) return j == 2 ? USE_GENERAL : stands();
        Q.n2 = M.f.cnt[F_N2];
        stage = 2;
    }
}

// Last phase: the shot's result and diagnostics.
template <bool WIN, int NW>
__device__ __forceinline__ int fast_end(const BatchArgs &A, const Slab &S, const DGraph &g, const unsigned *row,
                                        Team<NW> &T, FastShared<NW> &M, FastShot &Q, long long &w_out,
                                        unsigned long long &o_out, int *dg) {
    Fast &X = M.f;
    const int K = Q.K, n1 = Q.n1;
    // the islands together
    const int joined = X.cnt[F_NALL], nall = joined ? joined : X.cnt[F_N2];
    const int *const all = joined ? X.all : X.list + (K - nall);
    int ntop = 0, ncut = 0, tlast = 0, tnx = 0;
#pragma unroll 1
    for (int i = T.tid(); i < nall; i += T.NT) {
        const IslRec r = X.recs[all[i]];
        Q.L.w += r.w;
        Q.L.o ^= r.o;
        ntop += r.nm; ncut += r.ncut; tlast = max(tlast, r.tlast); tnx += r.nx;
    }
    int closed = 0;   // islands in closed form: their events
    if (dg) {
#pragma unroll 1
        for (int s = T.tid(); s < K; s += T.NT) {
            const int st = X.st()[s], t = X.px()[s];
            if (st != ST_ONE && st != ST_TWO) continue;
            if (st == ST_ONE) { ntop++; ncut += t <= X.tcut; }
            tlast = max(tlast, t);
            closed = 1;
        }
    }
    const int naged = X.cnt[F_AGED];
    if (A.max_events < 256LL * K + 4096) {
        // a budget set lower: unless the events are surely within it, the run over
        // everything counts exactly.  Each of its runs adds one step that finds no
        // event; a closed form of n > 1 events stands for at most n events, and as
        // a level-1 cluster for an extension and that step besides.
        if ((long long)T.add(Q.lev.nm + Q.lev.nx + ntop + tnx) + naged + n1 + 2 * K + 2 > A.max_events) return USE_GENERAL;
    }
    w_out = T.sum64(Q.L.w + Q.L.wr + Q.lev.w) / 2;
    o_out = T.xor64(Q.L.o ^ Q.L.ro ^ Q.lev.o);
    if (dg) {
        // parallel event count over level 1 and the top level (Methods,
        // "Numerical evaluation").  Bands: one per time at which regions of the
        // top level came of age (entries of islands joined since don't count)
        int aged = 0;
#pragma unroll 1
        for (int i = T.tid(); i < naged; i += T.NT) {
            auto live = [&](int k) { const int c = X.aged_c[k]; return X.comp()[c] == c && X.recs[c].size == X.aged_n[k]; };
            const int x = X.aged_t[i];
            int first = live(i);
#pragma unroll 1
            for (int j = 0; j < i && first; j++) first = !(X.aged_t[j] == x && live(j));
            aged += first;
        }
        aged = T.add(aged);
        closed = T.any(closed != 0);
        const int ncl = T.add(Q.L.ncl), nres = T.add(Q.L.nres);
        const int lnm = T.add(Q.lev.nm), lnx = T.add(Q.lev.nx), lmax = T.maxi(Q.lmax);
        ntop = T.add(ntop); ncut = T.add(ncut); tnx = T.add(tnx); tlast = T.maxi(tlast);
        // closed forms have one event each
        const int e1 = max(lmax, ncl > n1 ? 1 : 0), ntot = (ncl - n1) + lnm;
        if (T.tid() == 0) {
            dg[QEC_DIAG_E_IDEAL] = ntop > 0 ? max(e1, ncut) + ntop - ncut : e1;
            dg[QEC_DIAG_T_IDEAL] = ntop > 0 ? max(Q.L.t1, tlast) : Q.L.t1;
            dg[QEC_DIAG_EVENTS] = ntot + ntop;
            dg[QEC_DIAG_L1_CLUSTERS] = ncl;
            dg[QEC_DIAG_L1_DEFECTS] = nres;
            dg[QEC_DIAG_TOP_EVENTS] = ntop;
            dg[QEC_DIAG_BANDS] = lnx + tnx + aged + (nall > 0 || closed ? 1 : 0);
            dg[QEC_DIAG_DEFECTS] = K;
        }
    }
    if (WIN || g.internal_obs) {
        Shot C;
        C.g = g;
        C.row = row;
        C.K = K;
        C.L = X.L;
        C.band = X.band;
        C.real = 0;
        C.paths = 0;
        const unsigned long long po = walk_paths<WIN>(A, S, C, T, X.ev, X.cnt[F_NPATH], 1,
                                                      WIN ? A.carry + (row - A.syn) : nullptr);
        const int err = T.bcast(ldr(&S.ctr[C_ERR]));
        if (C.paths) release_tables(S, C, T, err != 0);
        if (err) return USE_GENERAL;
        o_out = WIN ? po : o_out ^ po;
    }
    return QEC_SHOT_OK;
}

// Detection events of a syndrome row (padding bits beyond n ignored).  One warp.
__device__ int count_defects(const DGraph &g, const unsigned *row, int lane) {
    int c = 0;
    for (int w = lane; w < g.words; w += WS) {
        unsigned v = __ldg(row + w);
        const int bit0 = w * 32;
        if (bit0 >= g.n) v = 0;
        else if (bit0 + 32 > g.n) v &= (1u << (g.n - bit0)) - 1u;
        c += __popc(v);
    }
    return (int)__reduce_add_sync(FULL, (unsigned)c);
}

// The general path: attempts with larger and larger tables.
template <bool WIN, int NW>
__device__ __noinline__ int decode_general(const BatchArgs &A, const Slab &S, const DGraph &g, const unsigned *row,
                                           Team<NW> T, unsigned long long deadline, long long &w,
                                           unsigned long long &o, int *dg) {
    int status = -1, mode = A.mode;
    for (unsigned scale = 1; scale <= 64 && status == -1;) {
        status = decode_attempt<WIN, NW>(A, mode, S, g, row, T, scale, deadline, w, o, dg);
        if (status == LEVEL1_OVERLAP) {
            status = -1;
            mode = QEC_MODE_GLOBAL;
        } else {
            scale *= 4;
        }
    }
    return status;
}

// One shot's place in the batch.
struct ShotRef {
    const DGraph *g;
    const unsigned *row;
    long long shot, off;
    int *dg;
};
__device__ __forceinline__ ShotRef shot_ref(const BatchArgs &A, long long shot) {
    int gi = A.graph_of_shot ? A.graph_of_shot[shot] : 0;
    if (gi < 0 || gi >= A.num_graphs) gi = 0;
    ShotRef r;
    r.g = &A.g[gi];
    r.shot = shot;
    r.off = A.syn_off ? A.syn_off[shot] : shot * (long long)r.g->words;
    r.row = A.syn + r.off;
    r.dg = A.diag_out ? A.diag_out + shot * QEC_DIAG_FIELDS : nullptr;
    return r;
}

// Write a shot's outputs (status < 0: it did not fit its slab).
template <bool WIN, int NW>
__device__ __forceinline__ void finish_shot(const BatchArgs &A, const ShotRef &r, Team<NW> &T, int status, long long w,
                                            unsigned long long o) {
    const bool retried = status < 0 && A.pass == 0 && A.single_shot < 0;   // goes to the overflow pass
    if (status < 0) {
        status = QEC_SHOT_CAPACITY;
        if (retried && T.tid() == 0) {
            const unsigned long long idx = atomicAdd(&A.queue[1], 1ull);
            A.overflow[idx] = (int)r.shot;
        }
        w = 0;
        o = 0;
    }
    if (r.dg && status != QEC_SHOT_OK && T.tid() < QEC_DIAG_FIELDS) r.dg[T.tid()] = 0;
    if constexpr (WIN) {
        // sliding window: nothing is committed by a failed shot
        if (status != QEC_SHOT_OK)
            for (int i = T.tid(); i < r.g->words; i += T.NT) A.carry[r.off + i] = 0u;
        if (T.tid() == 0) {
            if (status == QEC_SHOT_OK) A.cobs[r.shot] ^= o;
            else if (!retried) A.st_out[r.shot] = status;
        }
    } else if (T.tid() == 0) {
        A.w_out[r.shot] = w;
        A.obs_out[r.shot] = o;
        A.st_out[r.shot] = status;
        if (A.done && !retried) {
            // the results reach the host before the flag that publishes them
            __threadfence_system();
            asm volatile("st.release.sys.global.b32 [%0], %1;" :: "l"(A.done + r.shot), "r"(1) : "memory");
        }
    }
    T.sync();
}

// Decode one shot by a team.  POOL (NW = 1): every warp of the block calls at
// the same time, those without a shot with busy = false.
template <bool WIN, int NW, bool POOL>
__device__ __forceinline__ void decode_shot(const BatchArgs &A, const Slab &S, const ShotRef &r, bool busy, Team<NW> &T,
                                            FastShared<NW> &M, Pool &P, unsigned long long deadline) {
    if constexpr (NW > 1) {
        // a shot below the split threshold goes to the team's first warp
        // alone (a team's barriers cost more than its lanes save there)
        if (A.team_split > 1) {
            int K = 0;
            if (T.warp() == 0) K = count_defects(*r.g, r.row, T.lane);
            K = T.bcast(K);
            if (K < A.team_split) {
                if (T.warp() == 0) {
                    Team<1> T1;
                    T1.lane = T.lane;
                    FastShared<1> &M1 = reinterpret_cast<FastShared<1> &>(M);
                    if (T.lane == 0) fast_setup(S, A.caps, M1);
                    __syncwarp();
                    decode_shot<WIN, 1, false>(A, S, r, true, T1, M1, P, deadline);
                    if (T.lane == 0) fast_setup(S, A.caps, M);
                }
                T.sync();
                return;
            }
        }
    }
    long long w = 0;
    unsigned long long o = 0;
    FastShot Q;
    Q.n1 = Q.n2 = Q.K = 0;
    int status = QEC_SHOT_OK;
    if (busy) status = fast_begin<WIN, NW>(A, S, *r.g, r.row, T, M, Q, r.dg);
    if (POOL || status == HAS_ISLANDS) {
        const bool has = busy && status == HAS_ISLANDS;
        const int st = fast_islands<WIN, NW, POOL>(T, M, P, Q, has, r.dg);
        if (has) status = st == QEC_SHOT_OK ? fast_end<WIN, NW>(A, S, *r.g, r.row, T, M, Q, w, o, r.dg) : st;
    }
    if (!busy) return;
    if (status == USE_GENERAL && NW == 1 && A.defer && A.pass == 0) {
        status = -1;   // left to the blocks of the overflow pass
    } else if (status == USE_GENERAL || status == NOT_FAST) {
        T.sync();
        status = decode_general<WIN, NW>(A, S, *r.g, r.row, T, deadline, w, o, r.dg);
    }
    finish_shot<WIN, NW>(A, r, T, status, w, o);
}

// One team per warp (NW = 1, any block size that is a multiple of 32) or one
// team per block (NW > 1, blocks of exactly 32 NW threads).
template <bool WIN, int NW>
__global__ void __launch_bounds__(NW == 1 ? 32 * QEC_MAX_WARPS : 32 * NW, NW == 1 ? QEC_SM_WARPS / QEC_MAX_WARPS : (NW == 4 ? 4 : 1))
batch_kernel(const __grid_constant__ BatchArgs a) {
    extern __shared__ __align__(16) char dyn[];   // one FastShared per team
    __shared__ Pool pool;
    Team<NW> T;
    T.lane = threadIdx.x & 31;
    FastShared<NW> &M = reinterpret_cast<FastShared<NW> *>(dyn)[NW == 1 ? threadIdx.x >> 5 : 0];
    if constexpr (NW > 1) {
        __shared__ TeamShared tsh;
        T.sh = &tsh;
        T.tid_ = (int)threadIdx.x;
        T.warp_ = (int)(threadIdx.x >> 5);
        T.ph = 0;
    }
    const long long wid = NW == 1 ? (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) : (long long)blockIdx.x;
    Slab S;
    carve(a.slabs + wid * a.slab_bytes, a.caps, S);
    unsigned long long deadline = 0;
    if (a.watchdog_ns > 0) {
        unsigned long long t0 = T.tid() == 0 ? now_ns() : 0;
        deadline = T.bcast64(t0) + (unsigned long long)a.watchdog_ns;
    }
    if (NW == 1 && threadIdx.x == 0) pool.next = 0;
    if (T.tid() == 0) fast_setup(S, a.caps, M);
    __syncthreads();
    // a single shot is the work of the first team; otherwise team t starts with
    // item (its place in the block) x blocks + block, so that a small batch
    // spreads over the SMs, and goes on with whatever is next
    const bool one = a.single_shot >= 0;
    unsigned long long *counter = a.queue + (a.pass == 0 ? 0 : 2);
    const long long teams = NW == 1 ? (long long)gridDim.x * (blockDim.x >> 5) : (long long)gridDim.x;
    const long long limit = one ? 1 : (a.pass == 0 ? a.num_shots : (long long)min(a.queue[1], (unsigned long long)a.num_shots));
    long long item = NW == 1 ? (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x : (long long)blockIdx.x;
    for (long long it = 0; it < limit + 1; it++) {
        const bool busy = item < limit;
        if (NW == 1 ? !__syncthreads_or(busy) : !busy) break;
        ShotRef r{a.g, a.syn, 0, 0, nullptr};
        unsigned long long next = 0;
        if (busy) {
            r = shot_ref(a, one ? a.single_shot
                                : (a.pass == 0 ? (a.order ? (long long)a.order[item] : item) : (long long)a.overflow[item]));
            if (T.tid() == 0 && !one) next = atomicAdd(counter, 1ull);
        }
        decode_shot<WIN, NW, NW == 1>(a, S, r, busy, T, M, pool, deadline);
        item = busy && !one ? (long long)T.bcast64(next) + teams : limit;
    }
}

struct GraphOrder {
    int g[QEC_MAX_GRAPHS_PER_BATCH];
};

__global__ void graph_count_kernel(const int *gid, long long n, int ng, int *gcnt) {
    __shared__ int local[QEC_MAX_GRAPHS_PER_BATCH];
    for (int i = threadIdx.x; i < QEC_MAX_GRAPHS_PER_BATCH; i += blockDim.x) local[i] = 0;
    __syncthreads();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int g = gid[i];
        if (g < 0 || g >= ng) g = 0;
        atomicAdd(&local[g], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ng; i += blockDim.x)
        if (local[i]) atomicAdd(&gcnt[i], local[i]);
}

__global__ void graph_scan_kernel(int *gcnt, int ng, GraphOrder go) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int acc = 0;
    for (int k = 0; k < ng; k++) {
        const int g = go.g[k];
        gcnt[32 + g] = acc;
        acc += gcnt[g];
    }
}

__global__ void graph_scatter_kernel(const int *gid, long long n, int ng, int *gcnt, int *order) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int g = gid[i];
        if (g < 0 || g >= ng) g = 0;
        const int pos = atomicAdd(&gcnt[32 + g], 1);
        order[pos] = (int)i;
    }
}

}  // namespace

cudaError_t launch_graph_sort(const int *graph_of_shot, long long n, int ng, const int *gorder, int *gcnt,
                              int *order, cudaStream_t s) {
    GraphOrder go;
    for (int k = 0; k < QEC_MAX_GRAPHS_PER_BATCH; k++) go.g[k] = k < ng ? gorder[k] : 0;
    cudaError_t e = cudaMemsetAsync(gcnt, 0, 64 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 1024);
    graph_count_kernel<<<blocks, 256, 0, s>>>(graph_of_shot, n, ng, gcnt);
    graph_scan_kernel<<<1, 32, 0, s>>>(gcnt, ng, go);
    graph_scatter_kernel<<<blocks, 256, 0, s>>>(graph_of_shot, n, ng, gcnt, order);
    return cudaGetLastError();
}

long long slab_bytes_for(const SlabCaps &c) {
    Slab S;
    long long b = carve(reinterpret_cast<char *>(0), c, S);
    return (b + 255) & ~255LL;
}

SlabCaps caps_for_kcap(int kcap, int table_factor) {
    auto p2 = [](long long x) { long long r = 1; while (r < x) r <<= 1; return (int)r; };
    const long long f = table_factor < 1 ? 1 : table_factor;
    SlabCaps c;
    c.kc = kcap;
    c.hc = p2(64LL * f * kcap < 1024 ? 1024 : 64LL * f * kcap);
    c.ec = (int)(48 * f * kcap + 64);
    c.wc = (int)(48 * f * kcap + 64);
    c.phc = p2(16LL * f * f * kcap < 256 ? 256 : 16LL * f * f * kcap);   // dense shots: pairs grow ~ f^2
    c.nc = 2 * kcap + 16;
    c.wcap = QEC_STREAM_MAX_WORDS;   // rows up to 73,728 detectors; callers raise it for larger graphs
    c.cc = 24 * kcap + 64;
    return c;
}

namespace {

// Shared memory of a block, and the attribute that a kernel needs above 48 KB
// (set once per device, for the largest block).
template <int NW>
constexpr int smem_of(int block) { return (int)sizeof(FastShared<NW>) * (NW == 1 ? block / 32 : 1); }

template <bool WIN, int NW>
cudaError_t allow_smem() {
    static std::atomic<unsigned long long> ready{0};   // bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (ready.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(batch_kernel<WIN, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_of<NW>(32 * QEC_MAX_WARPS));
    if (e == cudaSuccess) ready.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

template <bool WIN, int NW>
cudaError_t launch_as(const BatchArgs &a, int grid, int block, cudaStream_t s) {
    const cudaError_t e = allow_smem<WIN, NW>();
    if (e != cudaSuccess) return e;
    batch_kernel<WIN, NW><<<grid, NW == 1 ? block : 32 * NW, smem_of<NW>(block), s>>>(a);
    return cudaGetLastError();
}

template <int NW>
int blocks_per_sm(int block) {
    int nb = 0;
    cudaError_t e = allow_smem<false, NW>();
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_kernel<false, NW>, block, (size_t)smem_of<NW>(block));
    return e == cudaSuccess && nb > 0 ? nb : 1;
}

}  // namespace

cudaError_t launch_batch(const BatchArgs &a, int grid, int block, cudaStream_t s, int team) {
    if (a.carry) return team == TEAM_BIG ? launch_as<true, TEAM_BIG>(a, grid, block, s) : launch_as<true, 1>(a, grid, block, s);
    if (team == TEAM_BIG) return launch_as<false, TEAM_BIG>(a, grid, block, s);
    if (team == TEAM_MID) return launch_as<false, TEAM_MID>(a, grid, block, s);
    return launch_as<false, 1>(a, grid, block, s);
}

int max_block_threads() {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, batch_kernel<false, 1>) != cudaSuccess) return 32;
    return fa.maxThreadsPerBlock > 0 ? fa.maxThreadsPerBlock : 32;
}

int occupancy_blocks(int block_threads) { return blocks_per_sm<1>(block_threads); }

int team_occupancy_blocks(int team) { return team == TEAM_BIG ? blocks_per_sm<TEAM_BIG>(32 * TEAM_BIG) : blocks_per_sm<TEAM_MID>(32 * TEAM_MID); }

namespace {

// 32 bits of `row` (of `words` words) starting at bit b (bits past the row are 0).
__device__ __forceinline__ unsigned bits32(const unsigned *row, long long words, long long b) {
    const long long w = b >> 5;
    const int sh = (int)(b & 31);
    const unsigned lo = w < words ? row[w] : 0u;
    const unsigned hi = (sh && w + 1 < words) ? row[w + 1] : 0u;
    return sh ? (lo >> sh) | (hi << (32 - sh)) : lo;
}

__device__ __forceinline__ unsigned low_mask(long long n) {   // bits [0, n) of a word, n clamped to [0, 32]
    return n <= 0 ? 0u : (n >= 32 ? ~0u : (1u << n) - 1u);
}

// One thread per (row, window word).
__global__ void window_assemble_kernel(const unsigned *src, long long src_words, long long bit_begin, int nbits,
                                       const unsigned *carry, long long carry_words, long long carry_begin,
                                       int carry_bits, unsigned *dst, long long dst_words, long long num_rows) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= num_rows * dst_words) return;
    const long long r = i / dst_words, w = i - r * dst_words;
    const long long b = w * 32;
    unsigned v = bits32(src + r * src_words, src_words, bit_begin + b) & low_mask(nbits - b);
    if (carry) v ^= bits32(carry + r * carry_words, carry_words, carry_begin + b) & low_mask(carry_bits - b);
    dst[i] = v;
}

}  // namespace

cudaError_t launch_window_assemble(const unsigned *src, long long src_words, long long bit_begin, int nbits,
                                   const unsigned *carry, long long carry_words, long long carry_begin,
                                   int carry_bits, unsigned *dst, long long dst_words, long long num_rows,
                                   cudaStream_t s) {
    const long long n = num_rows * dst_words;
    if (n <= 0) return cudaSuccess;
    const int block = 256;
    const long long grid = (n + block - 1) / block;
    window_assemble_kernel<<<(unsigned)grid, block, 0, s>>>(src, src_words, bit_begin, nbits, carry, carry_words,
                                                             carry_begin, carry_bits, dst, dst_words, num_rows);
    return cudaGetLastError();
}

cudaError_t launch_reset_queue(unsigned long long *queue, cudaStream_t s) {
    return cudaMemsetAsync(queue, 0, 4 * sizeof(unsigned long long), s);
}

}  // namespace qec

// gwfa_kernels.cu -- the graph wavefront alignment score loop on the GPU.
//
// One CTA runs the whole score loop of one query (Alg. 1): GwfExtend (Alg. 2, with the
// arc spills of Eq. 2's last case), the end test, GwfPrune (Alg. 4) and GwfExpand (Alg. 3),
// until the end cell (|q|, v_e, |v_e|) is on the wavefront.  A persistent grid of CTAs
// pulls query ids from an atomic counter.
//
// A score d is two steps with a barrier after each:
//   offset_pass   visits every tile (the 8 diagonals 8 kb .. 8 kb + 7 of one vertex) that
//                 may change, by four lanes with two diagonals each: GwfExpand of score
//                 d - 1 gathered into the tile (a lane's own sources and its neighbours' by
//                 shuffle, the two edge diagonals' from border words that the neighbour
//                 tiles left), GwfPrune on those sources, GwfExtend of the diagonals that
//                 improved, and the tile's own border words and list entries for score d + 1;
//   spill rounds  the arcs of the diagonals that reached |v| (rare: about 1% of the
//                 diagonals, none in many scores).  They come after the pass because a
//                 spill only fills a diagonal that GwfExpand left absent.  Neighbour tiles
//                 that a border word meets for the first time are looked up beside them.
// A tile is read and written once a score, by one thread group, with plain loads and
// stores: no offset is merged by an atomic, and all the data of a query live in one CTA,
// so they stay in L1 (39 cycles a load there, 275 from L2, 477 for an atomic, which also
// drops its line from L1; all measured).  For the same reason a record is written whole by
// the thread that claims it, not initialised beforehand: the dense records of 760 queries
// at a time fit L2 only while nothing else is fetched for them (10,000 reads 48.3 -> 35.3 ms).
// Measured against the form with separate extend and expand passes that max-merged
// candidates with atomics and probed the hash for each one leaving a tile (reads of
// 1-20 kb): 10,000 reads 101 -> 32 ms, 400 pruned 50 kb reads 50.7 -> 23 ms, one 10 kb
// read 7.7 -> 1.9 ms.
// What bounds it: of the ~13,000 cycles a score of one 10 kb read takes, the pass has 5,000
// (one visit per warp, bound by issue), the second step 7,700: a few warps walk the code
// of links and spills, one after the other, while the rest wait.  Memory is not it: with
// all claims in shared memory and the hash entries fetched ahead the step took as long.
//
// Data (per CTA slab, see SlabLayout; reused across queries):
//   H~     tile records, dense in order of first use, and an open-addressing hash from
//          (v << 32 | kb) to them.  The hash is probed for spills and when two
//          neighbouring tiles meet for the first time (they then hold each other's record
//          index).  Entries persist for the whole query (an entry blocks re-spilling,
//          Alg. 2); the hash is emptied when it ends, a record when it is claimed.
//   lists  (record, vertex) of the tiles to visit in this score and in the next: the tiles
//          with a diagonal in Q and those a border word was left for.  A flag per tile and
//          parity keeps them without repeats.
//
// Order independence (why parallel execution gives the paper's exact result and
// work counts): in Alg. 2 every diagonal of the closure is extended exactly once
// from its starting offset, and a spill only fills an absent diagonal; in Alg. 3
// a diagonal enters Q' iff the max of its candidates beats its old offset, and
// its new value is that max.  Both are independent of the queue order.  Ties of
// the walk base (pruning mode only) are broken by the largest base within one
// breadth-first round of spills, which is what the oracle does too.
#include <cuda_runtime.h>
#include <stdint.h>

#include "gwfa_internal.cuh"

namespace gwfa {

namespace {

// Settled offsets in pruning mode carry whether the diagonal is in Q; a spilled one is
// pending until the spills of its round have been merged.
constexpr long long kTagPend = 0, kTagDead = 2, kTagLive = 3;
constexpr uint32_t kBaseMask = 0x3FFFFFFFu;
constexpr uint32_t kNone = 0xFFFFFFFFu;      // no tile / unclaimed
constexpr uint32_t kNoTrace = 0x3FFFFFFFu;   // trace index of the start diagonal (no predecessor)
constexpr int kAbsent = -2;                  // exact mode: offset -1, not in Q
// Tiles whose "listed for the next score" flag is a bit in shared memory; tiles claimed
// beyond them use a stamp in global memory.  4 KB per parity and CTA.
constexpr uint32_t kBitTiles = 32768;
constexpr uint32_t kSmall = 64;   // spill-list entries kept in shared memory
constexpr uint32_t kLog2Claims = 9;
constexpr uint32_t kLink = 128;   // neighbours to be linked, a score's list in shared memory

template <bool P> struct VT;
template <> struct VT<false> { using T = int; };
template <> struct VT<true> { using T = long long; };

__device__ __forceinline__ long long pk(int j, long long tag, uint32_t base) {
    return ((long long)j << 32) | (tag << 30) | (long long)base;
}
__device__ __forceinline__ int pj(long long v) { return (int)(v >> 32); }
__device__ __forceinline__ uint32_t pbase(long long v) { return (uint32_t)(v & kBaseMask); }

template <bool P> struct Slab {
    TabEnt *table;
    RecT<typename VT<P>::T> *recs;
    uint32_t *touched, *stamp;
    uint2 *list[2], *req, *links;
    unsigned long long *tkey;   // the rest: pruning mode only
    uint32_t *freel, *reqt;
    int4 *req4;
    uint32_t *ins;
    uint2 *trace;
    TraceRec *trec;
    uint32_t cap, rcap, tmask;
};

template <bool P>
__device__ __forceinline__ Slab<P> carve(uint8_t *base, uint32_t log2cap, uint32_t threads) {
    SlabLayout L = slab_layout(log2cap, P, threads);
    Slab<P> s;
    s.table = (TabEnt *)(base + L.table);
    s.recs = (RecT<typename VT<P>::T> *)(base + L.recs);
    s.touched = (uint32_t *)(base + L.touched);
    s.stamp = (uint32_t *)(base + L.stamp);
    s.list[0] = (uint2 *)(base + L.list0);
    s.list[1] = (uint2 *)(base + L.list1);
    s.req = (uint2 *)(base + L.req);
    s.links = (uint2 *)(base + L.links);
    s.tkey = (unsigned long long *)(base + L.tkey);
    s.freel = (uint32_t *)(base + L.freel);
    s.reqt = (uint32_t *)(base + L.reqt);
    s.req4 = (int4 *)(base + L.req);
    s.ins = (uint32_t *)(base + L.ins);
    s.trace = (uint2 *)(base + L.trace);
    s.trec = (TraceRec *)(base + L.trec);
    s.cap = 1u << log2cap;
    s.rcap = slab_records(log2cap, threads);
    s.tmask = 2 * s.cap - 1;
    return s;
}

// Counters of one score; four of them rotate, so that a thread still reading those of
// score d never sees them cleared (score d + 2 does it, a barrier of d + 1 later).
struct Score {
    uint32_t nq;        // list length: tiles to visit in this score (filled by the score before)
    uint32_t nreq;      // arc-spill requests of the offset pass
    uint32_t cells, spills, visited, pruned;
    uint32_t amax;      // largest i + W~ (fits: i < 2^31, W~ < 2^31)
    int found, err;
    uint32_t nlink;     // neighbours to be linked after the pass
    int err_next;       // out of room for a tile that only the next score needs, or kLinksWait
    uint32_t link_stop; // with this many records in use links wait (kNone: they don't)
};

// CTA-shared state of the query being aligned.
struct Sh {
    uint32_t qid;
    uint32_t nt;        // records handed out this query
    uint32_t nclaim;    // tiles that hold a diagonal (the 3/4 load limit counts these)
    uint32_t nr[3];     // requests / insertions of the spill rounds, rotating
    uint32_t nins[2];
    uint32_t held;      // see tiles_held
    int nfree;          // memory bound: records on the free list
    uint32_t tlen;      // traceback: entries of T
    uint32_t peak;
    unsigned long long cells, visited, pruned, spills, evicted;
    unsigned long long end_vp;   // traceback: vertex << 32 | trace of a diagonal at the end point
    unsigned long long t_start;  // query start (global timer, ns)
    unsigned long long t_phase;  // statistics: start of the current pass
    unsigned long long st[6];    // statistics (thread 0 only), see gwfa_engine_set_stats
    Score score[4];
    // the first entries of the score's spill lists: exact mode 2 x kSmall requests (v, ku),
    // pruning mode kSmall requests, then kSmall insertions
    uint4 small[2 * kSmall];
    uint32_t claim[1 << kLog2Claims];   // exact mode: diagonals the spills of a score inserted
    uint2 link[kLink];            // (record | side << 31, vertex)
    uint32_t bits[2][kBitTiles / 32];
};
// With a record per thread behind it, see find_or_insert (a CTA's width is the kernel's).
template <int Threads> struct ShOf {
    Sh sh;
    uint32_t spare[Threads];
};
__device__ __forceinline__ uint32_t &spare_record(Sh &sh) { return ((uint32_t *)(&sh + 1))[threadIdx.x]; }

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// 16 bases starting at base position p of a packed stream.
__device__ __forceinline__ uint32_t window16(const uint32_t *__restrict__ w, uint32_t p) {
    const uint32_t *a = w + (p >> 4);
    return __funnelshift_r(__ldg(a), __ldg(a + 1), (p & 15) * 2);
}

struct QCtx {
    const uint32_t *qw;   // this query's packed words
    int n;
    uint32_t ve;
    bool free_end;        // the walk may end at any position of v_e (or anywhere: any_v)
    bool any_v;           // no end vertex
};

// End test of Alg. 1 on a diagonal just extended to offset j: the point (k + j, j)
// of v is the end point (|q|, |v_e|) of v_e; with a free walk end, any point of
// v_e on query position |q|; without an end vertex, any such point.
__device__ __forceinline__ bool at_end(const QCtx &q, uint32_t v, int k, int j, uint32_t lv) {
    if (k + j != q.n) return false;
    if (q.any_v) return true;
    return v == q.ve && (q.free_end || (uint32_t)j == lv);
}

// 16 query bases from position p.  Plain loads: the server kernel's CTAs write the words
// of their request themselves.
__device__ __forceinline__ uint32_t qwin(const QCtx &q, uint32_t p) {
    const uint32_t *a = q.qw + (p >> 4);
    return __funnelshift_r(a[0], a[1], (p & 15) * 2);
}

// LCP(q[i+1..|q|], v[j+1..|v|]) of Eq. 2 in 0-based positions: XOR of 16-base
// windows, the first differing base is the lowest set bit pair.
__device__ __forceinline__ int lcp(const QCtx &q, int i, const uint32_t *__restrict__ vw, int j, int lv) {
    const int maxl = min(q.n - i, lv - j);
    int l = 0;
    while (l < maxl) {
        const uint32_t x = qwin(q, (uint32_t)(i + l)) ^ window16(vw, (uint32_t)(j + l));
        if (x) {
            l += (__ffs(x) - 1) >> 1;
            break;
        }
        l += 16;
    }
    return min(l, maxl);
}

// Loads that are issued where they stand, ahead of a lookup they do not depend on.
__device__ __forceinline__ uint2 ld_early(const uint4 *p, int half) {
    uint2 r;
    asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"((const uint2 *)p + half));
    return r;
}

// Target of out-arc `a` of v, the `o`-th of its arcs.
__device__ __forceinline__ uint32_t arc_target(const DevGraph &g, uint32_t v, uint32_t a, uint32_t o) {
    return __ldg(o < 4 ? (const uint32_t *)&g.vx[2 * (uint64_t)v + 1] + o : &g.arc_dst[a]);
}

// LCP of a spilled diagonal (offset 0, query position i) when the XOR `x` of its first
// windows is already there.
__device__ __forceinline__ int lcp0(const QCtx &q, int i, const uint32_t *__restrict__ vw, int lv, uint32_t x) {
    const int maxl = min(q.n - i, lv);
    int l = x ? (__ffs(x) - 1) >> 1 : 16;
    if (!x) {
        while (l < maxl) {
            const uint32_t y = qwin(q, (uint32_t)(i + l)) ^ window16(vw, (uint32_t)l);
            if (y) {
                l += (__ffs(y) - 1) >> 1;
                break;
            }
            l += 16;
        }
    }
    return min(l, maxl);
}

// Atomics on slab memory (always device global memory) issued in the global state
// space; the slab pointers come from shared memory, where the compiler no longer
// knows their space.
__device__ __forceinline__ uint32_t g_exch(uint32_t *p, uint32_t v) {
    uint32_t r;
    asm volatile("atom.global.exch.b32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ int g_cas(int *p, int c, int v) {
    int r;
    asm volatile("atom.global.cas.b32 %0, [%1], %2, %3;" : "=r"(r) : "l"(p), "r"(c), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ long long g_max(long long *p, long long v) {
    long long r;
    asm volatile("atom.global.max.s64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(v) : "memory");
    return r;
}
__device__ __forceinline__ void g_max32(uint32_t *p, uint32_t v) {
    asm volatile("red.global.max.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A hash entry is one 16-byte unit: key and record index appear together, so whoever
// finds the key can use the record at once.
struct Ent {
    unsigned long long key, idx;
};
__device__ __forceinline__ Ent ld_ent(const TabEnt *p) {
    Ent e;
    asm volatile("{ .reg .b128 x; ld.relaxed.gpu.global.b128 x, [%2]; mov.b128 {%0, %1}, x; }"
                 : "=l"(e.key), "=l"(e.idx) : "l"(p) : "memory");
    return e;
}
__device__ __forceinline__ Ent cas_ent(TabEnt *p, unsigned long long key, unsigned long long idx) {
    Ent o;
    const unsigned long long empty = kEmptyKey;
    asm volatile("{ .reg .b128 c, n, o; mov.b128 c, {%3, %3}; mov.b128 n, {%4, %5};\n"
                 "  atom.relaxed.gpu.global.cas.b128 o, [%2], c, n; mov.b128 {%0, %1}, o; }"
                 : "=l"(o.key), "=l"(o.idx) : "l"(p), "l"(empty), "l"(key), "l"(idx) : "memory");
    return o;
}

__device__ __forceinline__ unsigned long long tile_key(uint32_t v, int kb) {
    return ((unsigned long long)v << 32) | (uint32_t)kb;
}
__device__ __forceinline__ uint32_t tile_hash(unsigned long long key, uint32_t mask) {
    return (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 32) & mask;
}

// The load limit: 3/4 of the slab's tiles may come to hold a diagonal.
template <bool P> __device__ __forceinline__ uint32_t load_limit(const Slab<P> &s) { return (s.cap >> 1) + (s.cap >> 2); }

// Records that hold a diagonal (or, pruning mode, held one since the last eviction), counted
// by the whole CTA.  The tiles that the links of a score claim belong to the next score, and
// a query that ends in this one does not need them; which of both claimed a tile depends on
// timing, but only the spills have put a diagonal into it.
template <bool P> __device__ __noinline__ uint32_t tiles_held(const Slab<P> &s, Sh &sh) {
    __syncthreads();
    if (threadIdx.x == 0) sh.held = 0;
    __syncthreads();
    uint32_t c = 0;
    for (uint32_t t = threadIdx.x; t < min(sh.nt, s.rcap); t += blockDim.x) {
        if (s.touched[t] == kNone) continue;
        bool any = false;
        if constexpr (P) any = s.recs[t].side[1].counted != 0;
        for (int ln = 0; ln < kTile; ++ln) any = any || s.recs[t].vals[ln] >= 0;
        c += any;
    }
    if (c) atomicAdd(&sh.held, c);
    __syncthreads();
    return sh.held;
}

// An empty record of a tile at kb, written by the thread that claims it, in whole lines:
// they stay in L1, and records need no initialisation before a query nor wiping after it.
template <bool P> __device__ __forceinline__ void empty_record(const Slab<P> &s, uint32_t idx, int kb) {
    uint4 *p = (uint4 *)&s.recs[idx];
    const uint32_t o = 0xFFFFFFFFu;
    if constexpr (P) {
#pragma unroll
        for (int i = 0; i < 8; ++i) p[i] = i == 5 || i == 7 ? make_uint4(o, (uint32_t)kb, 0u, 0u) : make_uint4(o, o, o, o);
    } else {
        p[0] = p[1] = make_uint4(o - 1, o - 1, o - 1, o - 1);   // kAbsent
        p[2] = p[3] = make_uint4(o, o, o, (uint32_t)kb);
    }
    s.touched[idx] = kNone;
    if (idx >= kBitTiles) s.stamp[idx] = kNone;
}

// Links claim tiles beside the spills of a score.  Such a tile belongs to the next score, which
// a query that ends in this one does not need, and with pruning it often stays empty, while a
// spill must find room as long as the tiles that hold a diagonal are within the load limit.
// So links leave the records that the spills may still ask for, and two a thread: one that a
// race has left over, and one that it takes right now.  The rest of the links follows after
// the spills (check_room).
constexpr int kLinksWait = 1;
template <bool P> __device__ __forceinline__ uint32_t records_in_use(const Slab<P> &s, const Sh &sh) {
    return min(sh.nt, s.rcap) - (P ? max(sh.nfree, 0) : 0);
}
template <bool P> __device__ __forceinline__ uint32_t link_stop(const Slab<P> &s, const Sh &sh) {
    return (uint32_t)max((int)(s.rcap - load_limit(s) + sh.nclaim) - 2 * (int)blockDim.x, 0);
}

// Record of tile (v, kb), claimed if absent; -1 (and *err) when the slab is full.  The first
// probe is inline, the rest (and the claim) is not.  A claim puts key and record into the table
// at once, so it brings a record along, and where several threads meet at one new tile (the
// eight diagonals of a neighbour do, and the two vertices of a bubble) all but one are left
// with theirs.  Such a thread keeps it for its next claim: a slab then has at most one record a
// thread in use beside its tiles, and what it has room for does not depend on how often they
// meet (without, 255 spills at once into 32 tiles used 255 records, and a read under the memory
// bound lost one at every bubble, for good).  To claim the key first and have the others wait
// for the record costs them a poll (10,000 reads 32.5 -> 37.5 ms).
template <bool P>
__device__ __noinline__ int find_or_insert_slow(const Slab<P> &s, Sh &sh, unsigned long long key, uint32_t h, Ent e,
                                                int *err) {
    uint32_t idx = kNone;
    for (int probe = 0; probe < 256; ++probe) {
        if (probe > 0) e = ld_ent(&s.table[h]);
        if (e.key == kEmptyKey) {
            if (idx == kNone) {
                idx = spare_record(sh);
                if (idx != kNone) {
                    spare_record(sh) = kNone;
                } else {
                    if constexpr (P) {
                        const int f = sh.nfree > 0 ? atomicSub(&sh.nfree, 1) : 0;
                        idx = f > 0 ? s.freel[f - 1] : atomicAdd(&sh.nt, 1u);
                    } else {
                        idx = atomicAdd(&sh.nt, 1u);
                    }
                    if (idx >= s.rcap) break;
                }
                empty_record<P>(s, idx, (int)(uint32_t)key);
                if constexpr (P) s.tkey[idx] = key;
                __threadfence_block();   // before the key that leads others to it
            }
            e = cas_ent(&s.table[h], key, idx);
            if (e.key == kEmptyKey) {
                s.touched[idx] = h;
                if constexpr (!P) atomicAdd(&sh.nclaim, 1u);   // a claimed tile always gets a diagonal
                return (int)idx;
            }
        }
        if (e.key == key) {
            if (idx != kNone) {
                spare_record(sh) = idx;
                if constexpr (P) s.tkey[idx] = kEmptyKey;
            }
            __threadfence_block();
            return (int)e.idx;
        }
        h = (h + 1) & s.tmask;
    }
    *err = GWFA_ERR_CAPACITY;
    return -1;
}
template <bool P>
__device__ __forceinline__ int find_or_insert(const Slab<P> &s, Sh &sh, uint32_t v, int kb, int *err) {
    const unsigned long long key = tile_key(v, kb);
    const uint32_t h = tile_hash(key, s.tmask);
    const Ent e = ld_ent(&s.table[h]);
    if (e.key != key) return find_or_insert_slow<P>(s, sh, key, h, e, err);
    __threadfence_block();   // see empty_record
    return (int)e.idx;
}

// List a tile for the next score; true for the one caller that has to append it.
template <bool P>
__device__ __forceinline__ bool list_once(const Slab<P> &s, Sh &sh, uint32_t idx, int d) {
    if (idx < kBitTiles) {
        const uint32_t bit = 1u << (idx & 31);
        return !(atomicOr(&sh.bits[(d + 1) & 1][idx >> 5], bit) & bit);
    }
    return g_exch(&s.stamp[idx], (uint32_t)(d + 1)) != (uint32_t)(d + 1);
}

// The neighbour tile on side sd (0 left, 1 right), linked on first use.
template <bool P>
__device__ __noinline__ uint32_t link_neighbour(const Slab<P> &s, Sh &sh, uint32_t idx, uint32_t v, int kb, int sd,
                                                Score &S) {
    // (the look at the room stands where a tile is claimed: in the claiming function, which
    // spills use too, it cost 10,000 reads 33.5 ms, 33.1 so; a second copy of that function for
    // links 32.9, but 100 reads of 1 kb 170.6 us instead of 167.7, in code to fetch)
    const unsigned long long key = tile_key(v, sd ? kb + 1 : kb - 1);
    const uint32_t h = tile_hash(key, s.tmask);
    const Ent e = ld_ent(&s.table[h]);
    int t = (int)e.idx;
    if (e.key != key) {
        if ((P ? records_in_use<P>(s, sh) : sh.nt) >= S.link_stop) {
            atomicCAS(&S.err_next, 0, kLinksWait);
            return kNone;
        }
        t = find_or_insert_slow<P>(s, sh, key, h, e, &S.err_next);
        if (t < 0) return kNone;
    }
    __threadfence_block();   // see empty_record
    s.recs[idx].side[sd].link = (uint32_t)t;
    s.recs[t].side[sd ^ 1].link = idx;
    return (uint32_t)t;
}

// Leave the candidate that an edge diagonal at offset j sends over side sd of its tile
// with the neighbour tile t, for score d + 1.
template <bool P>
__device__ __forceinline__ void leave_border(const Slab<P> &s, uint32_t t, int sd, int j, uint32_t base, int d,
                                             uint32_t tr, bool traceback) {
    const int c = sd ? j : j + 1;   // (k+1, j) to the right, (k-1, j+1) to the left
    if constexpr (P) {
        s.recs[t].side[sd ^ 1].in[(d + 1) & 1] = ((long long)c << 32) | base;
        if (traceback) s.trec[t].in[sd ^ 1][(d + 1) & 1] = tr;
    } else {
        s.recs[t].side[sd ^ 1].in[(d + 1) & 1] = c;
    }
}

// What a diagonal extended outside its tile's visit (a spilled one) owes the next score:
// its tile listed, and its candidate over the tile's edge handed to the neighbour tile.
template <bool P>
__device__ void enter_next(const Slab<P> &s, Sh &sh, const QCtx &q, uint32_t idx, uint32_t v, int k, int j,
                           uint32_t base, uint32_t lv, int d, uint32_t tr, bool traceback) {
    uint32_t *nq = &sh.score[(d + 1) & 3].nq;
    uint2 *next = s.list[(d + 1) & 1];
    if (list_once<P>(s, sh, idx, d)) next[atomicAdd(nq, 1u)] = make_uint2(idx, v);
    const int ln = k & 7;
    const int sd = ln == 7;
    if ((ln == 0 && (uint32_t)j < lv) || (ln == 7 && k + j < q.n)) {
        uint32_t t = s.recs[idx].side[sd].link;
        if (t == kNone) t = link_neighbour<P>(s, sh, idx, v, k >> 3, sd, sh.score[d & 3]);
        if (t == kNone) return;
        leave_border<P>(s, t, sd, j, base, d, tr, traceback);
        if (list_once<P>(s, sh, t, d)) next[atomicAdd(nq, 1u)] = make_uint2(t, v);
    }
}

// The border words of the pass whose neighbour had no link yet, one thread each, from the
// CTA's last threads down (the spills, done in the same step, start with its first): a
// hash lookup, often with a claim, is two dependent L2 round trips and more, and in the
// pass it would hold up the warp's other tiles.
template <bool P>
__device__ __forceinline__ void link_pending(const Slab<P> &s, Sh &sh, int d, uint32_t n, bool traceback) {
    uint32_t *nq = &sh.score[(d + 1) & 3].nq;
    for (uint32_t i = blockDim.x - 1 - threadIdx.x; i < n; i += blockDim.x) {
        const uint2 rq = i < kLink ? sh.link[i] : s.links[i];
        const uint32_t idx = rq.x & 0x7FFFFFFFu;
        const int sd = (int)(rq.x >> 31), ln = sd ? 7 : 0;
        const uint32_t t = link_neighbour<P>(s, sh, idx, rq.y, s.recs[idx].side[0].kb, sd, sh.score[d & 3]);
        if (t == kNone) continue;
        if constexpr (P) {
            const long long v = s.recs[idx].vals[ln];
            leave_border<P>(s, t, sd, pj(v), pbase(v), d, traceback ? s.trec[idx].tr[ln] : 0u, traceback);
        } else {
            leave_border<P>(s, t, sd, s.recs[idx].vals[ln] >> 1, 0u, d, 0u, false);
        }
        if (list_once<P>(s, sh, t, d)) s.list[(d + 1) & 1][atomicAdd(nq, 1u)] = make_uint2(t, rq.y);
    }
}

// GwfPushTrace (Alg. 5): record "vertex v, reached with trace t" and return its
// index in T.  Unlike Alg. 5, equal (v, t) pairs are not merged through a map:
// T then holds one entry per spilling diagonal, which bounds it by the spill count
// and gives the same walk.
__device__ __forceinline__ uint32_t push_trace(const Slab<true> &s, Sh &sh, uint32_t v, uint32_t t, int *err) {
    const uint32_t idx = atomicAdd(&sh.tlen, 1u);
    if (idx >= 2 * s.cap || idx >= kNoTrace) {
        atomicCAS(err, 0, GWFA_ERR_CAPACITY);
        return kNoTrace;
    }
    s.trace[idx] = make_uint2(v, t);
    return idx;
}

// Spill lists: the first entries in shared memory, the rest in the slab.  Exact mode logs a
// score's requests of all rounds, at most one a diagonal that the score extends, so the
// 6 cap diagonals of the tiles that the load limit admits always fit (a run of one base can
// bring them all to the end of their vertices in one score).  More than 2 cap requests are
// so rare that those beyond are kept as the diagonal alone (record << 3 | diagonal), in half
// the space; vertex and position are looked up when such a request is read.
__device__ __forceinline__ uint32_t req_cap(const Slab<false> &s) { return 6 * s.cap; }

__device__ __forceinline__ void put_req(const Slab<false> &s, Sh &sh, uint32_t i, uint32_t v, int ku, uint32_t diag,
                                        int *err) {
    if (i < 4 * kSmall) ((uint2 *)sh.small)[i] = make_uint2(v, (uint32_t)ku);
    else if (i < 2 * s.cap) s.req[i] = make_uint2(v, (uint32_t)ku);
    else if (i < req_cap(s)) ((uint32_t *)s.req)[i + 2 * s.cap] = diag;
    else atomicCAS(err, 0, GWFA_ERR_CAPACITY);
}
__device__ __noinline__ uint2 get_req_diag(const DevGraph &g, const Slab<false> &s, uint32_t i) {
    const uint32_t x = ((const uint32_t *)s.req)[i + 2 * s.cap];
    const unsigned long long key = ld_ent(&s.table[s.touched[x >> 3]]).key;
    const uint32_t v = (uint32_t)(key >> 32);
    return make_uint2(v, (uint32_t)((int)(uint32_t)key * kTile + (int)(x & 7)) + __ldg(&g.vx[2 * (uint64_t)v]).y);
}
__device__ __forceinline__ uint2 get_req(const DevGraph &g, const Slab<false> &s, const Sh &sh, uint32_t i) {
    if (i < 4 * kSmall) return ((const uint2 *)sh.small)[i];
    return i < 2 * s.cap ? s.req[i] : get_req_diag(g, s, i);
}
// Pruning mode: insertion i of a round, (record, vertex, diagonal).  There is room for the
// 6 cap diagonals that the load limit admits (a vertex with many arcs inserts more than it
// requests); beyond the first ones an entry is record << 3 | diagonal.
__device__ __forceinline__ void put_ins(const Slab<true> &s, Sh &sh, uint32_t i, uint32_t rec, uint32_t v, int k, int *err) {
    if (i < kSmall) sh.small[kSmall + i] = make_uint4(rec, v, (uint32_t)k, 0u);
    else if (i < 6 * s.cap) s.ins[i] = rec << 3 | (uint32_t)(k & 7);
    else atomicCAS(err, 0, GWFA_ERR_CAPACITY);
}
__device__ __forceinline__ uint4 get_ins(const Slab<true> &s, const Sh &sh, uint32_t i) {
    if (i < kSmall) return sh.small[kSmall + i];
    const uint32_t x = s.ins[i];
    const unsigned long long key = s.tkey[x >> 3];
    return make_uint4(x >> 3, (uint32_t)(key >> 32), (uint32_t)key * kTile + (x & 7), 0u);
}
__device__ __forceinline__ int4 get_req4(const Slab<true> &s, const Sh &sh, uint32_t i) {
    return i < kSmall ? ((const int4 *)sh.small)[i] : s.req4[i];
}

// Pruning mode: a settled diagonal reached |v|: offset 0 with the walk base past v goes
// to (u, k + |v|) for every arc (v, u), after the pass (see apply_spills).
__device__ __forceinline__ void request_spill(const Slab<true> &s, Sh &sh, uint32_t at, uint32_t lv, uint32_t v,
                                              int k, uint32_t base, uint32_t tr, bool traceback, int *err) {
    const uint32_t nb = base + lv;
    if (nb > kBaseMask) atomicCAS(err, 0, GWFA_ERR_CAPACITY);
    const uint32_t t = traceback ? push_trace(s, sh, v, tr, err) : 0u;
    if (at < s.cap) {
        *(at < kSmall ? (int4 *)&sh.small[at] : &s.req4[at]) = make_int4(k + (int)lv, (int)nb, (int)v, 0);
        if (traceback) s.reqt[at] = t;
    } else {
        atomicCAS(err, 0, GWFA_ERR_CAPACITY);
    }
}

// LCP of two diagonals of one vertex, their first windows loaded together; a diagonal
// with m = 0 is not extended (its positions are 0, so that the loads stay in bounds).
__device__ __forceinline__ void lcp2(const QCtx &q, const uint32_t *__restrict__ vw, const int (&i)[2],
                                     const int (&j)[2], const int (&m)[2], int (&l)[2]) {
    uint32_t x[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) x[u] = qwin(q, (uint32_t)i[u]) ^ window16(vw, (uint32_t)j[u]);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        l[u] = x[u] ? (__ffs(x[u]) - 1) >> 1 : 16;
        if (!x[u] && m[u] > 16) {
            do {
                const uint32_t y = qwin(q, (uint32_t)(i[u] + l[u])) ^ window16(vw, (uint32_t)(j[u] + l[u]));
                if (y) {
                    l[u] += (__ffs(y) - 1) >> 1;
                    break;
                }
                l[u] += 16;
            } while (l[u] < m[u]);
        }
        l[u] = min(l[u], m[u]);
    }
}

// GwfExpand (Alg. 3) of the score before with GwfPrune (Alg. 4) on its sources, and
// GwfExtend (Alg. 2) of this one, in one visit of every listed tile by four lanes with two
// diagonals each: a lane gathers its diagonals' candidates (their own and their
// neighbours', by shuffle from the next lanes, from the tile's border words at its edges),
// keeps the largest where it beats the offset, extends those along equal bases, stores
// them, and hands the next score the tile's list entry and the candidates that leave the
// tile.  Arc spills, and neighbours met for the first time, are only requested here.
// The work around the two comparisons of a lane (entry, record, flags, lists) is most of
// its instructions, so eight tiles share them in a warp.
template <bool P, bool TB>
__device__ __forceinline__ void offset_pass(const DevGraph &g, const Slab<P> &s, Sh &sh, const QCtx &q, int d,
                                            bool prune_on, int max_lag) {
    using T = typename VT<P>::T;
    const unsigned full = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, sub = lane & 3;
    const int par = d & 1;
    Score &S = sh.score[d & 3];
    uint32_t *nq = &sh.score[(d + 1) & 3].nq;
    const uint32_t n_list = S.nq;
    const int sd = sub >> 1;   // the side whose border words this lane reads (lanes 0 and 3 use them)
    uint32_t cells = 0, visited = 0, pruned = 0, amax = 0;
    // the flags of the list being read are spent: clear them for score d + 1
    const uint32_t nw = min((sh.nt + 31) >> 5, kBitTiles / 32);
    for (uint32_t w = threadIdx.x; w < nw; w += blockDim.x) sh.bits[par][w] = 0u;
    for (uint32_t wb = (threadIdx.x >> 5) * 8; wb < n_list; wb += (blockDim.x >> 5) * 8) {
        const uint32_t e = wb + (lane >> 2);
        const bool on = e < n_list;
        const uint2 ent = s.list[par][on ? e : wb];
        RecT<T> *rec = &s.recs[ent.x];
        const uint2 vi = __ldg((const uint2 *)&g.vx[2 * (uint64_t)ent.y]);   // label word, |v|
        T raw[2], in;
        uint32_t link, counted = 0;
        int k[2];
        if constexpr (P) {
            const longlong2 r2 = *(const longlong2 *)&rec->vals[2 * sub];
            raw[0] = r2.x;
            raw[1] = r2.y;
            in = rec->side[sd].in[par];
            const uint4 lk = *(const uint4 *)&rec->side[sd].link;
            link = lk.x;
            k[0] = (int)lk.y * kTile + 2 * sub;
            counted = lk.z;
        } else {
            const int2 r2 = *(const int2 *)&rec->vals[2 * sub];
            raw[0] = r2.x;
            raw[1] = r2.y;
            const int4 sw = *(const int4 *)&rec->side[sd];
            in = par ? sw.y : sw.x;
            link = (uint32_t)sw.z;
            k[0] = sw.w * kTile + 2 * sub;
        }
        k[1] = k[0] + 1;
        uint32_t tr[2] = {0u, 0u}, trn[2] = {0u, 0u}, tin = 0u;
        if constexpr (TB) {
            const uint2 t2 = *(const uint2 *)&s.trec[ent.x].tr[2 * sub];
            tr[0] = t2.x;
            tr[1] = t2.y;
            tin = s.trec[ent.x].in[sd][par];
        }
        if (on && (sub == 0 || sub == 3) && in >= 0) rec->side[sd].in[par] = (T)-1;   // consumed
        else in = (T)-1;
        if (!on) raw[0] = raw[1] = P ? (T)-1 : (T)kAbsent;
        bool live[2], inq[2];
        int j[2];
        uint32_t base[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            base[u] = 0u;
            if constexpr (P) {
                live[u] = raw[u] >= 0 && ((raw[u] >> 30) & 3) == kTagLive;
                j[u] = pj(raw[u]);
                base[u] = pbase(raw[u]);
            } else {
                live[u] = raw[u] & 1;
                j[u] = raw[u] >> 1;
            }
        }
        if (d == 0) {   // the start diagonals are in Q as they are
            inq[0] = live[0];
            inq[1] = live[1];
            trn[0] = tr[0];
            trn[1] = tr[1];
        } else if constexpr (P) {
            if (prune_on) {
                // a source that lags is dropped (its offset stays)
                const long long am = (long long)sh.score[(d + 3) & 3].amax;
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (live[u] && am - ((long long)k[u] + 2ll * j[u] + base[u]) >= (long long)max_lag) {
                        live[u] = false;
                        ++pruned;
                    }
                // and so is one over the edge: (k - 1, c) on the left, (k + 1, c - 1) on the right
                if (in >= 0) {
                    const long long a = (long long)(sub == 0 ? k[0] : k[1]) - 1 + 2ll * pj(in) + pbase(in);
                    if (am - a >= (long long)max_lag) in = (T)-1;
                }
            }
            long long c_ins[2], c_del[2], mis[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const bool ins = live[u] && k[u] + j[u] < q.n, del = live[u] && j[u] < (int)vi.y;
                c_ins[u] = ins ? ((long long)j[u] << 32) | base[u] : -1ll;
                c_del[u] = del ? ((long long)(j[u] + 1) << 32) | base[u] : -1ll;
                mis[u] = ins ? c_del[u] : -1ll;
            }
            long long left = __shfl_up_sync(full, c_ins[1], 1, 4), right = __shfl_down_sync(full, c_del[0], 1, 4);
            uint32_t tl = 0u, tn = 0u;
            if constexpr (TB) {
                tl = __shfl_up_sync(full, tr[1], 1, 4);
                tn = __shfl_down_sync(full, tr[0], 1, 4);
                if (sub == 0) tl = tin;
                if (sub == 3) tn = tin;
            }
            if (sub == 0) left = in;
            if (sub == 3) right = in;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const long long cl = u ? c_ins[0] : left, cr = u ? right : c_del[1];
                long long c = mis[u];
                if (cl > c) c = cl;
                if (cr > c) c = cr;
                inq[u] = c >= 0 && pj(c) > j[u];   // j = -1 where absent
                if constexpr (TB) {
                    // sources of equal offset and base are equally good predecessors: the
                    // largest trace index, for a deterministic choice
                    if (mis[u] == c) trn[u] = tr[u];
                    if (cl == c) trn[u] = max(trn[u], u ? tr[0] : tl);
                    if (cr == c) trn[u] = max(trn[u], u ? tn : tr[1]);
                }
                if (inq[u]) {
                    if (raw[u] < 0) ++visited;
                    j[u] = pj(c);
                    base[u] = pbase(c);
                }
            }
        } else {
            int c_ins[2], c_del[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                c_ins[u] = live[u] && k[u] + j[u] < q.n ? j[u] : -1;
                c_del[u] = live[u] && j[u] < (int)vi.y ? j[u] + 1 : -1;
            }
            int left = __shfl_up_sync(full, c_ins[1], 1, 4), right = __shfl_down_sync(full, c_del[0], 1, 4);
            if (sub == 0) left = in;
            if (sub == 3) right = in;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int c = max(c_ins[u] >= 0 ? c_del[u] : -1, u ? max(c_ins[0], right) : max(left, c_del[1]));
                inq[u] = c > j[u];
                j[u] = max(c, j[u]);
            }
        }
        {
            int i[2], jj[2], m[2], l[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                i[u] = inq[u] ? k[u] + j[u] : 0;
                jj[u] = inq[u] ? j[u] : 0;
                m[u] = inq[u] ? min(q.n - i[u], (int)vi.y - j[u]) : 0;
            }
            lcp2(q, g.words + vi.x, i, jj, m, l);
            j[0] += l[0];
            j[1] += l[1];
        }
        if constexpr (P) {
            // a tile that holds a diagonal for the first time (claimed here or by a spill)
            const unsigned has = __ballot_sync(full, inq[0] || inq[1] || raw[0] >= 0 || raw[1] >= 0);
            if (sub == 3 && !counted && on && ((has >> (lane & 28)) & 15u)) {
                rec->side[1].counted = 1u;
                if (atomicAdd(&sh.nclaim, 1u) + 1 > load_limit(s)) atomicCAS(&S.err, 0, GWFA_ERR_CAPACITY);
            }
            if (on) {
                longlong2 r2;
                r2.x = inq[0] || raw[0] >= 0 ? pk(j[0], inq[0] ? kTagLive : kTagDead, base[0]) : -1ll;
                r2.y = inq[1] || raw[1] >= 0 ? pk(j[1], inq[1] ? kTagLive : kTagDead, base[1]) : -1ll;
                *(longlong2 *)&rec->vals[2 * sub] = r2;
                if (TB) *(uint2 *)&s.trec[ent.x].tr[2 * sub] = make_uint2(inq[0] ? trn[0] : tr[0], inq[1] ? trn[1] : tr[1]);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (inq[u]) amax = max(amax, (uint32_t)(k[u] + j[u]) + (uint32_t)j[u] + base[u]);
        } else {
            // right for every diagonal: an absent one keeps -2, one outside Q its offset
            if (on) *(int2 *)&rec->vals[2 * sub] = make_int2((j[0] << 1) | (inq[0] ? 1 : 0), (j[1] << 1) | (inq[1] ? 1 : 0));
        }
        bool spill[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            spill[u] = inq[u] && j[u] == (int)vi.y;
            if (inq[u] && k[u] + j[u] == q.n && at_end(q, ent.y, k[u], j[u], vi.y)) {
                S.found = 1;
                // one 64-bit store, so that the vertex and its trace stay a pair when
                // several diagonals reach a free end in the same score
                if constexpr (P) sh.end_vp = ((unsigned long long)ent.y << 32) | trn[u];
            }
        }
        const unsigned qm0 = __ballot_sync(full, inq[0]), qm1 = __ballot_sync(full, inq[1]);
        cells += __popc(qm0) + __popc(qm1);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (spill[u]) {
                const uint32_t at = atomicAdd(&S.nreq, 1u);
                if constexpr (P) request_spill(s, sh, at, vi.y, ent.y, k[u], base[u], trn[u], TB, &S.err);
                else put_req(s, sh, at, ent.y, k[u] + (int)vi.y, ent.x << 3 | (uint32_t)(2 * sub + u), &S.err);
            }
        // the next score visits this tile if it has a diagonal in Q (lane 1 lists it), and
        // a neighbour that an edge diagonal's candidate enters (lanes 0 and 3)
        uint32_t target = ent.x;
        bool want = sub == 1 && (((qm0 | qm1) >> (lane & 28)) & 15u);
        if ((sub == 0 && inq[0] && j[0] < (int)vi.y) || (sub == 3 && inq[1] && k[1] + j[1] < q.n)) {
            if (link == kNone) {
                const uint32_t i = atomicAdd(&S.nlink, 1u);
                *(i < kLink ? &sh.link[i] : &s.links[i]) = make_uint2(ent.x | ((uint32_t)sd << 31), ent.y);
            } else {
                leave_border<P>(s, link, sd, sd ? j[1] : j[0], sd ? base[1] : base[0], d, sd ? trn[1] : trn[0], TB);
                target = link;
                want = true;
            }
        }
        __syncwarp();
        const bool fresh = want && list_once<P>(s, sh, target, d);
        const unsigned nm = __ballot_sync(full, fresh);
        if (nm) {
            uint32_t b = 0;
            if (lane == 0) b = atomicAdd(nq, (uint32_t)__popc(nm));
            b = __shfl_sync(full, b, 0) + __popc(nm & ((1u << lane) - 1));
            if (fresh) s.list[par ^ 1][b] = make_uint2(target, ent.y);
        }
    }
    if (lane == 0 && cells) atomicAdd(&S.cells, cells);
    if constexpr (P) {
        visited = __reduce_add_sync(full, visited);
        pruned = __reduce_add_sync(full, pruned);
        amax = __reduce_max_sync(full, amax);
        if (lane == 0) {
            if (visited) atomicAdd(&S.visited, visited);
            if (pruned) atomicAdd(&S.pruned, pruned);
            if (amax) atomicMax(&S.amax, amax);
        }
    }
}

// Exact mode: the one thread that may insert diagonal `ln` of record idx in this score.  The
// claims of a score are kept in a small hash in shared memory (entry: score mod 32, record,
// diagonal; 0 or another score = free): an atomic on the offset itself takes 477 cycles
// and drops the record's line from L1.  An entry is never freed within a score, so a
// thread that finds no room can fall back to that atomic: everyone else with the same
// diagonal finds none either.
__device__ __forceinline__ bool claim_lane(const Slab<false> &s, Sh &sh, uint32_t idx, int ln, int d) {
    const uint32_t tag = (uint32_t)d & 31u, key = tag << 27 | idx << 3 | (uint32_t)ln;
    uint32_t h = (idx << 3 | (uint32_t)ln) * 0x9E3779B1u >> (32 - kLog2Claims);
    for (int probe = 0; probe < 16; ++probe) {
        uint32_t e = sh.claim[h];
        if (e == 0u || e >> 27 != tag) {
            const uint32_t old = e;
            e = atomicCAS(&sh.claim[h], old, key);
            if (e == old) return true;
        }
        if (e == key) return false;
        h = (h + 1) & ((1u << kLog2Claims) - 1);
    }
    return g_cas(&s.recs[idx].vals[ln], kAbsent, 1) == kAbsent;
}

// Exact mode: requests [r0, r0 + n) of the score's log: offset 0 to (u, ku) for every arc
// (v, u) where it is absent (Alg. 2's arc loop).  A spill is a chain of dependent L2 round
// trips (arc, hash entry, offset, label) and a score has a few dozen of them: a pair of
// lanes takes one, an arc a lane (most vertices have one or two).  Packed into few warps
// they run in step: with 1, 2, 4 or 8 requests a warp (four lanes each) 10,000 reads take
// 74.9, 59.6, 52.9 or 48.9 ms, with 16 46.9.  A diagonal that a lane inserts is extended by
// it at once; if that one reaches its vertex's end too, its pair goes on with it (or it is
// logged for the next round when the lane has one waiting already).
__device__ __forceinline__ void spill_round(const DevGraph &g, const Slab<false> &s, Sh &sh, const QCtx &q, int d,
                                            uint32_t r0, uint32_t n, uint32_t *next_count) {
    Score &S = sh.score[d & 3];
    const unsigned full = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, arc = lane & 1;
    uint32_t won = 0;
    for (uint32_t b = (threadIdx.x >> 5) * 16; b < n; b += blockDim.x >> 1) {
        const uint32_t r = b + (uint32_t)(lane >> 1);
        uint2 rq = r < n ? get_req(g, s, sh, r0 + r) : make_uint2(kNone, 0u);
        uint2 wait = make_uint2(kNone, 0u);   // this lane's inserted diagonal that spills in turn
        for (;;) {
            if (rq.x != kNone) {
                const uint4 *vr = &g.vx[2 * (uint64_t)rq.x];
                const uint2 ar = ld_early(vr, 1);
                uint32_t u = __ldg((const uint32_t *)(vr + 1) + arc);   // valid where there is such an arc
                const int ku = (int)rq.y;
                for (uint32_t o = (uint32_t)arc; ar.x + o < ar.y; o += 2) {
                    if (o >= 2) u = arc_target(g, rq.x, ar.x + o, o);
                    const uint2 ui = ld_early(&g.vx[2 * (uint64_t)u], 0);
                    const int su = find_or_insert<false>(s, sh, u, ku >> 3, &S.err);
                    if (su < 0) break;
                    // the offset and the first windows together; most spills end here, the
                    // diagonal being there already
                    const int raw = s.recs[su].vals[ku & 7];
                    const uint32_t x = qwin(q, (uint32_t)ku) ^ __ldg(g.words + ui.x);
                    if (raw != kAbsent || !claim_lane(s, sh, (uint32_t)su, ku & 7, d)) continue;
                    ++won;
                    const int l = lcp0(q, ku, g.words + ui.x, (int)ui.y, x);
                    s.recs[su].vals[ku & 7] = (l << 1) | 1;
                    if (at_end(q, u, ku, l, ui.y)) S.found = 1;
                    enter_next<false>(s, sh, q, (uint32_t)su, u, ku, l, 0u, ui.y, d, 0u, false);
                    if ((uint32_t)l == ui.y) {
                        if (wait.x == kNone) wait = make_uint2(u, (uint32_t)(ku + l));
                        else put_req(s, sh, r0 + n + atomicAdd(next_count, 1u), u, ku + l,
                                     (uint32_t)su << 3 | (uint32_t)(ku & 7), &S.err);
                    }
                }
            }
            const unsigned m = __ballot_sync(full, wait.x != kNone);
            if (!m) break;
            const unsigned m2 = (m >> (lane & 30)) & 3u;
            const int src = m2 ? __ffs(m2) - 1 : 0;
            rq.x = __shfl_sync(full, wait.x, src, 2);
            rq.y = __shfl_sync(full, wait.y, src, 2);
            if (arc == src) wait.x = kNone;
        }
    }
    won = __reduce_add_sync(full, won);
    if (lane == 0 && won) {
        atomicAdd(&S.cells, won);
        atomicAdd(&S.spills, won);
    }
}

// Pruning mode, by `nthr` threads (a warp or the CTA): offset 0 with walk base nb on
// (u, ku) for every request of the round, a quad of lanes a request and a lane an arc; the
// inserted diagonals go to the round's insertion list.  A spill never changes a diagonal
// that was present before the round (Alg. 2's presence test: a settled offset of 0 is
// larger than any pending one), and spills of one round into one diagonal merge by the
// larger walk base.
__device__ __forceinline__ void apply_spills(const DevGraph &g, const Slab<true> &s, Sh &sh, int d, uint32_t n,
                                             uint32_t *n_ins, uint32_t nthr, bool traceback) {
    Score &S = sh.score[d & 3];
    uint32_t won = 0;
    for (uint32_t r = threadIdx.x >> 2; r < min(n, s.cap); r += nthr >> 2) {
        const int4 rq = get_req4(s, sh, r);
        const int ku = rq.x;
        const long long cand = pk(0, kTagPend, (uint32_t)rq.y);
        const uint2 ar = __ldg((const uint2 *)&g.vx[2 * (uint64_t)(uint32_t)rq.z].z);
        for (uint32_t o = threadIdx.x & 3; ar.x + o < ar.y; o += 4) {
            const uint32_t u = arc_target(g, (uint32_t)rq.z, ar.x + o, o);
            const int su = find_or_insert<true>(s, sh, u, ku >> 3, &sh.score[d & 3].err);
            if (su < 0) break;
            if (g_max(&s.recs[su].vals[ku & 7], cand) >= 0) continue;
            ++won;
            if (traceback) s.trec[su].tr[ku & 7] = 0u;   // set by resolve_spill_traces
            put_ins(s, sh, atomicAdd(n_ins, 1u), (uint32_t)su, u, ku, &S.err);
        }
    }
    if (won) {
        atomicAdd(&S.cells, won);
        atomicAdd(&S.spills, won);
        atomicAdd(&S.visited, won);
    }
}

// Traceback with pruning, after apply_spills (and a barrier): every diagonal a spill
// inserted in this round holds the largest base among its spills, still tagged pending;
// each request whose base is that one offers its T index and the largest index wins (any
// of them is a walk of that base, so the choice only has to be deterministic).
__device__ __forceinline__ void resolve_spill_traces(const DevGraph &g, const Slab<true> &s, Sh &sh, int d, uint32_t n,
                                                     uint32_t nthr) {
    for (uint32_t r = threadIdx.x >> 2; r < min(n, s.cap); r += nthr >> 2) {
        const int4 rq = get_req4(s, sh, r);
        const int ku = rq.x;
        const long long cand = pk(0, kTagPend, (uint32_t)rq.y);
        const uint2 ar = __ldg((const uint2 *)&g.vx[2 * (uint64_t)(uint32_t)rq.z].z);
        for (uint32_t o = threadIdx.x & 3; ar.x + o < ar.y; o += 4) {
            const uint32_t u = arc_target(g, (uint32_t)rq.z, ar.x + o, o);
            const int su = find_or_insert<true>(s, sh, u, ku >> 3, &sh.score[d & 3].err);
            if (su < 0) return;
            if (s.recs[su].vals[ku & 7] == cand) g_max32(&s.trec[su].tr[ku & 7], s.reqt[r]);
        }
    }
}

// Pruning mode without traceback, one warp, at most 8 requests of at most four arcs (nearly
// always so): the whole round in one step, a lane an arc.  Every spill of the round is in
// this warp, so a match of the lanes finds those into one diagonal (the largest base wins),
// and the offset needs neither atomic nor second look; the label is compared before it is
// known who wins.  Returns false, having done nothing, if a vertex has more arcs.
__device__ __forceinline__ bool spill_step(const DevGraph &g, const Slab<true> &s, Sh &sh, const QCtx &q, int d,
                                           uint32_t n, uint32_t *n_req) {
    Score &S = sh.score[d & 3];
    const unsigned full = 0xFFFFFFFFu;
    const uint32_t lane = threadIdx.x & 31, r = lane >> 2, arc = lane & 3;
    int4 rq = make_int4(0, 0, 0, 0);
    uint2 ar = make_uint2(0u, 0u);
    uint32_t u = 0;
    if (r < n) {
        rq = get_req4(s, sh, r);
        const uint4 *vr = &g.vx[2 * (uint64_t)(uint32_t)rq.z];
        ar = ld_early(vr, 1);
        u = __ldg((const uint32_t *)(vr + 1) + arc);
    }
    if (__any_sync(full, ar.y - ar.x > 4)) return false;
    const int ku = rq.x, ln = ku & 7;
    int su = -1, j = 0;
    uint32_t base = (uint32_t)rq.y;
    uint2 ui = make_uint2(0u, 0u);
    bool want = ar.x + arc < ar.y;
    if (want) {
        ui = ld_early(&g.vx[2 * (uint64_t)u], 0);
        su = find_or_insert<true>(s, sh, u, ku >> 3, &sh.score[d & 3].err);
        want = su >= 0;
        if (want) {
            const long long raw = s.recs[su].vals[ln];
            const uint32_t x = qwin(q, (uint32_t)ku) ^ __ldg(g.words + ui.x);
            want = raw < 0;
            if (want) j = lcp0(q, ku, g.words + ui.x, (int)ui.y, x);
        }
    }
    __syncwarp();   // the old offsets are read: now they may be written
    const unsigned w = __ballot_sync(full, want);
    if (__popc(w) > 1) {
        const uint32_t key = want ? (uint32_t)su << 3 | (uint32_t)ln : ~lane;
        const unsigned peers = __match_any_sync(full, key);
        for (unsigned m = w; m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const uint32_t b = __shfl_sync(full, base, l);
            if (peers >> l & 1u) base = max(base, b);
        }
        want = want && (int)lane == __ffs(peers) - 1;
    }
    const uint32_t won = (uint32_t)__popc(__ballot_sync(full, want));
    if (want) {
        s.recs[su].vals[ln] = pk(j, kTagLive, base);
        atomicMax(&S.amax, (uint32_t)(ku + j) + (uint32_t)j + base);
        if (at_end(q, u, ku, j, ui.y)) {
            S.found = 1;
            sh.end_vp = (unsigned long long)u << 32;
        }
        enter_next<true>(s, sh, q, (uint32_t)su, u, ku, j, base, ui.y, d, 0u, false);
    }
    __syncwarp();   // every request of this round is read: the next round's may be written
    if (want && (uint32_t)j == ui.y)
        request_spill(s, sh, atomicAdd(n_req, 1u), ui.y, u, ku, base, 0u, false, &S.err);
    if (lane == 0 && won) {
        S.cells += won;
        S.spills += won;
        S.visited += won;
    }
    return true;
}

// Pruning mode: extend the diagonals inserted by the round; those that reach their
// vertex's end request the next round's spills.
__device__ __forceinline__ void extend_spilled(const DevGraph &g, const Slab<true> &s, Sh &sh, const QCtx &q, int d,
                                               uint32_t n, uint32_t *n_req, uint32_t nthr, bool traceback) {
    Score &S = sh.score[d & 3];
    for (uint32_t r = threadIdx.x; r < min(n, 6 * s.cap); r += nthr) {
        const uint4 in = get_ins(s, sh, r);
        const int k = (int)in.z;
        const uint2 vi = __ldg((const uint2 *)&g.vx[2 * (uint64_t)in.y]);
        const uint32_t base = pbase(s.recs[in.x].vals[k & 7]);
        const uint32_t tr = traceback ? s.trec[in.x].tr[k & 7] : 0u;
        const int j = lcp(q, k, g.words + vi.x, 0, (int)vi.y);
        s.recs[in.x].vals[k & 7] = pk(j, kTagLive, base);
        atomicMax(&S.amax, (uint32_t)(k + j) + (uint32_t)j + base);
        if (at_end(q, in.y, k, j, vi.y)) {
            S.found = 1;
            sh.end_vp = ((unsigned long long)in.y << 32) | tr;
        }
        enter_next<true>(s, sh, q, in.x, in.y, k, j, base, vi.y, d, tr, traceback);
        if ((uint32_t)j == vi.y)
            request_spill(s, sh, atomicAdd(n_req, 1u), vi.y, in.y, k, base, tr, traceback, &S.err);
    }
}

// Empty the hash entries of a query; in exact mode, which never removes a diagonal from
// H~, also count the diagonals its records hold (the visited ones).
template <bool P> __device__ void wipe(const Slab<P> &s, Sh &sh) {
    const uint32_t nt = min(sh.nt, s.rcap);
    for (uint32_t t = threadIdx.x; t < nt; t += blockDim.x) {
        const uint32_t h = s.touched[t];
        if (h != kNone) *(uint4 *)&s.table[h] = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    if constexpr (!P) {
        uint32_t c = 0;
        for (uint32_t t = threadIdx.x; t < 2 * nt; t += blockDim.x) {
            const int4 v = *(const int4 *)&s.recs[t >> 1].vals[4 * (t & 1)];
            c += (v.x >= 0) + (v.y >= 0) + (v.z >= 0) + (v.w >= 0);
        }
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if ((threadIdx.x & 31) == 0 && c) atomicAdd(&sh.visited, (unsigned long long)c);
    }
}

// Memory bound on H~ (pruning mode, called every evict_every scores between the offset
// pass and the arc spills, so right after GwfExpand as far as the entries outside Q are
// concerned): the diagonals in Q and those whose anti-diagonal a = i + W~ lags the score
// before's a_max by less than `lag` are kept, the others are removed (sh.evicted).  The
// hash is rebuilt from the tiles that still hold a diagonal or are listed for the next
// score; the records of the others go to the free list.  Records never move, so lists,
// flags and border words stay valid; the links between neighbours, which could point to a
// freed record, are dropped and found again on use.  A removed diagonal may be inserted
// again later, like any absent one.
__device__ __noinline__ void evict_behind(const Slab<true> &s, Sh &sh, long long amax, long long lag, int d) {
    const uint32_t nt = min(sh.nt, s.rcap);
    for (uint32_t t = threadIdx.x; t < nt; t += blockDim.x) {
        const uint32_t h = s.touched[t];
        if (h != kNone) *(uint4 *)&s.table[h] = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    if (threadIdx.x == 0) {
        sh.nclaim = 0;
        if (sh.nfree < 0) sh.nfree = 0;
    }
    __syncthreads();
    uint32_t ev = 0;
    for (uint32_t t = threadIdx.x; t < nt; t += blockDim.x) {
        const unsigned long long key = s.tkey[t];
        if (key == kEmptyKey) continue;   // free, or some thread's spare
        const int kb = (int)(uint32_t)(key & 0xFFFFFFFFull);
        bool any = false;
#pragma unroll
        for (int ln = 0; ln < kTile; ++ln) {
            const long long v = s.recs[t].vals[ln];
            if (v < 0) continue;
            const long long a = (long long)(kb * kTile + ln) + 2ll * pj(v) + (long long)pbase(v);
            if (((v >> 30) & 3) == kTagLive || amax - a < lag) {
                any = true;
            } else {
                s.recs[t].vals[ln] = -1ll;
                ++ev;
            }
        }
        s.recs[t].side[0].link = s.recs[t].side[1].link = kNone;
        s.recs[t].side[1].counted = any ? 1u : 0u;
        const bool listed = t < kBitTiles ? (sh.bits[(d + 1) & 1][t >> 5] >> (t & 31)) & 1u
                                          : s.stamp[t] == (uint32_t)(d + 1);
        if (any) atomicAdd(&sh.nclaim, 1u);
        if (any || listed) {
            uint32_t h = tile_hash(key, s.tmask);
            while (cas_ent(&s.table[h], key, t).key != kEmptyKey) h = (h + 1) & s.tmask;   // at most half full
            s.touched[t] = h;
        } else {
            s.tkey[t] = kEmptyKey;
            s.touched[t] = kNone;
            s.freel[atomicAdd(&sh.nfree, 1)] = t;
        }
    }
    ev = __reduce_add_sync(0xFFFFFFFFu, ev);
    if ((threadIdx.x & 31) == 0 && ev) atomicAdd(&sh.evicted, (unsigned long long)ev);
    __syncthreads();
    if (threadIdx.x == 0) sh.score[d & 3].link_stop = link_stop<true>(s, sh);
    __syncthreads();
}

// Whether the slab has room for score d, over the tiles that it needs, and for the next one,
// unless this is the last.  The links that waited for the spills get their turn here: every
// diagonal in Q at an edge of its tile (all such tiles are listed by now) hands its candidate
// over, to most neighbours for the second time, which does nothing.  In pruning mode the empty
// tiles are cleared away first if the records might not do.
enum Room { kRoom, kNoRoom, kNoRoomNext };
template <bool P>
__device__ __noinline__ Room check_room(const uint4 *vx, const Slab<P> &s, Sh &sh, int n, int d, bool last, bool traceback) {
    Score &S = sh.score[d & 3];
    uint32_t *nq = &sh.score[(d + 1) & 3].nq;
    const bool over = !P && sh.nclaim > load_limit(s);
    if ((over || (P && S.found)) && tiles_held<P>(s, sh) > load_limit(s)) return kNoRoom;
    if (last) return kRoom;
    if (over || S.err_next != kLinksWait) return kNoRoomNext;
    const uint32_t listed = *nq;
    if constexpr (P) {
        if (s.rcap - records_in_use<P>(s, sh) < 2 * listed + blockDim.x) evict_behind(s, sh, 0, 1ll << 62, d);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        S.err_next = P && sh.nclaim > load_limit(s) ? GWFA_ERR_CAPACITY : 0;
        S.link_stop = kNone;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 2 * listed; i += blockDim.x) {
        const uint2 ent = s.list[(d + 1) & 1][i >> 1];
        const int sd = (int)(i & 1), ln = sd ? 7 : 0, kb = s.recs[ent.x].side[0].kb;
        const auto v = s.recs[ent.x].vals[ln];
        bool live;
        int j;
        uint32_t base = 0u;
        if constexpr (P) {
            live = v >= 0 && ((v >> 30) & 3) == kTagLive;
            j = pj(v);
            base = pbase(v);
        } else {
            live = v & 1;
            j = v >> 1;
        }
        if (!live || (sd ? kb * kTile + 7 + j >= n : j >= (int)__ldg(&vx[2 * (uint64_t)ent.y]).y)) continue;
        const uint32_t t = link_neighbour<P>(s, sh, ent.x, ent.y, kb, sd, sh.score[d & 3]);
        if (t == kNone) continue;
        leave_border<P>(s, t, sd, j, base, d, traceback ? s.trec[ent.x].tr[ln] : 0u, traceback);
        if (list_once<P>(s, sh, t, d)) s.list[(d + 1) & 1][atomicAdd(nq, 1u)] = make_uint2(t, ent.y);
    }
    __syncthreads();
    return S.err_next || (!P && sh.nclaim > load_limit(s)) ? kNoRoomNext : kRoom;
}

template <bool P, bool TB>
__device__ __forceinline__ void align_one(const TierArgs &A, const Slab<P> &s, Sh &sh, uint32_t qid) {
    const DevGraph &g = A.g;
    const uint64_t qo = A.q_off[qid];
    QCtx q;
    q.n = (int)(A.q_off[qid + 1] - qo);
    q.qw = A.qwords + (qo >> 4) + qid;
    const uint32_t vs = A.v_s[qid];
    q.ve = A.v_e[qid];
    int pre = 0;
    if (A.qstatus) pre = A.qstatus[qid];
    q.any_v = (A.ends & GWFA_EXTEND) != 0;
    q.free_end = (A.ends & (GWFA_FREE_END | GWFA_EXTEND)) != 0;
    if (q.any_v) q.ve = vs;   // no end vertex: v_e is not read
    if (!pre && (vs >= g.nv || q.ve >= g.nv)) pre = GWFA_ERR_INVALID;
    if (pre) {
        if (threadIdx.x == 0) {
            gwfa_result r = {};
            r.status = pre;
            r.edit_distance = -1;
            A.out[qid] = r;
        }
        return;
    }
    // Alg. 1 initialisation: H~_{v_s,0} <- 0, Q <- [(v_s, 0)], d <- 0
    spare_record(sh) = kNone;
    if (threadIdx.x == 0) {
        sh.t_start = globaltimer_ns();
        for (int i = 0; i < 6; ++i) sh.st[i] = 0;
        for (int i = 0; i < 4; ++i) sh.score[i] = Score{};
        sh.nt = sh.nclaim = 0;
        sh.nfree = 0;
        sh.cells = sh.visited = sh.pruned = sh.spills = sh.evicted = 0;
        sh.peak = 0;
        sh.tlen = 0;
        sh.end_vp = ((unsigned long long)q.ve << 32) | kNoTrace;
        const int t = find_or_insert<P>(s, sh, vs, 0, &sh.score[0].err);
        if (t >= 0) {
            if constexpr (P) {
                s.recs[t].vals[0] = pk(0, kTagLive, 0u);
                if (TB) s.trec[t].tr[0] = kNoTrace;
                sh.visited = 1;
            } else {
                s.recs[t].vals[0] = 1;
            }
            s.list[0][0] = make_uint2((uint32_t)t, vs);
            sh.score[0].nq = 1;
        }
    }
    for (uint32_t w = threadIdx.x; w < kBitTiles / 32; w += blockDim.x) sh.bits[0][w] = sh.bits[1][w] = 0u;
    if constexpr (!P)
        for (uint32_t w = threadIdx.x; w < 1u << kLog2Claims; w += blockDim.x) sh.claim[w] = 0u;
    __syncthreads();
    if (A.ends & GWFA_FREE_START) {
        // free walk start (Sec. 2.1 variant): query position 0 also faces every
        // position j of v_s, i.e. the diagonals (v_s, -j) start with offset j
        const int lvs = (int)__ldg(&g.vinfo[vs]).y;
        const int ntile = (lvs + kTile - 1) / kTile;   // tiles kb = -1 .. -ntile
        for (int i = threadIdx.x; i < ntile; i += blockDim.x) {
            const int kb = -1 - i;
            const int t = find_or_insert<P>(s, sh, vs, kb, &sh.score[0].err);
            if (t < 0) continue;
            uint32_t cnt = 0;
            for (int ln = 0; ln < kTile; ++ln) {
                const int j = -(kb * kTile + ln);
                if (j > lvs) continue;
                ++cnt;
                if constexpr (P) {
                    s.recs[t].vals[ln] = pk(j, kTagLive, 0u);
                    if (TB) s.trec[t].tr[ln] = kNoTrace;
                } else {
                    s.recs[t].vals[ln] = (j << 1) | 1;
                }
            }
            if constexpr (P) {
                atomicAdd(&sh.visited, (unsigned long long)cnt);
            }
            s.list[0][atomicAdd(&sh.score[0].nq, 1u)] = make_uint2((uint32_t)t, vs);
        }
        __syncthreads();
    }

    int d = 0, status = 0;
    for (;; ++d) {
        Score &S = sh.score[d & 3];
        if (threadIdx.x == blockDim.x - 32) {   // the last warp: the first to run out of tiles
            sh.score[(d + 2) & 3] = Score{};
            S.link_stop = link_stop<P>(s, sh);
            sh.nr[0] = 0;
            sh.nins[0] = 0;
        }
        if (A.stats && threadIdx.x == 0) sh.t_phase = globaltimer_ns();
        // ---- GwfExpand of the last score (Alg. 3, with GwfPrune, Alg. 4) and GwfExtend of this one
        bool prune_on = false;
        long long amax = 0;
        if constexpr (P) {
            amax = (long long)sh.score[(d + 3) & 3].amax;
            prune_on = A.max_lag > 0 && amax > (long long)A.max_lag;
            offset_pass<P, TB>(g, s, sh, q, d, prune_on, A.max_lag);
        } else {
            offset_pass<P, false>(g, s, sh, q, d, false, 0);
        }
        __syncthreads();
        if (A.stats && threadIdx.x == 0) {
            const unsigned long long t = globaltimer_ns();
            sh.st[0] += t - sh.t_phase;
            sh.t_phase = t;
            sh.st[2] += 1;
            sh.st[3] += S.nq;
            sh.st[4] += sh.score[(d + 1) & 3].nq;
            sh.st[5] = max(sh.st[5], (unsigned long long)S.nq);
        }
        if (S.cells == 0) {   // GwfExpand left Q empty (or there was no room for v_s)
            status = S.err ? S.err : P && A.max_lag > 0 ? GWFA_ERR_EMPTY_FRONTIER : GWFA_ERR_UNREACHABLE;
            break;
        }
        if constexpr (P) {
            if (!TB && A.evict_lag > 0 && d > 0 && d % A.evict_every == 0) evict_behind(s, sh, amax, A.evict_lag, d);
        }
        // ---- arc spills, in rounds until no extended diagonal reaches its vertex's end
        uint32_t n = S.nreq;
        const uint32_t nl = S.nlink;
        if (nl) link_pending<P>(s, sh, d, nl, TB);
        if constexpr (P) {
            // few requests (the usual case): one warp does every round by itself, and the
            // others wait once instead of twice or three times a round
            const bool solo = n <= 32;
            const uint32_t nthr = solo ? 32u : blockDim.x;
            auto sync = [&]() {
                if (solo) __syncwarp();
                else __syncthreads();
            };
            const bool any = n > 0 || nl > 0;
            if (!solo || threadIdx.x < 32) {
                for (int round = 0; n; ++round) {
                    uint32_t *next_count = &sh.nr[round % 3], *n_ins = &sh.nins[round & 1];
                    if (threadIdx.x == 0) {
                        sh.nr[(round + 1) % 3] = 0;
                        sh.nins[(round + 1) & 1] = 0;
                    }
                    if (solo && n <= 8 && !TB && spill_step(g, s, sh, q, d, n, next_count)) {
                        __syncwarp();
                        n = *next_count;
                        if (A.stats && threadIdx.x == 0 && n) sh.st[2] += 1;
                        continue;
                    }
                    apply_spills(g, s, sh, d, n, n_ins, nthr, TB);
                    sync();
                    if (TB) {
                        resolve_spill_traces(g, s, sh, d, n, nthr);
                        sync();
                    }
                    extend_spilled(g, s, sh, q, d, *n_ins, next_count, nthr, TB);
                    sync();
                    n = *next_count;
                    if (A.stats && threadIdx.x == 0 && n) sh.st[2] += 1;
                }
            }
            if (solo && any) __syncthreads();
        } else {
            // the log's end: more requests than it holds were refused, and end the score
            uint32_t r0 = 0;
            n = min(n, req_cap(s));
            for (int round = 0; n; ++round) {
                uint32_t *next_count = &sh.nr[round % 3];
                if (threadIdx.x == 0) sh.nr[(round + 1) % 3] = 0;
                spill_round(g, s, sh, q, d, r0, n, next_count);
                r0 += n;
                __syncthreads();
                n = *next_count;
                n = min(n, req_cap(s) - r0);
                if (A.stats && threadIdx.x == 0 && n) sh.st[2] += 1;
            }
            if (nl && !r0) __syncthreads();
        }
        if (threadIdx.x == blockDim.x - 32) {
            sh.cells += S.cells;
            sh.spills += S.spills;
            sh.peak = max(sh.peak, S.cells);
            if constexpr (P) {
                sh.visited += S.visited;
                sh.pruned += S.pruned;
            }
        }
        if (A.stats && threadIdx.x == 0) sh.st[1] += globaltimer_ns() - sh.t_phase;
        if (S.err) { status = S.err; break; }
        // rare: a query passes here once, or in pruning mode ends with most of the slab in use
        Room room = kRoom;
        if (S.err_next || (P ? S.found && sh.nt > load_limit(s) : sh.nclaim > load_limit(s)))
            room = check_room<P>(g.vx, s, sh, q.n, d, S.found || (A.max_score >= 0 && d >= A.max_score), TB);
        if (room == kNoRoom) { status = GWFA_ERR_CAPACITY; break; }
        if (S.found) break;   // end test of Alg. 1
        if (A.max_score >= 0 && d >= A.max_score) { status = GWFA_ERR_SCORE_LIMIT; break; }
        if (room == kNoRoomNext) { status = GWFA_ERR_CAPACITY; ++d; break; }
    }
    __syncthreads();
    const uint32_t n_tiles = A.stats ? tiles_held<P>(s, sh) : 0u;
    if constexpr (P) {
        if (threadIdx.x == 0) {
            const Score &S = sh.score[d & 3];
            // the diagonals a failing last pass dropped or inserted
            if (S.cells == 0) {
                sh.visited += S.visited;
                sh.pruned += S.pruned;
            }
            if (TB && status == 0) {
                // GwfTraceback (Alg. 6): push the end vertex, then follow T back to the
                // start and write the walk in order
                const uint32_t te = push_trace(s, sh, (uint32_t)(sh.end_vp >> 32), (uint32_t)sh.end_vp & 0xFFFFFFFFu,
                                               &sh.score[0].err);
                uint32_t len = 0;
                for (uint32_t t = te; t != kNoTrace && len <= sh.tlen; t = s.trace[t].y) ++len;
                if (A.path_len) A.path_len[qid] = len;
                uint32_t pos = len;
                for (uint32_t t = te; t != kNoTrace && pos > 0; t = s.trace[t].y) {
                    --pos;
                    if (A.paths && pos < A.path_cap) A.paths[(uint64_t)qid * A.path_cap + pos] = s.trace[t].x;
                }
            }
        }
    }
    wipe<P>(s, sh);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (status == GWFA_ERR_CAPACITY && A.retry) {
            const uint32_t r = atomicAdd(A.retry_count, 1u);
            A.retry[r] = qid;   // the retry list has room for every query
        } else {
            gwfa_result r = {};
            r.status = status;
            r.edit_distance = status == 0 ? d : -1;
            r.is_upper_bound = sh.pruned > 0 ? 1 : 0;
            r.n_scores = (uint32_t)(d + 1);
            r.cells = sh.cells;
            r.visited = sh.visited;
            r.peak_frontier = sh.peak;
            r.pruned = sh.pruned;
            r.spills = sh.spills;
            r.evicted = sh.evicted;
            r.device_us = (uint32_t)min((globaltimer_ns() - sh.t_start) / 1000ull, 0xFFFFFFFFull);
            A.out[qid] = r;
            if (A.stats) {
                unsigned long long *o = A.stats + (uint64_t)qid * kStatWords;
                for (int i = 0; i < 6; ++i) o[i] = sh.st[i];
                o[6] = n_tiles;
                o[7] = (unsigned long long)(d + 1);
            }
        }
    }
}

// The persistent loop of a CTA: pull a query id, run its score loop, repeat.
template <bool P, bool TB, int Threads>
__device__ __forceinline__ void align_queries(const TierArgs &A) {
    __shared__ ShOf<Threads> shared;
    Sh &sh = shared.sh;
    // the slab's array pointers are the same for every thread: held once in shared
    // memory rather than in each thread's registers (where, at 32 registers, they
    // were spilled to local memory and reloaded through L1/L2 in the hot phases);
    // visible to all threads after the first barrier of the loop below
    __shared__ Slab<P> s;
    if (A.len_hi) {
        const uint64_t len = (A.q_off[A.n_all] - A.q_off[0]) / A.n_all;
        if (len < A.len_lo || len >= A.len_hi) return;   // the same for every thread of the grid
    }
    if (threadIdx.x == 0) s = carve<P>(A.slabs + (uint64_t)blockIdx.x * A.slab_bytes, A.log2cap, A.slab_threads);
    const uint32_t count = A.list_count ? *A.list_count : A.count_val;
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t t = atomicAdd(A.head, 1u);
            sh.qid = t < count ? (A.list ? A.list[A.list_offset + t] : A.list_offset + t) : 0xFFFFFFFFu;
        }
        __syncthreads();
        const uint32_t qid = sh.qid;
        __syncthreads();
        if (qid == 0xFFFFFFFFu) break;
        align_one<P, TB>(A, s, sh, qid);
    }
}

// Up to kNarrow threads: the throughput shape, 6 CTAs per SM at 40 registers: 10,000 reads of
// 1-20 kb take 32.0 ms, 34.5 at 5 with 48, 55 at 7 (36 registers spill), 38 for eight CTAs of
// 192 threads, 35.7 for four of 384.  Pruning mode, with 64-bit offsets, 4 at 64: 400 pruned
// 50 kb reads 23.3 ms, 24.2 at 5 with 48, 26.5 at 6.  Traceback is a kernel of its own: with
// the switch at run time the pruning kernel's code was twice as long, and the few warps that
// do a score's spills are bound by the instructions they fetch (24.5 -> 23.3 ms together
// with spill_step).
template <bool P, bool TB>
__global__ void __launch_bounds__(kNarrow, P ? 4 : 6) align_kernel(TierArgs A) {
    align_queries<P, TB, kNarrow>(A);
}

// Up to 1024 threads, 64 registers: more groups on one query, for batches and queries
// whose own latency is the bound.
template <bool P, bool TB>
__global__ void __launch_bounds__(1024, 1) align_kernel_wide(TierArgs A) {
    align_queries<P, TB, 1024>(A);
}

__device__ __forceinline__ unsigned long long ld_acquire_sys(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_sys(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Serving: a persistent kernel whose CTAs take requests from host-published rings
// (continuous batching: a CTA starts a new request as soon as it finishes one).
// The first CTAs serve class 1 (large slabs) and also take class-0 requests whenever no
// class-1 request waits, so large slabs are never left idle while small requests queue; the
// last n_small serve class 0 (small hash slabs).  So where a configuration has more CTAs
// than the GPU holds (14 an SM by their shared memory), those that wait for room are of the
// class that others serve too.  Every
// wait is bounded: a CTA idle for wait_limit polls votes idle (and withdraws the
// vote if work comes); the CTAs leave together once every CTA has voted, or after
// 16 x wait_limit polls in any case, and the host relaunches the kernel when work
// comes.  Leaving together keeps the full set of CTAs whenever the kernel runs.
// CTAs per SM are a template parameter: with fewer of them a thread has more registers (64,
// 40 or 32 at 2, 3 or 4).
template <bool P, int PerSm>
__global__ void __launch_bounds__(512, PerSm) server_kernel(ServerArgs S) {
    uint32_t *const qst = S.stage + (uint64_t)blockIdx.x * S.slot_words;   // the request's packed words
    __shared__ ShOf<512> shared;
    Sh &sh = shared.sh;
    __shared__ unsigned long long s_ticket;
    __shared__ uint64_t s_qoff[2];
    __shared__ uint32_t s_vs, s_ve;
    __shared__ int s_go, s_ring;
    const uint32_t n_big = S.n_ctas - S.n_small;
    const int cls = blockIdx.x < n_big ? 1 : 0;
    uint8_t *base = cls == 0 ? S.slabs + (uint64_t)(blockIdx.x - n_big) * S.slab_bytes[0]
                             : S.slabs + S.big_offset + (uint64_t)blockIdx.x * S.slab_bytes[1];
    __shared__ Slab<P> s;   // as in align_queries; visible after the first poll barrier
    if (threadIdx.x == 0) s = carve<P>(base, S.log2cap[cls], kMaxThreads);
    for (;;) {
        if (threadIdx.x == 0) {
            int go = 0;
            uint32_t polls = 0;
            bool voted = false;
            for (;;) {
                if (ld_acquire_sys(S.stop)) break;
                // the CTA's own ring first; a large-slab CTA then looks at ring 0
                int rc = -1;
                unsigned long long h = 0;
                for (int c = cls; c >= 0; --c) {
                    const unsigned long long hc = atomicAdd(S.head + c, 0ull);
                    if (hc < ld_acquire_sys(S.tail[c])) {
                        rc = c;
                        h = hc;
                        break;
                    }
                }
                if (rc >= 0) {
                    if (voted) {
                        atomicSub(S.idle_votes, 1u);
                        voted = false;
                    }
                    polls = 0;
                    if (atomicCAS(S.head + rc, h, h + 1) == h) {
                        s_ticket = h;
                        s_ring = rc;
                        go = 1;
                        break;
                    }
                    continue;
                }
                ++polls;
                if (!voted && polls > S.wait_limit) {
                    atomicAdd(S.idle_votes, 1u);
                    voted = true;
                }
                if (voted && (atomicAdd(S.idle_votes, 0u) >= S.n_ctas || polls > 16u * S.wait_limit)) {
                    atomicAdd(S.timeouts, 1ull);
                    break;
                }
                __nanosleep(S.sleep_ns);
            }
            s_go = go;
        }
        __syncthreads();
        if (!s_go) break;
        const unsigned long long ticket = s_ticket;
        const int rc = s_ring;   // the ring the request came from (its result goes back there)
        const uint32_t slot = (uint32_t)(ticket % S.ring);
        const ReqDesc *d = S.desc[rc] + slot;
        const uint32_t n = __ldcv(&d->n);
        const uint32_t nw = (n + 15) >> 4;
        const uint32_t *src = S.arena[rc] + (uint64_t)slot * S.slot_words;
        for (uint32_t w = threadIdx.x; w < nw + 2; w += blockDim.x) qst[w] = w < nw ? __ldcv(src + w) : 0u;
        if (threadIdx.x == 0) {
            s_qoff[0] = 0;
            s_qoff[1] = n;
            s_vs = __ldcv(&d->v_s);
            s_ve = __ldcv(&d->v_e);
        }
        __syncthreads();
        TierArgs A{};
        A.g = S.g;
        A.qwords = qst;
        A.q_off = s_qoff;
        A.v_s = &s_vs;
        A.v_e = &s_ve;
        A.out = S.results[rc] + slot;
        A.max_lag = S.max_lag;
        A.max_score = S.max_score;
        align_one<P, false>(A, s, sh, 0);
        if (threadIdx.x == 0) {
            __threadfence_system();
            st_release_sys(S.done[rc] + slot, ticket + 1);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ int base_code(unsigned char c) {
    switch (c) {
    case 'A': case 'a': return 0;
    case 'C': case 'c': return 1;
    case 'G': case 'g': return 2;
    case 'T': case 't': return 3;
    default: return -1;
    }
}

// 2-bit packing of the queries (a2): one warp per query, one 16-base word per lane.
__global__ void pack_kernel(uint32_t nq, const char *__restrict__ q, const uint64_t *__restrict__ off,
                            uint32_t *__restrict__ words, int32_t *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    const uint32_t wpb = blockDim.x >> 5;
    for (uint32_t qi = blockIdx.x * wpb + (threadIdx.x >> 5); qi < nq; qi += gridDim.x * wpb) {
        const uint64_t a = off[qi], n = off[qi + 1] - a;
        const uint64_t w0 = (a >> 4) + qi, nw = (n + 15) >> 4;
        bool bad = false;
        for (uint64_t t = lane; t < nw; t += 32) {
            uint32_t w = 0;
            for (int c = 0; c < 16; ++c) {
                const uint64_t p = t * 16 + c;
                if (p < n) {
                    int code = base_code((unsigned char)q[a + p]);
                    if (code < 0) { bad = true; code = 0; }
                    w |= (uint32_t)code << (2 * c);
                }
            }
            words[w0 + t] = w;
        }
        bad = __any_sync(0xFFFFFFFFu, bad);
        if (lane == 0 && status) status[qi] = bad ? GWFA_ERR_INVALID : 0;
    }
    if (blockIdx.x == 0 && threadIdx.x < 2) words[(off[nq] >> 4) + nq + threadIdx.x] = 0;
}

// A queue order for a batch that comes without one: longest first, by the length's exponent
// and five bits of its mantissa (a counting sort of one block; the order within a class of
// lengths is left to the atomics, results do not depend on it).  A query that starts last
// ends last, and the longest take a hundred times the median.
__global__ void __launch_bounds__(1024) order_kernel(uint32_t n, const uint64_t *__restrict__ off,
                                                     uint32_t *__restrict__ order) {
    __shared__ uint32_t at[1024], warp_sum[32];
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    auto cls = [&](uint32_t i) {
        const uint32_t len = (uint32_t)min(off[i + 1] - off[i], (uint64_t)0x7FFFFFFF);
        const uint32_t e = 31 - __clz(len | 1u);
        return 1023u - (e << 5 | ((len << (31 - e)) >> 26 & 31u));   // longest: class 0
    };
    at[tid] = 0;
    __syncthreads();
    for (uint32_t i = tid; i < n; i += 1024) atomicAdd(&at[cls(i)], 1u);
    __syncthreads();
    const uint32_t mine = at[tid];
    uint32_t x = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) warp_sum[tid >> 5] = x;
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t w = 0; w < tid >> 5; ++w) before += warp_sum[w];
    at[tid] = before + x - mine;
    __syncthreads();
    for (uint32_t i = tid; i < n; i += 1024) order[atomicAdd(&at[cls(i)], 1u)] = i;
}

// Slabs start with an empty hash (all ones); everything else is written before it is read.
__global__ void slab_init_kernel(uint8_t *slabs, uint64_t slab_bytes, uint32_t n_slabs, uint64_t table_bytes) {
    const uint64_t per = table_bytes / 16, total = per * n_slabs;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x)
        *(uint4 *)(slabs + (i / per) * slab_bytes + (i % per) * 16) = make_uint4(~0u, ~0u, ~0u, ~0u);
}

}  // namespace

// the alignment kernel of a mode and CTA width
static void (*align_entry(bool prune, bool traceback, uint32_t threads))(TierArgs) {
    if (threads > kNarrow)
        return !prune ? align_kernel_wide<false, false> : traceback ? align_kernel_wide<true, true> : align_kernel_wide<true, false>;
    return !prune ? align_kernel<false, false> : traceback ? align_kernel<true, true> : align_kernel<true, false>;
}

cudaError_t launch_align(const TierArgs &a, bool prune, uint32_t ctas, uint32_t threads,
                         cudaStream_t st) {
    align_entry(prune, a.traceback != 0, threads)<<<ctas, threads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_server(const ServerArgs &a, bool prune, uint32_t ctas, uint32_t threads, int sms,
                          cudaStream_t st) {
    // the fewest CTAs per SM that hold them all (above 4 per SM narrower ones still fit)
    const uint32_t per_sm = (ctas + (uint32_t)sms - 1) / (uint32_t)sms;
    void (*k)(ServerArgs) = per_sm <= 2 ? (prune ? server_kernel<true, 2> : server_kernel<false, 2>)
                            : per_sm == 3 ? (prune ? server_kernel<true, 3> : server_kernel<false, 3>)
                                          : (prune ? server_kernel<true, 4> : server_kernel<false, 4>);
    k<<<ctas, threads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_pack(uint32_t nq, const char *d_q, const uint64_t *d_off, uint32_t *d_words,
                        int32_t *d_status, cudaStream_t st) {
    uint32_t blocks = (nq + 7) / 8;
    if (blocks == 0) blocks = 1;
    if (blocks > 65535) blocks = 65535;
    pack_kernel<<<blocks, 256, 0, st>>>(nq, d_q, d_off, d_words, d_status);
    return cudaGetLastError();
}

cudaError_t launch_order(uint32_t n, const uint64_t *d_off, uint32_t *d_order, cudaStream_t st) {
    order_kernel<<<1, 1024, 0, st>>>(n, d_off, d_order);
    return cudaGetLastError();
}

cudaError_t launch_slab_init(uint8_t *slabs, uint64_t slab_bytes, uint32_t n_slabs, uint32_t log2cap,
                             bool prune, cudaStream_t st) {
    const SlabLayout L = slab_layout(log2cap, prune);
    const uint64_t n16 = L.recs / 16 * n_slabs;
    if (n16 == 0) return cudaSuccess;
    uint64_t blocks = (n16 + 255) / 256;
    if (blocks > 8192) blocks = 8192;
    slab_init_kernel<<<(unsigned)blocks, 256, 0, st>>>(slabs, slab_bytes, n_slabs, L.recs);
    return cudaGetLastError();
}

// Load the alignment kernels into the context now.  With lazy module loading a
// kernel's code is loaded at its first launch, and that load can wait for kernels
// already running; an engine runs several of them side by side (its classes
// beside tier 0), so it touches them all before the first one starts.
cudaError_t preload_kernels() {
    cudaFuncAttributes fa;
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 6 && e == cudaSuccess; ++i)
        e = cudaFuncGetAttributes(&fa, align_entry(i % 3 > 0, i % 3 > 1, i < 3 ? kNarrow : 1024u));
    return e;
}

int align_occupancy(bool prune, uint32_t threads, int *blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, align_entry(prune, false, threads),
                                                         (int)threads, 0) == cudaSuccess ? 0 : -1;
}

}  // namespace gwfa

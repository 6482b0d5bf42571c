// Device-resident k-LPM scheduling path for sm_100a: flattened radix tree, batched longest-prefix
// match, k-LPM selection, schedule replay with LRU eviction.  See include/klpm.h for the ABI.
//
// Layout in HBM
//   nodes   : structure of arrays indexed by node id (0 = root): parent, depth_start, span_len, nchild
//             (int32), span_off, last_access (int64), dead (uint8).  Ids are never reused.
//   pool    : append-only int32 token pool; node v's edge label is pool[span_off[v] .. +span_len[v]).
//             Edges are placed so that span_off = depth_start (mod 4): the pool tokens that pair with
//             query positions 4i..4i+3 are one aligned 128-bit load.  A split never moves tokens, so
//             "pool index of the last matched token" identifies a position in the tree for as long as
//             the tree lives, and the pieces of a leaf that was cut stay one contiguous run
//             (chain_end in the child table, end_node[] per pool token: see walk_chain).
//   children: one open-addressing hash table for the whole tree keyed by (parent id, first token of the
//             child's edge).  An entry is one 32-byte sector and carries what a walk needs for the hop
//             (child id, edge length, edge offset, end of its contiguous run), so a hop costs one
//             dependent sector read.
//   LRU     : last_access holds logical clocks.  Only the node where a processed prompt's cached part
//             ends and its new leaf are stamped; when a leaf is evicted its stamp is handed to its
//             parent if newer.  For every leaf this equals the clock of the last processed prompt
//             whose path covers it, which is all eviction looks at.  clock_owner[c] names the node
//             holding stamp c, so the least recently used leaf is found by a cursor that only moves
//             forward over clock values.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <atomic>
#include <new>

#include "klpm.h"

#define FULL_MASK 0xffffffffu
#define KLPM_ABI_VERSION 3

namespace {

struct alignas(32) Entry {
    unsigned long long key;   // ((parent + 1) << 32) | first token ; 0 = empty slot
    int32_t child;            // node id, or -1 if the child was evicted (slot is reused on re-insert)
    int32_t span_len;
    int64_t span_off;
    int64_t chain_end;        // pool index one past the contiguous pool run this edge is part of (see walk_chain)
};

struct TreeState {
    long long n_nodes;      // next free node id
    long long pool_used;
    long long tokens_live;
    long long live_nodes;   // root excluded
    long long clock;
    long long lru_cursor;
    long long evictions;
    int status;
    int detail;             // which check recorded the status (a debugging aid, see rt_status_detail)
};

struct TreeDev {
    int32_t* parent;
    int32_t* depth_start;
    int32_t* span_len;
    int32_t* nchild;
    int32_t* first_tok;       // first token of the node's edge (= pool[span_off])
    int64_t* span_off;
    int64_t* last_access;
    uint8_t* dead;
    int32_t* clock_owner;
    Entry* table;
    unsigned long long table_mask;
    int32_t* pool;
    int32_t* end_node;        // per pool index: id of the node whose edge ends with that token, else -1
    TreeState* st;
    long long max_nodes, max_pool, max_clock, budget;
};

// ------------------------------------------------------------------------------------------------
// loads: RO = the kernel never writes what it reads (read-only path), otherwise L2-coherent loads
// ------------------------------------------------------------------------------------------------
template <bool RO> __device__ __forceinline__ int32_t ld32(const int32_t* p) { return RO ? __ldg(p) : __ldcg(p); }
template <bool RO> __device__ __forceinline__ Entry ld_entry(const Entry* e) {
    const int4* p = reinterpret_cast<const int4*>(e);
    int4 a = RO ? __ldg(p) : __ldcg(p);
    int4 b = RO ? __ldg(p + 1) : __ldcg(p + 1);
    Entry r;
    r.key = ((unsigned long long)(unsigned)a.y << 32) | (unsigned)a.x;
    r.child = a.z;
    r.span_len = a.w;
    r.span_off = (int64_t)(((unsigned long long)(unsigned)b.y << 32) | (unsigned)b.x);
    r.chain_end = (int64_t)(((unsigned long long)(unsigned)b.w << 32) | (unsigned)b.z);
    return r;
}

__device__ __forceinline__ unsigned long long make_key(int32_t parent, int32_t tok) {
    return ((unsigned long long)(unsigned)(parent + 1) << 32) | (unsigned)tok;
}
// Table hash: the two key halves are combined with the golden-ratio multiplier and run through the
// 32-bit finaliser of MurmurHash3 (public domain, A. Appleby).  32-bit arithmetic keeps a hop cheap.
__device__ __forceinline__ unsigned long long hash_key(unsigned long long k) {
    unsigned h = (unsigned)(k >> 32) * 0x9E3779B1u + (unsigned)k;
    h ^= h >> 16; h *= 0x85ebca6bu; h ^= h >> 13; h *= 0xc2b2ae35u; h ^= h >> 16;
    return (unsigned long long)h;
}

__device__ __forceinline__ void set_status(TreeState* st, int code, int detail = 0) {
    if (atomicCAS(&st->status, 0, code) == 0) st->detail = detail;
}

// A child lookup that probed every slot of the table without meeting the key or an empty slot gives up; the
// walk then reports a shorter match, and the status word says that it is not to be trusted.
__device__ __noinline__ void probe_limit(TreeState* st) {       // (a pointer: a reference to T would put the kernel's copy of it on the stack)
    if ((threadIdx.x & 31) == 0) set_status(st, RT_ERR_LIMIT, 106);
}

// First index in [0, n) where a and b differ, or n.  Warp-cooperative: every lane gets the result.
// Lane l reads elements l, l+32, l+64, ... of each chunk: each load instruction of the warp is one
// contiguous 128-byte request, whatever the 4-byte phase of the two streams.  U * 128 tokens of both
// streams are requested before the first of them is examined, so a long common prefix costs one memory
// latency per U * 128 tokens.
template <bool RO, int U = 4>
__device__ __forceinline__ int32_t first_mismatch(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int32_t n) {
    const int lane = threadIdx.x & 31;
    constexpr int R = 4 * U;
    for (int32_t base = 0; base < n; base += 32 * R) {
        int32_t x[R], y[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            int32_t idx = base + j * 32 + lane;
            bool in = idx < n;
            x[j] = in ? ld32<RO>(a + idx) : 0;
            y[j] = in ? ld32<RO>(b + idx) : 0;
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
            if (base + j * 32 >= n) break;                  // warp-uniform
            unsigned bad = __ballot_sync(FULL_MASK, x[j] != y[j]);
            if (bad) return base + j * 32 + (__ffs(bad) - 1);
        }
    }
    return n;
}

struct Term {
    int32_t m;      // matched tokens
    int32_t node;   // node whose edge holds the last matched token (0 = root)
    int32_t off;    // tokens of that edge matched
    int64_t pos;    // pool index of the last matched token, -1 at the root
    int32_t full;   // 1 if the match ends exactly at the end of that node's edge (or at the root)
};

// Longest prefix of q on a root path.  Warp-cooperative and warp-uniform.  (cur0, m0): a node boundary the walk may
// start from instead of the root -- the first m0 tokens of q are known to end exactly at the end of cur0's edge.
template <bool RO>
__device__ Term walk(const TreeDev& T, const int32_t* __restrict__ q, int32_t len, int32_t cur0 = 0, int32_t m0 = 0) {
    Term t; t.m = m0; t.node = cur0; t.off = 0; t.pos = -1; t.full = 1;
    if (len <= m0) return t;
    unsigned long long key = make_key(cur0, ld32<RO>(q + m0));
    unsigned long long slot = hash_key(key) & T.table_mask;
    Entry c = ld_entry<RO>(T.table + slot);
    for (;;) {
        unsigned long long probes = 0;
        while (c.key != key) {
            if (c.key == 0ULL) return t;
            if (++probes > T.table_mask) { probe_limit(T.st); return t; }      // no empty slot: cannot happen below load 1
            slot = (slot + 1) & T.table_mask;
            c = ld_entry<RO>(T.table + slot);
        }
        if (c.child < 0) return t;
        const int32_t rem = len - t.m;
        const int32_t n = c.span_len < rem ? c.span_len : rem;
        const bool has_next = c.span_len < rem;
        // issue the probe of the next hop before comparing this edge: it depends only on this entry
        unsigned long long key2 = 0, slot2 = 0;
        Entry nx; nx.key = 0; nx.child = -1; nx.span_len = 0; nx.span_off = 0; nx.chain_end = 0;
        if (has_next) {
            key2 = make_key(c.child, ld32<RO>(q + t.m + c.span_len));
            slot2 = hash_key(key2) & T.table_mask;
            nx = ld_entry<RO>(T.table + slot2);
        }
        const int32_t i = first_mismatch<RO>(q + t.m, T.pool + c.span_off, n);
        t.m += i;
        t.node = c.child;
        t.off = i;
        t.pos = c.span_off + i - 1;     // i >= 1: the first token is the key
        t.full = i == c.span_len;
        if (i < c.span_len || !has_next) return t;
        key = key2; slot = slot2; c = nx;
    }
}

// The walk of the read-only batched kernel on a tree that never evicts (no budget).
//
// A leaf's edge is written to the pool as one contiguous run, and later cuts only put node boundaries
// inside that run: the pieces stay adjacent, each the one child of the previous for the token that
// follows.  So a query that enters such a run at the start of a node matches exactly as far as it agrees
// with the contiguous pool tokens, whatever the number of boundaries it crosses; no child lookup is needed
// inside the run.  Every table entry carries chain_end, the pool index where its run ends, and
// end_node[] tells whether a pool token is the last one of a node: a lookup is only made where the
// comparison stops on a node boundary (another child may continue there) or the run is exhausted.
// The comparison itself is a stream: 128-bit loads of both sides, two 128-token chunks in flight.
//
// Coordinates are depths (token positions in the query).  Every edge is placed so that
// span_off = depth_start (mod 4), hence the pool tokens of depths 4i..4i+3 are one aligned 128-bit load.
// The query side is read with aligned 128-bit loads too and shifted across lanes when the query does not
// start on a 16-byte boundary.  The 16-byte units that hold the query's first and last token are read
// whole: the token buffer must be 16-byte aligned (as cudaMalloc'd memory is).
struct QWin {
    const int32_t* qa;   // q rounded down to 16 bytes
    int32_t s;           // tokens q is past that boundary (0..3)
    int32_t len;
};

// Query tokens are read once and never again: they are loaded with the streaming hint, so that the pool tokens --
// which other queries of the same trunk are about to read -- are what stays in L2.
__device__ __forceinline__ int4 ld_query4(const int4* p) { return __ldcs(p); }

// tokens of depths cb + 4 lane .. + 3 (cb a multiple of 4); zeros where nothing needs to be read
__device__ __forceinline__ int4 qwin_load(const QWin& Q, int32_t cb, int lane) {
    const int4 z = make_int4(0, 0, 0, 0);
    const int32_t p0 = cb + 4 * lane;
    int4 v = (p0 - Q.s < Q.len) ? ld_query4(reinterpret_cast<const int4*>(Q.qa + p0)) : z;
    if (Q.s == 0) return v;                                            // warp-uniform
    int4 e = (cb + 128 - Q.s < Q.len) ? ld_query4(reinterpret_cast<const int4*>(Q.qa + cb + 128)) : z;
    int4 n;
    n.x = __shfl_down_sync(FULL_MASK, v.x, 1); n.y = __shfl_down_sync(FULL_MASK, v.y, 1); n.z = __shfl_down_sync(FULL_MASK, v.z, 1);
    if (lane == 31) { n.x = e.x; n.y = e.y; n.z = e.z; }
    if (Q.s == 1) return make_int4(v.y, v.z, v.w, n.x);
    if (Q.s == 2) return make_int4(v.z, v.w, n.x, n.y);
    return make_int4(v.w, n.x, n.y, n.z);
}

// First depth >= lo of this 128-token chunk (lane l: depths p0 .. p0+3) where A and P differ, or -1.
__device__ __forceinline__ int32_t chunk_mismatch(const int4& A, const int4& P, int32_t p0, int32_t lo) {
    int32_t dx = P.x ^ A.x, dy = P.y ^ A.y, dz = P.z ^ A.z, dw = P.w ^ A.w;
    const int32_t hm = lo - p0;                     // leading tokens of this lane that are before lo
    if (hm > 0) dx = 0;
    if (hm > 1) dy = 0;
    if (hm > 2) dz = 0;
    const int32_t fc = dx ? 0 : dy ? 1 : dz ? 2 : dw ? 3 : 4;
    const unsigned bad = __ballot_sync(FULL_MASK, fc < 4);
    if (!bad) return -1;
    const int L = __ffs(bad) - 1;
    return __shfl_sync(FULL_MASK, p0 + fc, L);
}

// First depth in [lo, hi) where the query differs from pool_d[depth], or hi.  pool_d is the pool pointer
// shifted so that pool_d[p] pairs with depth p; it is 16-byte aligned.
#ifndef KLPM_PREFETCH_DIST
#define KLPM_PREFETCH_DIST 2
#endif
// One 128-token chunk with every bound checked: depths below lo and at or above hi take no part.  Returns the first
// depth where the two sides differ (hi at most), or -1.
__device__ __forceinline__ int32_t compare_chunk_edge(const QWin& Q, const int4* __restrict__ pool4, int32_t cb, int32_t lo, int32_t hi, int lane) {
    const int32_t p = cb + 4 * lane;
    const int4 A = qwin_load(Q, cb, lane);
    int4 P = A;
    if (p + 4 > lo && p < hi) P = __ldg(pool4 + (p >> 2));
    const int32_t r = chunk_mismatch(A, P, p, lo);
    if (r < 0) return -1;
    return r < hi ? r : hi;
}

// Both streams of the chunk KLPM_PREFETCH_DIST ahead are asked into L2 (no register waits for them), so that its
// loads find them there: a warp keeps more than one chunk of memory latency in flight.
__device__ __forceinline__ void prefetch_chunk(const QWin& Q, const int4* __restrict__ pool4, int32_t cb, int32_t hi, int lane) {
#if KLPM_PREFETCH_DIST > 0
    const int32_t pf = cb + 128 * KLPM_PREFETCH_DIST + 4 * lane;
    if (pf < hi) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pool4 + (pf >> 2)));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(Q.qa + pf));
    }
#endif
}

__device__ __forceinline__ int32_t compare_run(const QWin& Q, const int32_t* __restrict__ pool_d, int32_t lo, int32_t hi, int lane) {
    const int4* __restrict__ pool4 = reinterpret_cast<const int4*>(pool_d);
    const int4* __restrict__ qa4 = reinterpret_cast<const int4*>(Q.qa);
    int32_t cb = lo & ~127;
    // the chunk that holds lo
    prefetch_chunk(Q, pool4, cb, hi, lane);
    int32_t r = compare_chunk_edge(Q, pool4, cb, lo, hi, lane);
    if (r >= 0) return r;
    cb += 128;
    // chunks that lie wholly inside [lo, hi): nothing to mask, nothing to bound, and the exact position of a difference
    // is only worked out once a difference has been seen
    for (; cb + 128 <= hi; cb += 128) {
        prefetch_chunk(Q, pool4, cb, hi, lane);
        const int32_t i4 = (cb >> 2) + lane;
        int4 v = ld_query4(qa4 + i4);
        const int4 P = __ldg(pool4 + i4);
        if (Q.s != 0) {                                                    // warp-uniform
            const int4 e = ld_query4(qa4 + (cb >> 2) + 32);
            int32_t nx = __shfl_down_sync(FULL_MASK, v.x, 1), ny = __shfl_down_sync(FULL_MASK, v.y, 1), nz = __shfl_down_sync(FULL_MASK, v.z, 1);
            if (lane == 31) { nx = e.x; ny = e.y; nz = e.z; }
            if (Q.s == 1) v = make_int4(v.y, v.z, v.w, nx);
            else if (Q.s == 2) v = make_int4(v.z, v.w, nx, ny);
            else v = make_int4(v.w, nx, ny, nz);
        }
        const int32_t dx = v.x ^ P.x, dy = v.y ^ P.y, dz = v.z ^ P.z, dw = v.w ^ P.w;
        const unsigned bad = __ballot_sync(FULL_MASK, (dx | dy | dz | dw) != 0);
        if (bad) {
            const int32_t fc = dx ? 0 : dy ? 1 : dz ? 2 : 3;
            return __shfl_sync(FULL_MASK, cb + 4 * lane + fc, __ffs(bad) - 1);
        }
    }
    // the ragged end
    if (cb < hi) {
        r = compare_chunk_edge(Q, pool4, cb, lo, hi, lane);
        if (r >= 0) return r;
    }
    return hi;
}

// id of the live node whose edge ends with pool token `pos`, or -1.  Entries of end_node[] can be stale
// after a rollback, so a candidate is checked against the node arrays.
struct EndIndex {             // what is needed to resolve end_node[] entries, passed by value
    const int32_t* end_node; const int64_t* span_off; const int32_t* span_len; const uint8_t* dead;
    const TreeState* st;
};
__device__ __forceinline__ EndIndex end_index(const TreeDev& T) {
    EndIndex X; X.end_node = T.end_node; X.span_off = T.span_off; X.span_len = T.span_len; X.dead = T.dead; X.st = T.st;
    return X;
}
__device__ __forceinline__ int32_t node_ending_at(const EndIndex X, int64_t pos, long long n_nodes) {
    const int32_t e = __ldg(X.end_node + pos);
    if (e <= 0 || e >= n_nodes) return -1;
    if (__ldg(X.span_off + e) + __ldg(X.span_len + e) - 1 != pos || __ldg(X.dead + e)) return -1;
    return e;
}

// The node of this run whose edge ends first after pool token `pos` (the match stopped inside its edge).
__device__ __noinline__ int32_t node_after(const EndIndex X, int64_t pos, int64_t chain_end) {
    const int lane = threadIdx.x & 31;
    const long long n_nodes = *reinterpret_cast<const volatile long long*>(&X.st->n_nodes);
    for (int64_t p = pos + 1; p < chain_end; p += 32) {
        const int32_t cand = (p + lane < chain_end) ? node_ending_at(X, p + lane, n_nodes) : -1;
        const unsigned hit = __ballot_sync(FULL_MASK, cand >= 0);
        if (hit) return __shfl_sync(FULL_MASK, cand, __ffs(hit) - 1);
    }
    return -1;
}

// Returns the match length; *node / *off (where the match ended) are filled when want_node is set.
// With WANT_POS, *last_pos receives the pool index of the last matched token (-1 if nothing matched) and
// *last_end the end of the contiguous run that token lies in (what node_after needs to name the node later).
template <bool WANT_POS = false>
__device__ __forceinline__ int32_t walk_chain(const TreeDev& T, const int32_t* __restrict__ q, int32_t len, bool want_node,
                              int32_t* node, int32_t* off, int64_t* last_pos = nullptr, int64_t* last_end = nullptr) {
    const int lane = threadIdx.x & 31;
    *node = 0; *off = 0;
    if (WANT_POS) { *last_pos = -1; *last_end = 0; }
    if (len <= 0) return 0;
    QWin Q;
    Q.s = (int32_t)((reinterpret_cast<uintptr_t>(q) >> 2) & 3);
    Q.qa = q - Q.s;
    Q.len = len;
    int32_t m = 0, cur = 0;
    for (;;) {
        const unsigned long long key = make_key(cur, __ldg(q + m));
        unsigned long long slot = hash_key(key) & T.table_mask;
        Entry c = ld_entry<true>(T.table + slot);
        unsigned long long probes = 0;
        while (c.key != key) {
            if (c.key == 0ULL) return m;
            if (++probes > T.table_mask) { probe_limit(T.st); return m; }      // no empty slot: cannot happen below load 1
            slot = (slot + 1) & T.table_mask;
            c = ld_entry<true>(T.table + slot);
        }
        if (c.child < 0) return m;
        int64_t run = c.chain_end - c.span_off;
        if (run > (int64_t)(len - m)) run = len - m;
        const int32_t x = compare_run(Q, T.pool + (c.span_off - (int64_t)m), m, m + (int32_t)run, lane);
        const int64_t pos = c.span_off + (x - m) - 1;          // x > m: the first token is the key
        m = x;
        if (WANT_POS) { *last_pos = pos; *last_end = c.chain_end; }
        const int32_t e = node_ending_at(end_index(T), pos, *reinterpret_cast<const volatile long long*>(&T.st->n_nodes));
        if (e < 0) {                                           // stopped inside an edge
            if (want_node) {
                const int32_t f = node_after(end_index(T), pos, c.chain_end);
                if (f >= 0) { *node = f; *off = m - __ldg(T.depth_start + f); }
            }
            return m;
        }
        if (want_node) { *node = e; *off = __ldg(T.span_len + e); }
        if (m >= len) return m;
        cur = e;
    }
}

// ------------------------------------------------------------------------------------------------
// single-thread tree updates (callers serialise them)
// ------------------------------------------------------------------------------------------------
__device__ long long table_find(const TreeDev& T, int32_t parent, int32_t tok) {
    unsigned long long key = make_key(parent, tok);
    unsigned long long slot = hash_key(key) & T.table_mask;
    for (unsigned long long probes = 0; probes <= T.table_mask; ++probes) {
        unsigned long long k = __ldcg(&T.table[slot].key);
        if (k == key) return (long long)slot;
        if (k == 0ULL) return -1;
        slot = (slot + 1) & T.table_mask;
    }
    return -1;
}

__device__ bool table_put(const TreeDev& T, int32_t parent, int32_t tok, int32_t child, int32_t span_len, int64_t span_off,
                          int64_t chain_end) {
    unsigned long long key = make_key(parent, tok);
    unsigned long long slot = hash_key(key) & T.table_mask;
    for (unsigned long long probes = 0; probes <= T.table_mask; ++probes) {
        unsigned long long k = __ldcg(&T.table[slot].key);
        if (k == key || k == 0ULL) {
            Entry* e = T.table + slot;
            e->child = child; e->span_len = span_len; e->span_off = span_off; e->chain_end = chain_end;
            e->key = key;
            return true;
        }
        slot = (slot + 1) & T.table_mask;
    }
    return false;
}

// What a caller has already read for an insertion, so that the serial part need not wait for memory again:
// the tokens that key the table operations and the keys seen in the slots those operations probe first.
struct InsertPre {
    int32_t xm, pt, ft;                       // x[m]; pool token just below the cut; first token of the cut edge
    unsigned long long k_leaf, k_low, k_par;  // keys seen in the first slots of (end, xm), (upper, pt), (parent, ft)
};

__device__ long long table_find_seen(const TreeDev& T, int32_t parent, int32_t tok, unsigned long long seen) {
    const unsigned long long key = make_key(parent, tok);
    if (seen == key) return (long long)(hash_key(key) & T.table_mask);
    return table_find(T, parent, tok);
}

// table_put that trusts `seen` for the first slot unless that slot is `taken` (written since it was read).
__device__ long long table_put_seen(const TreeDev& T, int32_t parent, int32_t tok, int32_t child, int32_t span_len, int64_t span_off,
                                   int64_t chain_end, unsigned long long seen, long long taken) {
    const unsigned long long key = make_key(parent, tok);
    unsigned long long slot = hash_key(key) & T.table_mask;
    bool first = (long long)slot != taken;
    for (unsigned long long probes = 0; probes <= T.table_mask; ++probes) {
        const unsigned long long k = first ? seen : __ldcg(&T.table[slot].key);
        first = false;
        if (k == key || k == 0ULL) {
            Entry* e = T.table + slot;
            e->child = child; e->span_len = span_len; e->span_off = span_off; e->chain_end = chain_end;
            e->key = key;
            return (long long)slot;
        }
        slot = (slot + 1) & T.table_mask;
    }
    return -1;
}

// Node boundary `o` tokens into v's edge (0 < o < span_len[v]): a new node takes the upper part and v's
// place under v's parent; v keeps the lower part, its children and its id.  Returns the new node;
// *low_slot receives the table slot that now holds (new node, first token of the lower part).
__device__ int32_t split_node(const TreeDev& T, int32_t v, int32_t o, const InsertPre* pre, long long* low_slot) {
    TreeState* S = T.st;
    int32_t u = (int32_t)S->n_nodes++;
    S->live_nodes++;
    int32_t par = T.parent[v], ds = T.depth_start[v], len = T.span_len[v];
    int64_t off = T.span_off[v];
    T.parent[u] = par; T.depth_start[u] = ds; T.span_off[u] = off; T.span_len[u] = o;
    T.nchild[u] = 1; T.dead[u] = 0; T.last_access[u] = T.last_access[v];
    const int32_t ft = pre ? pre->ft : __ldcg(T.pool + off);
    const int32_t pt = pre ? pre->pt : __ldcg(T.pool + off + o);
    T.first_tok[u] = ft; T.first_tok[v] = pt;
    const long long slot = pre ? table_find_seen(T, par, ft, pre->k_par) : table_find(T, par, ft);
    int64_t chain_end = off + len;
    if (slot >= 0) { T.table[slot].child = u; T.table[slot].span_len = o; chain_end = T.table[slot].chain_end; }
    else set_status(S, RT_ERR_LIMIT, 101);
    T.span_off[v] = off + o; T.span_len[v] = len - o; T.depth_start[v] = ds + o; T.parent[v] = u;
    const long long ls = pre ? table_put_seen(T, u, pt, v, len - o, off + o, chain_end, pre->k_low, -1)
                             : table_put_seen(T, u, pt, v, len - o, off + o, chain_end, 0ULL, (long long)(hash_key(make_key(u, pt)) & T.table_mask));
    if (ls < 0) set_status(S, RT_ERR_CAPACITY);
    *low_slot = ls;
    T.end_node[off + o - 1] = u;
    return u;
}

__device__ void evict_leaf(const TreeDev& T, int32_t v) {
    TreeState* S = T.st;
    int32_t P = T.parent[v];
    T.dead[v] = 1;
    long long slot = table_find(T, P, __ldcg(T.pool + T.span_off[v]));
    if (slot >= 0) T.table[slot].child = -1;
    T.nchild[P]--;
    S->tokens_live -= T.span_len[v];
    S->live_nodes--;
    S->evictions++;
    if (P != 0 && T.last_access[v] >= T.last_access[P]) {
        T.last_access[P] = T.last_access[v];
        T.clock_owner[T.last_access[v]] = P;
    }
}

struct InsertOut {
    int32_t leaf;      // id of the new leaf, -1 if the prompt was fully cached
    int32_t unc;       // tokens to copy into the pool
    int64_t leaf_off;  // pool offset of the new leaf's edge
    int32_t evicted;   // 1 if any leaf was evicted
    int32_t ok;        // 0 if the prompt could not be stored (status word says why)
};

// Store prompt x (|x| = len) whose cached part is m tokens long and ends in `hint` or an ancestor of it.
// Everything except copying the new leaf's tokens into the pool.  One thread.
__device__ void insert_serial(const TreeDev& T, const int32_t* x, int32_t len, int32_t m, int32_t hint, InsertOut* out,
                              const InsertPre* pre = nullptr) {
    TreeState* S = T.st;
    out->leaf = -1; out->unc = 0; out->leaf_off = 0; out->evicted = 0; out->ok = 0;
    if (S->clock + 1 >= T.max_clock || S->n_nodes + 2 > T.max_nodes) { set_status(S, RT_ERR_CAPACITY); return; }
    const long long clock = ++S->clock;
    int32_t a = hint;
    while (a != 0 && m <= T.depth_start[a]) a = T.parent[a];
    const int32_t o = a == 0 ? 0 : m - T.depth_start[a];
    int32_t end = a;
    long long low_slot = -1;
    if (a != 0 && o < T.span_len[a]) end = split_node(T, a, o, pre, &low_slot);
    if (end != 0) { T.last_access[end] = clock; T.clock_owner[clock] = end; }
    const int32_t unc = len - m;
    if (T.budget > 0) {
        while (S->tokens_live + unc > T.budget) {
            long long cur = S->lru_cursor;
            int32_t victim = -1;
            while (cur < clock) {
                int32_t v = T.clock_owner[cur];
                if (v > 0 && !T.dead[v] && T.last_access[v] == cur && T.nchild[v] == 0) { victim = v; break; }
                ++cur;
            }
            S->lru_cursor = cur;
            if (victim < 0) { set_status(S, RT_ERR_BUDGET); return; }
            evict_leaf(T, victim);
            out->evicted = 1;
        }
    }
    if (unc > 0) {
        if (S->pool_used + unc + 6 > T.max_pool) { set_status(S, RT_ERR_CAPACITY); return; }
        int32_t leaf = (int32_t)S->n_nodes++;
        const int64_t off = ((S->pool_used + 3) & ~3LL) + (m & 3);    // span_off = depth_start (mod 4)
        S->pool_used = off + unc;
        T.parent[leaf] = end; T.depth_start[leaf] = m; T.span_off[leaf] = off; T.span_len[leaf] = unc;
        T.nchild[leaf] = 0; T.dead[leaf] = 0; T.last_access[leaf] = clock;
        T.clock_owner[clock] = leaf;
        T.nchild[end]++;
        const int32_t xm = pre ? pre->xm : __ldcg(x + m);
        T.first_tok[leaf] = xm;
        const long long put = pre ? table_put_seen(T, end, xm, leaf, unc, off, off + unc, pre->k_leaf, low_slot)
                                  : (table_put(T, end, xm, leaf, unc, off, off + unc) ? 0 : -1);
        if (put < 0) { set_status(S, RT_ERR_CAPACITY); return; }
        T.end_node[off + unc - 1] = leaf;
        S->tokens_live += unc;
        S->live_nodes++;
        out->leaf = leaf; out->unc = unc; out->leaf_off = off;
    }
    out->ok = 1;
}

// ------------------------------------------------------------------------------------------------
// rt_match_batch
// ------------------------------------------------------------------------------------------------
#ifndef KLPM_MATCH_MIN_BLOCKS
#define KLPM_MATCH_MIN_BLOCKS 8
#endif
// One warp per query, queries handed out by an atomic counter (persistent grid).
// Trees without a budget: stream along contiguous pool runs.
//
// Queries are taken in the order of `perm`: the host buckets them by their first token first, so that queries which
// start down the same root child -- and therefore read the same pool tokens -- are in flight at the same time and all
// but the first of them find those tokens in L2.
//
// With STATE the kernel also records, per query, what the scheduling loop needs to start from this match instead
// of walking the query again (MatchState: where the match ended, the run that position lies in, the next token).
struct alignas(32) MatchState {
    long long pos;        // pool index of the last matched token, -1 if nothing matched
    long long chain_end;  // end of the contiguous pool run `pos` lies in (trees with a budget: the node `pos` lies in)
    int32_t m;            // match length
    int32_t ntok;         // the query token right after the match (0 if the whole query matched)
    unsigned long long tag;   // which match call wrote this record
};
static_assert(sizeof(MatchState) == sizeof(klpm_match_state), "klpm_match_state is the ABI's view of MatchState");

template <bool STATE>
__global__ void __launch_bounds__(256, KLPM_MATCH_MIN_BLOCKS)
match_chain_kernel(TreeDev T, const int32_t* __restrict__ qtok, const int64_t* __restrict__ qoff, int32_t nq,
                   const int32_t* __restrict__ perm, int32_t* __restrict__ mlen, int32_t* __restrict__ tnode,
                   int32_t* __restrict__ toff, MatchState* __restrict__ state, unsigned long long tag,
                   unsigned long long* counter) {
    const int lane = threadIdx.x & 31;
    const bool want_node = tnode != nullptr || toff != nullptr;
    for (;;) {
        unsigned long long c = 0;
        if (lane == 0) c = atomicAdd(counter, 1ULL);
        c = __shfl_sync(FULL_MASK, c, 0);
        if (c >= (unsigned long long)nq) return;
        const int64_t i = __ldg(perm + c);
        const int64_t lo = __ldg(qoff + i);
        int64_t len = __ldg(qoff + i + 1) - lo;
        if (len < 0 || len > 0x7fffffffLL) { if (lane == 0) set_status(T.st, RT_ERR_INVALID); len = 0; }
        int32_t node, off;
        int64_t pos = -1, cend = 0;
        const int32_t m = STATE ? walk_chain<true>(T, qtok + lo, (int32_t)len, want_node, &node, &off, &pos, &cend)
                                : walk_chain<false>(T, qtok + lo, (int32_t)len, want_node, &node, &off);
        if (lane == 0) {
            if (mlen) mlen[i] = m;
            if (tnode) tnode[i] = node;
            if (toff) toff[i] = off;
            if (STATE) {
                const int32_t ntok = m < (int32_t)len ? __ldg(qtok + lo + m) : 0;
                int4* dst = reinterpret_cast<int4*>(state + i);
                __stcg(dst, make_int4((int)(unsigned)(unsigned long long)pos, (int)(unsigned)((unsigned long long)pos >> 32),
                                      (int)(unsigned)(unsigned long long)cend, (int)(unsigned)((unsigned long long)cend >> 32)));
                __stcg(dst + 1, make_int4(m, ntok, (int)(unsigned)tag, (int)(unsigned)(tag >> 32)));
            }
        }
    }
}

// The order in which the batched match takes the queries: bucketed by first token (counting sort over a hash of
// it; the order inside a bucket is whatever the atomics give -- results do not depend on it).  One addition per warp and
// bucket: where a few system prompts start every query, one per query took 40 us per kernel for 65,536 queries, now 6.
#define KLPM_ORDER_BUCKETS 8192
__device__ __forceinline__ unsigned order_bucket(const int32_t* __restrict__ qtok, const int64_t* __restrict__ qoff, int32_t i) {
    const int64_t lo = __ldg(qoff + i);
    if (__ldg(qoff + i + 1) <= lo) return 0u;
    unsigned h = (unsigned)__ldg(qtok + lo) * 0x9E3779B1u;
    return h >> 19;                                         // 13 bits: KLPM_ORDER_BUCKETS
}
__global__ void order_hist_kernel(const int32_t* __restrict__ qtok, const int64_t* __restrict__ qoff, int32_t nq,
                                  unsigned* __restrict__ hist, unsigned short* __restrict__ bucket) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned b = i < nq ? order_bucket(qtok, qoff, i) : 0xffffffffu;
    const unsigned same = __match_any_sync(FULL_MASK, b);
    if (i >= nq) return;
    bucket[i] = (unsigned short)b;
    if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(hist + b, (unsigned)__popc(same));
}
// hist[b] <- number of queries in buckets below b (one CTA of 1,024 threads, 8 buckets each)
__global__ void __launch_bounds__(1024) order_scan_kernel(unsigned* hist) {
    __shared__ unsigned s_w[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int PER = KLPM_ORDER_BUCKETS / 1024;
    unsigned v[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { v[j] = hist[tid * PER + j]; sum += v[j]; }
    unsigned inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const unsigned o = __shfl_up_sync(FULL_MASK, inc, d); if (lane >= d) inc += o; }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        unsigned w = s_w[lane], wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const unsigned o = __shfl_up_sync(FULL_MASK, wi, d); if (lane >= d) wi += o; }
        s_w[lane] = wi - w;
    }
    __syncthreads();
    unsigned run = s_w[warp] + inc - sum;
#pragma unroll
    for (int j = 0; j < PER; ++j) { hist[tid * PER + j] = run; run += v[j]; }
}
__global__ void order_scatter_kernel(const unsigned short* __restrict__ bucket, int32_t nq, unsigned* __restrict__ cursor,
                                     int32_t* __restrict__ perm) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const unsigned b = i < nq ? (unsigned)bucket[i] : 0xffffffffu;
    const unsigned same = __match_any_sync(FULL_MASK, b);
    const int lead = __ffs(same) - 1;
    unsigned at = 0;
    if (i < nq && lane == lead) at = atomicAdd(cursor + b, (unsigned)__popc(same));
    at = __shfl_sync(FULL_MASK, at, lead) + (unsigned)__popc(same & ((1u << lane) - 1u));
    if (i < nq) perm[at] = i;
}

// Trees with a budget (evicted children break the runs): hop by hop.
__global__ void __launch_bounds__(256)
match_batch_kernel(TreeDev T, const int32_t* __restrict__ qtok, const int64_t* __restrict__ qoff, int32_t nq,
                   const int32_t* __restrict__ perm, int32_t* __restrict__ mlen, int32_t* __restrict__ tnode,
                   int32_t* __restrict__ toff, MatchState* __restrict__ state, unsigned long long tag,
                   unsigned long long* counter) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned long long c = 0;
        if (lane == 0) c = atomicAdd(counter, 1ULL);
        c = __shfl_sync(FULL_MASK, c, 0);
        if (c >= (unsigned long long)nq) return;
        const int64_t i = __ldg(perm + c);
        const int64_t lo = __ldg(qoff + i), hi = __ldg(qoff + i + 1);
        int64_t len = hi - lo;
        if (len < 0 || len > 0x7fffffffLL) { if (lane == 0) set_status(T.st, RT_ERR_INVALID); len = 0; }
        Term t = walk<true>(T, qtok + lo, (int32_t)len);
        if (lane == 0) {
            if (mlen) mlen[i] = t.m;
            if (tnode) tnode[i] = t.node;
            if (toff) toff[i] = t.off;
            if (state) {
                MatchState r;
                // trees with a budget have no use for the run's end; the field carries the node the match ended in instead
                r.pos = t.pos; r.chain_end = t.node; r.m = t.m; r.ntok = t.m < (int32_t)len ? __ldg(qtok + lo + t.m) : 0; r.tag = tag;
                state[i] = r;
            }
        }
    }
}

// The batched match for few queries: one CTA per query, every warp of it walks (redundantly: the lookups are
// broadcasts) and compares its own 512 tokens of the stretch at hand, so a long edge costs one memory latency per
// 512 x warps tokens instead of one per 512 (match_batch_kernel) or 128 (match_chain_kernel).  With few queries that
// latency is all there is: no batch order, no work counter to clear, the grid is the batch.  CHAIN: streams along
// contiguous pool runs (trees without a budget), otherwise hop by hop.
// 32 queries of 1,024 to 8,192 tokens, caches cold: 10 us (match_batch_kernel 21), on a tree without a budget 12 us
// (match_chain_kernel 33).
// With `in_order` (1: the first part of a call, 2: a later one) the batch is about to be inserted one prompt after the other, which ends at
// the first prompt that is not one (a negative length, or more tokens than an int32 counts): nothing from there on is
// looked at, here either.  The insertion itself reports it.
__device__ __forceinline__ int32_t wide_mismatch(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int32_t n,
                                                 int32_t* s_min, unsigned& phase) {
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (nwarps == 1) return first_mismatch<true>(a, b, n);
    for (int32_t base = 0; base < n; base += nwarps * 512) {     // (n is the same in every thread of the CTA)
        const int32_t lo = base + warp * 512;
        const unsigned p = phase % 3u, q = (phase + 1u) % 3u;    // three words in turn: the next one is reset a barrier ahead
        ++phase;
        if (lo < n) {
            const int32_t seg = n - lo < 512 ? n - lo : 512;
            const int32_t r = first_mismatch<true>(a + lo, b + lo, seg);
            if (r < seg && (threadIdx.x & 31) == 0) atomicMin(s_min + p, lo + r);
        }
        if (threadIdx.x == 0) s_min[q] = 0x7fffffff;
        __syncthreads();
        const int32_t m = s_min[p];
        if (m != 0x7fffffff) return m;
    }
    return n;
}

template <bool CHAIN>
__global__ void __launch_bounds__(256, 4)
match_wide_kernel(TreeDev T, const int32_t* __restrict__ qtok, const int64_t* __restrict__ qoff, int32_t* __restrict__ mlen,
                  int32_t* __restrict__ tnode, int32_t* __restrict__ toff, MatchState* __restrict__ state, unsigned long long tag,
                  int32_t in_order, const int32_t* stop) {
    __shared__ int32_t s_min[3];
    if (threadIdx.x < 3) s_min[threadIdx.x] = 0x7fffffff;
    const int64_t i = blockIdx.x;
    const int64_t lo = __ldg(qoff + i), hi = __ldg(qoff + i + 1);
    bool bad = false;
    if (in_order) {
        bad = in_order == 2 && *stop != 0;
        for (int64_t j = threadIdx.x; j <= i; j += blockDim.x) {
            const int64_t l = __ldg(qoff + j + 1) - __ldg(qoff + j);
            bad = bad || l < 0 || l > 0x7fffffffLL;
        }
    }
    if (__syncthreads_or(bad)) return;
    unsigned phase = 0;
    int64_t len64 = hi - lo;
    if (len64 < 0 || len64 > 0x7fffffffLL) { if (threadIdx.x == 0) set_status(T.st, RT_ERR_INVALID); len64 = 0; }
    const int32_t len = (int32_t)len64;
    const int32_t* q = qtok + lo;
    const EndIndex X = end_index(T);
    const long long n_nodes = CHAIN ? *reinterpret_cast<const volatile long long*>(&T.st->n_nodes) : 0;
    int32_t m = 0, cur = 0, node = 0, off = 0;
    int64_t pos = -1, cend = 0;
    while (m < len) {
        const unsigned long long key = make_key(cur, __ldg(q + m));
        unsigned long long slot = hash_key(key) & T.table_mask;
        Entry c = ld_entry<true>(T.table + slot);
        unsigned long long probes = 0;
        bool found = true;
        while (c.key != key) {
            if (c.key == 0ULL) { found = false; break; }
            if (++probes > T.table_mask) { probe_limit(T.st); found = false; break; }      // no empty slot: cannot happen below load 1
            slot = (slot + 1) & T.table_mask;
            c = ld_entry<true>(T.table + slot);
        }
        if (!found || c.child < 0) break;
        int64_t run = CHAIN ? c.chain_end - c.span_off : (int64_t)c.span_len;
        if (run > (int64_t)(len - m)) run = len - m;
        const int32_t x = wide_mismatch(q + m, T.pool + c.span_off, (int32_t)run, s_min, phase);     // x >= 1: the first token is the key
        if (x <= 0) { probe_limit(T.st); break; }                 // (an entry that does not lead to its token: cannot happen)
        m += x;
        pos = c.span_off + x - 1;
        if (CHAIN) {
            cend = c.chain_end;
            const int32_t e = node_ending_at(X, pos, n_nodes);
            if (e < 0) {                                          // stopped inside an edge
                if (tnode || toff) {
                    const int32_t f = node_after(X, pos, cend);
                    if (f >= 0) { node = f; off = m - __ldg(T.depth_start + f); }
                }
                break;
            }
            node = e;
            if (tnode || toff) off = __ldg(T.span_len + e);
            cur = e;
        } else {
            node = c.child; off = x; cend = c.child;              // (trees with a budget: the record carries the node)
            if (x < c.span_len) break;
            cur = c.child;
        }
    }
    if (threadIdx.x == 0) {
        if (mlen) mlen[i] = m;
        if (tnode) tnode[i] = node;
        if (toff) toff[i] = off;
        if (state) {
            MatchState r;
            r.pos = pos; r.chain_end = cend; r.m = m; r.ntok = m < len ? __ldg(q + m) : 0; r.tag = tag;
            state[i] = r;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// sequential processing of prompts by one CTA: rt_insert and klpm_replay (its plain form, debug setting run_one_by_one)
// ------------------------------------------------------------------------------------------------
struct SeqArgs {
    const int32_t* tok; const int64_t* off; const int64_t* arrival; const int32_t* order;
    int32_t n;                       // prompts to process
    int32_t n_queries;               // prompts in the CSR arrays: entries of `order` must be below this
    long long c_num, c_den, start_tick;
    int32_t* uncached; int64_t* ttft; int64_t* completion;   // indexed by query
};

__global__ void __launch_bounds__(1024)
sequential_kernel(TreeDev T, SeqArgs A) {
    __shared__ Term s_term;
    __shared__ InsertOut s_out;
    long long now = A.start_tick;
    for (int32_t k = 0; k < A.n; ++k) {
        const int32_t j = A.order ? __ldg(A.order + k) : k;
        if (j < 0 || j >= A.n_queries) {           // not a query: nothing of it is read or written (uniform over the CTA)
            if (threadIdx.x == 0) set_status(T.st, RT_ERR_INVALID, 108);
            return;
        }
        const int64_t lo = __ldg(A.off + j), hi = __ldg(A.off + j + 1);
        if (hi < lo || hi - lo > 0x7fffffffLL) {
            if (threadIdx.x == 0) set_status(T.st, RT_ERR_INVALID, 108);
            return;
        }
        const int32_t len = (int32_t)(hi - lo);
        const int32_t* x = A.tok + lo;
        if (threadIdx.x < 32) {
            Term t = walk<false>(T, x, len);
            if (threadIdx.x == 0) {
                s_term = t;
                insert_serial(T, x, len, t.m, t.node, &s_out);
                if (s_out.ok) {
                    int32_t unc = len - t.m;
                    if (A.uncached) {
                        long long tj = __ldg(A.arrival + j);
                        long long begin = now > tj ? now : tj;
                        long long R = begin + (A.c_den + A.c_num * (long long)len) * (long long)unc;
                        A.uncached[j] = unc; A.ttft[j] = R - tj;
                        if (A.completion) A.completion[j] = R;
                        now = R;
                    }
                }
            }
        }
        __syncthreads();
        if (!s_out.ok) return;
        const int32_t unc = s_out.unc, m = s_term.m;
        int32_t* dst = T.pool + s_out.leaf_off;
        for (int32_t i = threadIdx.x; i < unc; i += blockDim.x) dst[i] = __ldg(x + m + i);
        __threadfence();
        __syncthreads();
    }
}

// rt_insert one prompt after the other (a budget, or per-prompt results asked for).  Every prompt has been matched against
// the tree as it was before the call (pm, pnode: match length, node), all of them at once; warp 0 then goes through the
// prompts.  The match as it is now follows from that one without comparing its tokens again: walk up from the node while
// it has been cut above the match or evicted (an evicted node takes its tokens along), and look for a child only where
// the match ends on a node boundary.  The insertion is insert_serial with the warp's lanes side by side: the three hash
// probes at once, 32 clock values per look for the least recently used leaf (kept in registers from prompt to prompt, as
// in lru_tree_warp).  The other warps copy a prompt's new tokens while warp 0 is at the next one.
// What bounds it: the chain of L2 round trips per prompt.  16 prompts into a full cache: 57 us (3.5 us a prompt;
// one thread that walked from the root, probed and scanned the clock one value at a time took 131).
// A long call is cut into parts of KLPM_INSERT_PART prompts, so that the matches fit memory the tree has had from the start and
// the call allocates nothing; a part that ends early says so to the ones behind it (*stop).
#define KLPM_INSERT_PART 1024
struct InsertArgs { const int32_t* tok; const int64_t* off; int32_t n; int32_t* new_tokens; const int32_t* pm; const int32_t* pnode; int32_t* stop; int32_t first; };

__device__ __forceinline__ long long probe_for(const TreeDev& T, unsigned long long key, bool find, Entry* e, long long not_this) {
    unsigned long long slot = hash_key(key) & T.table_mask;
    for (unsigned long long probes = 0; probes <= T.table_mask; ++probes) {
        *e = ld_entry<false>(T.table + slot);
        if ((long long)slot != not_this) {
            if (e->key == key) return (long long)slot;
            if (e->key == 0ULL) return find ? -1 : (long long)slot;
        }
        slot = (slot + 1) & T.table_mask;
    }
    return -1;
}

__global__ void __launch_bounds__(512)
insert_seq_kernel(TreeDev T, InsertArgs A) {
    __shared__ long long s_dst; __shared__ int32_t s_m, s_unc, s_ok, s_bad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!A.first && __ldcg(A.stop)) return;                 // (uniform over the CTA)
    TreeState st = *T.st;
    long long wbase = st.lru_cursor, wend = wbase;          // the window of clock values (see lru_tree_warp)
    int32_t wv = 0;
    bool wok = false;
    if (threadIdx.x == 0) { s_ok = 1; s_bad = 0; }
    __syncthreads();
    for (int32_t k = 0; k < A.n; ++k) {
        const int64_t lo = __ldg(A.off + k), hi = __ldg(A.off + k + 1);
        if (hi < lo || hi - lo > 0x7fffffffLL) {            // (uniform over the CTA)
            if (threadIdx.x == 0) { set_status(T.st, RT_ERR_INVALID, 108); s_bad = 1; }
            break;
        }
        const int32_t len = (int32_t)(hi - lo);
        const int32_t* x = A.tok + lo;
        int32_t m = 0, a = 0;
        if (warp == 0) {
            m = __ldcg(A.pm + k); a = __ldcg(A.pnode + k);
            while (a != 0) {
                const int32_t ds = T.depth_start[a];
                if (T.dead[a]) { if (ds < m) m = ds; }
                else if (m > ds) break;
                a = T.parent[a];
            }
        }
        __syncthreads();                                    // the tokens of the prompt before are in the pool
        if (warp == 0) {
            int32_t ds = T.depth_start[a], sl = T.span_len[a];
            int32_t o = a == 0 ? 0 : m - ds;
            if (a == 0 || o == sl) {                        // on a node boundary: another child may continue there now
                const Term t = walk<false>(T, x, len, a, m);
                if (t.m > m) { m = t.m; a = t.node; ds = T.depth_start[a]; sl = T.span_len[a]; o = m - ds; }
            }
            const int32_t unc = len - m;
            bool ok = true;
            long long dst = 0;
            int32_t copy = 0;
            if (st.clock + 1 >= T.max_clock || st.n_nodes + 2 > T.max_nodes) { if (lane == 0) set_status(T.st, RT_ERR_CAPACITY); ok = false; }
            else {
                const long long clock = ++st.clock;
                const bool cut = a != 0 && o < sl;
                const int32_t par = T.parent[a];
                const long long so = T.span_off[a], la = T.last_access[a];
                const int32_t u = (int32_t)st.n_nodes;
                const int32_t end = cut ? u : a;
                int32_t ft = 0, pt = 0, xm = 0;
                if (cut) { ft = __ldcg(T.pool + so); pt = __ldcg(T.pool + so + o); }
                if (unc > 0) xm = __ldg(x + m);
                // lane 0: the entry of the edge that is cut; lane 1: where its lower part goes; lane 2: where the leaf goes
                Entry e; e.key = 0; e.child = 0; e.span_len = 0; e.span_off = 0; e.chain_end = 0;
                const unsigned long long key = lane == 0 ? make_key(par, ft) : lane == 1 ? make_key(u, pt) : make_key(end, xm);
                long long slot = -1;
                if ((lane < 2 && cut) || (lane == 2 && unc > 0)) slot = probe_for(T, key, lane == 0, &e, -1);
                __syncwarp();
                const long long s1 = __shfl_sync(FULL_MASK, slot, 1), s2 = __shfl_sync(FULL_MASK, slot, 2);
                if (lane == 2 && cut && unc > 0 && s1 == s2 && s1 >= 0) slot = probe_for(T, key, false, &e, s1);
                __syncwarp();
                if (cut) {
                    ++st.n_nodes; ++st.live_nodes;
                    const long long ce = __shfl_sync(FULL_MASK, slot >= 0 ? (long long)e.chain_end : (long long)(so + sl), 0);
                    if (lane == 0) {
                        if (slot >= 0) { T.table[slot].child = u; T.table[slot].span_len = o; }
                        else set_status(T.st, RT_ERR_LIMIT, 101);
                        T.parent[u] = par; T.depth_start[u] = ds; T.span_off[u] = so; T.span_len[u] = o;
                        T.nchild[u] = 1; T.dead[u] = 0; T.last_access[u] = la; T.first_tok[u] = ft; T.first_tok[a] = pt;
                        T.span_off[a] = so + o; T.span_len[a] = sl - o; T.depth_start[a] = ds + o; T.parent[a] = u;
                        T.end_node[so + o - 1] = u;
                    }
                    if (lane == 1) {
                        if (slot >= 0) {
                            Entry* d = T.table + slot;
                            d->child = a; d->span_len = sl - o; d->span_off = so + o; d->chain_end = ce; d->key = key;
                        } else set_status(T.st, RT_ERR_CAPACITY);
                    }
                }
                if (end != 0 && lane == 0) { T.last_access[end] = clock; T.clock_owner[clock] = end; }
                if (wv == end) wok = false;
                __syncwarp();
                while (T.budget > 0 && st.tokens_live + unc > T.budget) {
                    unsigned okm = __ballot_sync(FULL_MASK, wok);
                    while (!okm && wend < clock) {          // the next 32 clock values
                        wbase = wend;
                        const long long cc = wbase + lane;
                        wv = cc < clock ? T.clock_owner[cc] : 0;
                        wend = wbase + 32 < clock ? wbase + 32 : clock;
                        wok = wv > 0 && wv != end && !T.dead[wv] && T.last_access[wv] == cc && T.nchild[wv] == 0;
                        okm = __ballot_sync(FULL_MASK, wok);
                    }
                    if (!okm) { if (lane == 0) set_status(T.st, RT_ERR_BUDGET); ok = false; break; }
                    const int src = __ffs(okm) - 1;
                    const int32_t v = __shfl_sync(FULL_MASK, wv, src);
                    const long long stamp = wbase + src;
                    const int32_t P = T.parent[v], vl = T.span_len[v], vt = T.first_tok[v];
                    Entry ve;
                    const long long vs = probe_for(T, make_key(P, vt), true, &ve, -1);
                    const int32_t nc = T.nchild[P] - 1;
                    long long pl = T.last_access[P];
                    __syncwarp();
                    const bool hand = P != 0 && stamp >= pl;
                    if (hand) pl = stamp;
                    if (lane == 0) {
                        T.dead[v] = 1;
                        if (vs >= 0) T.table[vs].child = -1;
                        T.nchild[P] = nc;
                        if (hand) { T.last_access[P] = stamp; T.clock_owner[stamp] = P; }
                    }
                    if (lane == src) wok = false;
                    if (nc == 0 && P != 0 && P != end && pl >= wbase && pl < wend && lane == (int)(pl - wbase)) { wv = P; wok = true; }
                    st.tokens_live -= vl; --st.live_nodes; ++st.evictions;
                    __syncwarp();
                }
                if (ok && unc > 0) {
                    const long long ls = __shfl_sync(FULL_MASK, slot, 2);
                    if (st.pool_used + unc + 6 > T.max_pool || ls < 0) { if (lane == 0) set_status(T.st, RT_ERR_CAPACITY); ok = false; }
                    else {
                        const int32_t leaf = (int32_t)st.n_nodes++;
                        const long long off = ((st.pool_used + 3) & ~3LL) + (m & 3);      // span_off = depth_start (mod 4)
                        st.pool_used = off + unc;
                        ++st.live_nodes; st.tokens_live += unc;
                        if (lane == 2) {
                            Entry* d = T.table + slot;
                            d->child = leaf; d->span_len = unc; d->span_off = off; d->chain_end = off + unc; d->key = key;
                        }
                        if (lane == 0) {
                            T.parent[leaf] = end; T.depth_start[leaf] = m; T.span_off[leaf] = off; T.span_len[leaf] = unc;
                            T.nchild[leaf] = 0; T.dead[leaf] = 0; T.last_access[leaf] = clock; T.first_tok[leaf] = xm;
                            T.clock_owner[clock] = leaf;
                            T.nchild[end] = T.nchild[end] + 1;
                            T.end_node[off + unc - 1] = leaf;
                        }
                        dst = off; copy = unc;
                    }
                }
                if (ok && A.new_tokens && lane == 0) A.new_tokens[k] = unc;
            }
            __syncwarp();
            if (lane == 0) { s_dst = dst; s_m = m; s_unc = copy; s_ok = ok ? 1 : 0; }
        }
        __syncthreads();
        if (!s_ok) break;
        if (warp > 0) {
            int32_t* d = T.pool + s_dst;
            const int32_t mm = s_m, cnt = s_unc;
            for (int32_t i = threadIdx.x - 32; i < cnt; i += blockDim.x - 32) d[i] = __ldg(x + mm + i);
        }
    }
    if (threadIdx.x == 0) {                                 // the counters go back (a status recorded meanwhile stays)
        TreeState* S = T.st;
        S->n_nodes = st.n_nodes; S->pool_used = st.pool_used; S->tokens_live = st.tokens_live; S->live_nodes = st.live_nodes;
        S->clock = st.clock; S->lru_cursor = wbase; S->evictions = st.evictions;
        *A.stop = s_bad || !s_ok;
    }
}

// ------------------------------------------------------------------------------------------------
// klpm_select: one decision as a pure function
// ------------------------------------------------------------------------------------------------
struct Cand { int32_t m; int32_t idx; long long t; };   // idx < 0 = none

__device__ __forceinline__ bool better_lpm(const Cand& a, const Cand& b) {      // a beats b
    if (b.idx < 0) return a.idx >= 0;
    if (a.idx < 0) return false;
    if (a.m != b.m) return a.m > b.m;
    if (a.t != b.t) return a.t < b.t;
    return a.idx < b.idx;
}
__device__ __forceinline__ bool better_fcfs(const Cand& a, const Cand& b) {
    if (b.idx < 0) return a.idx >= 0;
    if (a.idx < 0) return false;
    if (a.t != b.t) return a.t < b.t;
    return a.idx < b.idx;
}
template <bool LPM> __device__ __forceinline__ Cand cand_best(Cand a, Cand b) {
    return (LPM ? better_lpm(b, a) : better_fcfs(b, a)) ? b : a;
}
template <bool LPM> __device__ __forceinline__ Cand warp_best(Cand c) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        Cand o;
        o.m = __shfl_xor_sync(FULL_MASK, c.m, d);
        o.idx = __shfl_xor_sync(FULL_MASK, c.idx, d);
        o.t = __shfl_xor_sync(FULL_MASK, c.t, d);
        c = cand_best<LPM>(c, o);
    }
    return c;
}
template <bool LPM> __device__ Cand block_best(Cand c, Cand* smem /*32*/) {
    c = warp_best<LPM>(c);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if (lane == 0) smem[w] = c;
    __syncthreads();
    Cand r; r.m = 0; r.idx = -1; r.t = 0;
    if (w == 0) {
        if (lane < nw) r = smem[lane];
        r = warp_best<LPM>(r);
    }
    return r;   // valid in warp 0
}

// Queues of up to KLPM_SELECT_SMALL: one CTA, eight queries per thread held in registers, the kk best one after the
// other.  A pick is four hardware reductions per warp (match, the two halves of the arrival, index), one barrier, and
// the same over the warps' winners, which every warp does for itself.  No scratch in global memory, no ticket.
// 4,001 queries (warm): the 3 best 7.3 us (select_topk_kernel 17.4, one pass over the queue per pick), one pick 7 (8.2);
// 32 queries, one pick 2.4 us (4.4).  At the line, 8,192 queries, calls back to back: one pick 6.2 us (10.6), the 3 best 8.6 (18.9),
// the 64 best 99 (255).  Longer queues do not fit the registers of one CTA; they are spread over CTAs.
#define KLPM_SELECT_SMALL 8192
struct PickKey { unsigned m, th, tl, idx; };      // match and arrival in a form that orders as unsigned; idx = 0xffffffff: none
__device__ __forceinline__ PickKey warp_pick(const PickKey k) {
    PickKey r;
    bool in = k.idx != 0xffffffffu;
    r.m = __reduce_max_sync(FULL_MASK, in ? k.m : 0u);
    in = in && k.m == r.m;
    r.th = __reduce_min_sync(FULL_MASK, in ? k.th : 0xffffffffu);
    in = in && k.th == r.th;
    r.tl = __reduce_min_sync(FULL_MASK, in ? k.tl : 0xffffffffu);
    in = in && k.tl == r.tl;
    r.idx = __reduce_min_sync(FULL_MASK, in ? k.idx : 0xffffffffu);
    return r;
}

template <bool LPM>
__global__ void __launch_bounds__(1024)
select_small_kernel(const int32_t* __restrict__ mlen, const int64_t* __restrict__ arrival, const uint8_t* __restrict__ waiting,
                    int32_t nq, int32_t kk, int32_t* __restrict__ out) {
    __shared__ PickKey s_k[2][32];
    constexpr int PER = KLPM_SELECT_SMALL / 1024;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarps = nthr >> 5;
    unsigned m[PER], th[PER], tl[PER], alive = 0;
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        const int32_t i = r * nthr + tid;
        m[r] = 0; th[r] = 0; tl[r] = 0;
        if (i < nq) {
            const unsigned long long t = (unsigned long long)__ldg(arrival + i) ^ 0x8000000000000000ULL;
            th[r] = (unsigned)(t >> 32); tl[r] = (unsigned)t;
            if (LPM) m[r] = (unsigned)__ldg(mlen + i) ^ 0x80000000u;
            if (__ldg(waiting + i)) alive |= 1u << r;
        }
    }
    for (int j = 0; j < kk; ++j) {
        PickKey best; best.m = 0; best.th = 0; best.tl = 0; best.idx = 0xffffffffu;
#pragma unroll
        for (int r = 0; r < PER; ++r) {                      // (ascending index: an equal one does not replace)
            const bool better = best.idx == 0xffffffffu || m[r] > best.m ||
                                (m[r] == best.m && (th[r] < best.th || (th[r] == best.th && tl[r] < best.tl)));
            if (((alive >> r) & 1u) && better) { best.m = m[r]; best.th = th[r]; best.tl = tl[r]; best.idx = (unsigned)(r * nthr + tid); }
        }
        best = warp_pick(best);
        if (nwarps > 1) {                                    // (two buffers in turn: one barrier per pick)
            if (lane == 0) s_k[j & 1][warp] = best;
            __syncthreads();
            best.idx = 0xffffffffu;
            if (lane < nwarps) best = s_k[j & 1][lane];
            best = warp_pick(best);
        }
        if (tid == 0) out[j] = (int32_t)best.idx;            // (none: -1)
        if (best.idx != 0xffffffffu && best.idx % (unsigned)nthr == (unsigned)tid) alive &= ~(1u << (best.idx / (unsigned)nthr));
    }
}

struct SelectScratch { Cand partial[1024]; unsigned int ticket; };

template <bool LPM>
__global__ void __launch_bounds__(512)
select_kernel(const int32_t* __restrict__ mlen, const int64_t* __restrict__ arrival, const uint8_t* __restrict__ waiting,
              int32_t nq, int32_t* pick, SelectScratch* sc) {
    __shared__ Cand s_c[32];
    __shared__ bool s_last;
    Cand best; best.m = 0; best.idx = -1; best.t = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nq; i += (int64_t)gridDim.x * blockDim.x) {
        if (__ldg(waiting + i)) {
            Cand c; c.m = LPM ? __ldg(mlen + i) : 0; c.idx = (int32_t)i; c.t = __ldg(arrival + i);
            best = cand_best<LPM>(best, c);
        }
    }
    best = block_best<LPM>(best, s_c);
    if (threadIdx.x == 0) {
        sc->partial[blockIdx.x] = best;
        __threadfence();
        unsigned t = atomicAdd(&sc->ticket, 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    Cand c; c.m = 0; c.idx = -1; c.t = 0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
        Cand o;
        o.m = __ldcg(&sc->partial[b].m); o.idx = __ldcg(&sc->partial[b].idx); o.t = __ldcg(&sc->partial[b].t);
        c = cand_best<LPM>(c, o);
    }
    __syncthreads();
    c = block_best<LPM>(c, s_c);
    if (threadIdx.x == 0) { *pick = c.idx; sc->ticket = 0; }
}

// ------------------------------------------------------------------------------------------------
// klpm_select_topk: the kk best longest-match candidates of one queue snapshot, best first.
// The j-th best is the best element strictly worse than the (j-1)-th in the total order
// (match desc, arrival asc, index asc), so no element is ever marked as taken: each CTA extracts its own
// kk best by kk passes over its slice, and the last CTA to finish merges the per-CTA lists the same way.
// ------------------------------------------------------------------------------------------------
#define KLPM_TOPK_MAX 64
#define KLPM_TOPK_BLOCKS 128
struct TopkScratch { Cand cand[KLPM_TOPK_BLOCKS * KLPM_TOPK_MAX]; unsigned int ticket; };

__global__ void __launch_bounds__(512)
select_topk_kernel(const int32_t* __restrict__ mlen, const int64_t* __restrict__ arrival, const uint8_t* __restrict__ waiting,
                   int32_t nq, int32_t kk, int32_t* out, TopkScratch* sc) {
    __shared__ Cand s_c[32];
    __shared__ Cand s_prev;
    __shared__ bool s_last;
    Cand prev; prev.m = 0; prev.idx = -1; prev.t = 0;          // idx < 0: no bound yet
    for (int j = 0; j < kk; ++j) {
        Cand best; best.m = 0; best.idx = -1; best.t = 0;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nq; i += (int64_t)gridDim.x * blockDim.x) {
            if (__ldg(waiting + i)) {
                Cand c; c.m = __ldg(mlen + i); c.idx = (int32_t)i; c.t = __ldg(arrival + i);
                if (prev.idx < 0 || better_lpm(prev, c)) best = cand_best<true>(best, c);
            }
        }
        best = block_best<true>(best, s_c);
        if (threadIdx.x == 0) { s_prev = best; sc->cand[blockIdx.x * KLPM_TOPK_MAX + j] = best; }
        __syncthreads();
        prev = s_prev;
        __syncthreads();
        if (prev.idx < 0) {                                     // slice exhausted: pad the rest
            if (threadIdx.x == 0) for (int r = j + 1; r < kk; ++r) sc->cand[blockIdx.x * KLPM_TOPK_MAX + r] = prev;
            break;
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    prev.m = 0; prev.idx = -1; prev.t = 0;
    bool done = false;
    for (int j = 0; j < kk; ++j) {
        Cand best; best.m = 0; best.idx = -1; best.t = 0;
        if (!done) {
            for (int e = threadIdx.x; e < (int)gridDim.x * kk; e += blockDim.x) {
                const Cand* src = &sc->cand[(e / kk) * KLPM_TOPK_MAX + (e % kk)];
                Cand c; c.m = __ldcg(&src->m); c.idx = __ldcg(&src->idx); c.t = __ldcg(&src->t);
                if (c.idx >= 0 && (prev.idx < 0 || better_lpm(prev, c))) best = cand_best<true>(best, c);
            }
        }
        __syncthreads();
        best = block_best<true>(best, s_c);
        if (threadIdx.x == 0) { s_prev = best; out[j] = best.idx; }
        __syncthreads();
        if (s_prev.idx < 0) done = true; else prev = s_prev;
        __syncthreads();
    }
    if (threadIdx.x == 0) sc->ticket = 0;
}

// ------------------------------------------------------------------------------------------------
// klpm_select_noalloc: the same decision as klpm_select, with the per-CTA partial results kept in a
// fixed array that is part of the library image instead of memory obtained from cudaMalloc.
// ------------------------------------------------------------------------------------------------
#define KLPM_SELECT_NOALLOC_BLOCKS 256
struct StaticSelectScratch { Cand partial[KLPM_SELECT_NOALLOC_BLOCKS]; unsigned int ticket; };
// 4 KiB + one counter per GPU that loads the library, held until the process exits.
static __device__ __align__(256) unsigned char g_select_static[sizeof(StaticSelectScratch)];

template <bool LPM>
__global__ void __launch_bounds__(512)
select_static_kernel(const int32_t* __restrict__ mlen, const int64_t* __restrict__ arrival, const uint8_t* __restrict__ waiting,
                     int32_t nq, int32_t* pick, StaticSelectScratch* sc) {
    __shared__ Cand s_c[32];
    __shared__ bool s_last;
    Cand best; best.m = 0; best.idx = -1; best.t = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nq; i += (int64_t)gridDim.x * blockDim.x) {
        if (__ldg(waiting + i)) {
            Cand c; c.m = LPM ? __ldg(mlen + i) : 0; c.idx = (int32_t)i; c.t = __ldg(arrival + i);
            best = cand_best<LPM>(best, c);
        }
    }
    best = block_best<LPM>(best, s_c);
    if (threadIdx.x == 0) {
        sc->partial[blockIdx.x] = best;
        __threadfence();
        s_last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    Cand c; c.m = 0; c.idx = -1; c.t = 0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
        Cand o;
        o.m = __ldcg(&sc->partial[b].m); o.idx = __ldcg(&sc->partial[b].idx); o.t = __ldcg(&sc->partial[b].t);
        c = cand_best<LPM>(c, o);
    }
    __syncthreads();
    c = block_best<LPM>(c, s_c);
    if (threadIdx.x == 0) *pick = c.idx;
}

// ------------------------------------------------------------------------------------------------
// klpm_run, one decision at a time on the tree itself: the whole loop as one cooperative kernel.
// Trees with a budget take this loop (eviction can shorten matches, so match lengths are kept against
// the tree as it changes); trees without one take the grouped loop further down.
//
// Slots are the queries ordered by (arrival, index).  Per decision c:
//   phase A (every CTA): bring the match state of the waiting slots up to date -- walk newly arrived
//     queries, drop queries out of evicted leaves, extend the queries that were tied with the prompt
//     processed last into its new leaf -- and reduce the keys (match << 32 | ~slot) to one per CTA;
//   phase B (CTA 0): pick (oldest waiting slot or largest key), charge by Definition 2, store the prompt.
// The two phases hand over through two monotone counters in global memory (`arrive`: CTAs that finished
// phase A; `seq`: decisions completed), and what phase A needs to know about the last decision travels
// in one broadcast record.  While the kernel runs only CTA 0 mutates the tree; it keeps the tree's
// counters in shared memory and writes them back at the end.
// ------------------------------------------------------------------------------------------------
struct RunBcast {
    long long now;            // completion time of the last processed query
    long long head;           // first slot not yet processed
    long long admitted;       // slots < admitted have a match state
    long long last_pos;       // position (pool index of last matched token) of the last processed prompt, before it was stored
    long long last_leaf_off;  // pool offset of the leaf it appended
    int32_t evicted;          // the last decision evicted something
    int32_t last_valid;       // the last decision appended a leaf
    int32_t last_q, last_m, last_len, last_leaf;
    int32_t abort;
    int32_t last_xm;          // first uncached token of the last processed prompt
};
struct RunSync { unsigned long long arrive; unsigned long long seq; };

struct RunArgs {
    const int32_t* tok; const int64_t* off; const int64_t* arrival;
    int32_t n;
    int32_t policy, k;
    long long c_num, c_den, start_tick;
    int32_t* order; int32_t* uncached; int64_t* ttft; int64_t* completion;
    // scratch (library-owned)
    int32_t* ord;          // slot -> query index, by (arrival, index)
    long long* sorted_t;   // slot -> arrival
    long long* soff;       // slot -> offset of the query's first token
    int32_t* slen;         // slot -> query length
    int32_t* m;            // slot -> current match length; -1 once processed
    int32_t* hint;         // slot -> node at or below the node where the match ends
    long long* pos;        // slot -> pool index of the last matched token (-1 = root)
    int32_t* ntok;         // slot -> the query token right after its match (meaningful while m < length)
    const int32_t* prank;  // slot -> rank of the slot by (tie priority, slot); null = ties go to the lower slot
    const int32_t* pinv;   // that rank -> slot
    int32_t score_mode;    // 0: score = match length; 1: score = floor(match * 2^31 / length)
    unsigned long long* partial;   // per CTA best key
    RunBcast* bc;
    RunSync* sy;
    long long wait_limit_ns;       // limit of every hand-over wait
};

#define KLPM_RUN_THREADS 512
#define KLPM_RUN_SLOTS 4          // slots per thread whose state is loaded together
#ifndef KLPM_RUN_SPT
#define KLPM_RUN_SPT 2            // slots per scanner thread the grid is sized for
#endif
#define KLPM_WAIT_LIMIT_NS 5000000000LL      // default limit of a hand-over wait: 5 s on the device's nanosecond timer

// Thread 0 of the CTA polls *p until it reaches target, then the CTA learns whether to go on.  The wait is
// bounded: after limit_ns (checked every 4,096 polls; a limit of 0 gives up at the first poll that fails) the
// status word gets RT_ERR_LIMIT, every CTA is told to leave, and this one returns false.
__device__ bool run_wait(volatile unsigned long long* p, unsigned long long target, RunBcast* bc, TreeState* st, long long limit_ns) {
    __shared__ int s_go;
    if (threadIdx.x == 0) {
        int go = 1;
        unsigned long long spins = 0, t0 = 0;
        while (*p < target) {
            if ((++spins & 4095ULL) == 0 || limit_ns == 0) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                if (limit_ns == 0 || now - t0 > (unsigned long long)limit_ns || spins > (1ULL << 40)) {
                    set_status(st, RT_ERR_LIMIT, 102); *(volatile int32_t*)&bc->abort = 1; go = 0; break;
                }
            }
        }
        __threadfence();
        if (*(volatile int32_t*)&bc->abort) go = 0;
        s_go = go;
    }
    __syncthreads();
    const bool go = s_go != 0;
    __syncthreads();
    return go;
}

// Time at which the next pick is made and the number of slots that have arrived by then (one thread).
// Everything below `admitted` has arrived already, so the search gallops from there.
__device__ void run_bound(const RunArgs& A, const RunBcast& b, long long* adm_new, long long* now_out) {
    long long now = b.now;
    if (b.head >= b.admitted && b.head < A.n) {   // nobody waiting: idle until the next arrival
        const long long th = __ldg(A.sorted_t + b.head);
        if (th > now) now = th;
    }
    long long lo = b.admitted > b.head ? b.admitted : b.head, hi = A.n;
    if (lo < hi && __ldg(A.sorted_t + lo) <= now) {
        long long step = 1;
        ++lo;
        while (lo + step <= hi && __ldg(A.sorted_t + lo + step - 1) <= now) { lo += step; step <<= 1; }
        if (lo + step < hi) hi = lo + step;
        while (lo < hi) { const long long mid = (lo + hi) >> 1; if (__ldg(A.sorted_t + mid) <= now) lo = mid + 1; else hi = mid; }
    }
    *adm_new = lo; *now_out = now;
}

// Phase A for one CTA of the `nscan` scanning CTAs: returns (in warp lanes) this thread's best key.
__device__ unsigned long long run_scan(const TreeDev& T, const RunArgs& A, const RunBcast& bc, long long adm_new,
                                       unsigned scan_id, unsigned nscan) {
    const int lane = threadIdx.x & 31;
    const long long TT = (long long)nscan * blockDim.x;
    const long long gtid = (long long)scan_id * blockDim.x + threadIdx.x;
    const long long head = bc.head, admitted = bc.admitted;
    const int evicted = bc.evicted, last_valid = bc.last_valid;
    const int32_t last_m = bc.last_m, last_len = bc.last_len, last_leaf = bc.last_leaf;
    const long long last_pos = bc.last_pos, last_leaf_off = bc.last_leaf_off;
    const int32_t last_xm = bc.last_xm;
    const int32_t* last_x = last_valid ? A.tok + __ldg(A.off + bc.last_q) : nullptr;
    unsigned long long best = 0;
    for (long long base = (head / TT) * TT; base < adm_new; base += TT * KLPM_RUN_SLOTS) {
        int32_t mm[KLPM_RUN_SLOTS], nn[KLPM_RUN_SLOTS];
        long long pp[KLPM_RUN_SLOTS];
#pragma unroll
        for (int u = 0; u < KLPM_RUN_SLOTS; ++u) {
            const long long r = base + u * TT + gtid;
            const bool have = r >= head && r < admitted && r < adm_new;
            mm[u] = have ? __ldcg(A.m + r) : -1;
            pp[u] = have ? __ldcg(A.pos + r) : -1;
            nn[u] = have ? __ldcg(A.ntok + r) : 0;
        }
#pragma unroll
        for (int u = 0; u < KLPM_RUN_SLOTS; ++u) {
            if (base + u * TT >= adm_new) break;                               // warp-uniform
            const long long r = base + u * TT + gtid;
            const bool fresh = r >= head && r >= admitted && r < adm_new;
            int32_t m = mm[u], hint = 0, ntok = nn[u];
            long long pos = pp[u];
            bool dirty = false;
            unsigned wm = __ballot_sync(FULL_MASK, fresh);
            if (wm) {                                  // newly arrived queries: full walk, one warp each
                const int32_t* q = nullptr; int32_t qlen = 0;
                if (fresh) { qlen = __ldg(A.slen + r); q = A.tok + __ldg(A.soff + r); }
                while (wm) {
                    const int src = __ffs(wm) - 1; wm &= wm - 1;
                    const int32_t* qq = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)q, src);
                    const int32_t ql = __shfl_sync(FULL_MASK, qlen, src);
                    Term t = walk<false>(T, qq, ql);
                    if (lane == src) { m = t.m; hint = t.node; pos = t.pos; ntok = t.m < ql ? __ldg(qq + t.m) : 0; dirty = true; }
                }
            }
            const bool waiting = fresh || m >= 0;
            if (waiting && !fresh && evicted) {        // drop out of evicted leaves
                hint = __ldcg(A.hint + r);
                int32_t a = hint;
                const int32_t m0 = m;
                while (a != 0) {
                    const bool dead = __ldcg(T.dead + a) != 0;
                    const int32_t ds = __ldcg(T.depth_start + a);
                    if (dead) { if (ds < m) m = ds; }
                    else if (m > ds) break;
                    a = __ldcg(T.parent + a);
                }
                if (a != hint || m != m0) {
                    hint = a;
                    pos = a == 0 ? -1 : __ldcg(T.span_off + a) + (m - __ldcg(T.depth_start + a)) - 1;
                    if (m != m0) ntok = m < __ldg(A.slen + r) ? __ldg(A.tok + __ldg(A.soff + r) + m) : 0;
                    dirty = true;
                } else {
                    hint = -1;                          // unchanged: do not rewrite
                }
            }
            // tied with the prompt processed last: it may now match into that prompt's new leaf
            bool cmp = false;
            const int32_t* q = nullptr; int32_t qlen = 0;
            if (waiting && !fresh && last_valid && pos == last_pos && m == last_m && ntok == last_xm) {
                qlen = __ldg(A.slen + r);
                q = A.tok + __ldg(A.soff + r);
                cmp = m < qlen;
            }
            unsigned cm = __ballot_sync(FULL_MASK, cmp);
            while (cm) {
                const int src = __ffs(cm) - 1; cm &= cm - 1;
                const int32_t* qq = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)q, src);
                const int32_t ql = __shfl_sync(FULL_MASK, qlen, src);
                const int32_t lim = (ql < last_len ? ql : last_len) - last_m;
                const int32_t e = first_mismatch<true>(qq + last_m, last_x + last_m, lim);
                if (lane == src) {
                    m = last_m + e; hint = last_leaf; pos = last_leaf_off + e - 1;
                    ntok = m < ql ? __ldg(qq + m) : 0;
                    dirty = true;
                }
            }
            if (waiting) {
                if (dirty) { A.m[r] = m; A.pos[r] = pos; A.ntok[r] = ntok; if (hint >= 0) A.hint[r] = hint; }
                unsigned hi = (unsigned)m;
                if (A.score_mode == 1) {
                    const int32_t ql = __ldg(A.slen + r);
                    hi = ql > 0 ? (unsigned)(((unsigned long long)(unsigned)m << 31) / (unsigned)ql) : 0u;
                }
                const unsigned lo = A.prank ? (unsigned)__ldg(A.prank + r) : (unsigned)r;
                const unsigned long long key = ((unsigned long long)hi << 32) | (0xffffffffu - lo);
                if (key > best) best = key;
            }
        }
    }
    return best;
}

__device__ __forceinline__ unsigned long long warp_max64(unsigned long long v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(FULL_MASK, v, d);
        if (o > v) v = o;
    }
    return v;
}

// CTA 0 is the sequencer (picks, charges, mutates the tree); CTAs 1..G-1 scan.  With a single CTA it does both.
// Without a budget, and when the next decision admits no new arrivals, the sequencer publishes its pick --
// including the id and pool offset its new leaf is going to get, which follow from the tree's counters --
// before it performs the insertion, so the scanners refresh the waiting queue for the next decision while
// the tree is being updated (they only read query tokens and their own slots' state then).
__global__ void __launch_bounds__(KLPM_RUN_THREADS)
run_kernel(TreeDev T, RunArgs A) {
    __shared__ unsigned long long s_red[KLPM_RUN_THREADS / 32];
    __shared__ long long s_bound[2];      // slots admitted by this decision, time at which the pick is made
    __shared__ InsertOut s_out;
    __shared__ int32_t s_j[2];            // match length and length of the picked prompt
    __shared__ const int32_t* s_x;
    __shared__ TreeState s_st;            // CTA 0: the tree's counters while the kernel runs
    __shared__ RunBcast s_bc;
    __shared__ int s_flag[2];             // CTA 0: publish-before-insert, predicted leaf
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned G = gridDim.x;
    const unsigned nscan = G > 1 ? G - 1 : 1;
    TreeState* const gst = T.st;

    if (blockIdx.x != 0) {
        // ------------------------------------------------------------ scanners
        for (long long c = 0; c < A.n; ++c) {
            if (!run_wait(&A.sy->seq, (unsigned long long)c, A.bc, gst, A.wait_limit_ns)) return;
            if (threadIdx.x == 0) {
                RunBcast b;
                const long long* src = reinterpret_cast<const long long*>(A.bc);
                long long* dst = reinterpret_cast<long long*>(&b);
#pragma unroll
                for (int i = 0; i < (int)(sizeof(RunBcast) / 8); ++i) dst[i] = __ldcg(src + i);
                s_bc = b;
                run_bound(A, b, &s_bound[0], &s_bound[1]);
            }
            __syncthreads();
            unsigned long long best = warp_max64(run_scan(T, A, s_bc, s_bound[0], blockIdx.x - 1, nscan));
            if (lane == 0) s_red[warp] = best;
            __syncthreads();
            if (threadIdx.x == 0) {
                unsigned long long b = 0;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) if (s_red[w] > b) b = s_red[w];
                A.partial[blockIdx.x - 1] = b;
                __threadfence();
                atomicAdd(&A.sy->arrive, 1ULL);
            }
        }
        return;
    }

    // ---------------------------------------------------------------- sequencer (CTA 0)
    TreeDev T0 = T;                        // its view of the tree: counters in shared memory
    T0.st = &s_st;
    if (threadIdx.x == 0) {
        s_st = *gst;
        RunBcast b;
        const long long* src = reinterpret_cast<const long long*>(A.bc);
        long long* dst = reinterpret_cast<long long*>(&b);
#pragma unroll
        for (int i = 0; i < (int)(sizeof(RunBcast) / 8); ++i) dst[i] = __ldcg(src + i);
        s_bc = b;
    }
    __syncthreads();
    bool ok = true;
    for (long long c = 0; c < A.n && ok; ++c) {
        if (threadIdx.x == 0) run_bound(A, s_bc, &s_bound[0], &s_bound[1]);
        __syncthreads();
        const long long head = s_bc.head, adm_new = s_bound[0];
        // The queries that arrive next will be walked from the root by a single warp while everybody waits: bring
        // their tokens into L2 now (slots are in arrival order, so these are known; a hint only).
        for (long long r = adm_new; r < adm_new + 2 && r < A.n; ++r) {
            const int32_t* q = A.tok + __ldg(A.soff + r);
            const int32_t qlen = __ldg(A.slen + r);
            for (int32_t i = threadIdx.x * 32; i < qlen; i += blockDim.x * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(q + i));
        }
        unsigned long long b = 0;
        if (G == 1) {
            unsigned long long best = warp_max64(run_scan(T, A, s_bc, adm_new, 0, 1));
            if (lane == 0) s_red[warp] = best;
            __syncthreads();
            if (warp == 0) b = warp_max64(lane < (int)(blockDim.x >> 5) ? s_red[lane] : 0ULL);
        } else {
            if (!run_wait(&A.sy->arrive, (unsigned long long)(c + 1) * nscan, A.bc, gst, A.wait_limit_ns)) { ok = false; break; }
            if (warp == 0) {
                for (unsigned g = lane; g < nscan; g += 32) { const unsigned long long o = __ldcg(A.partial + g); if (o > b) b = o; }
                b = warp_max64(b);
            }
        }
        // ---- pick (warp 0; lane 0 decides), charge by Definition 2
        if (warp == 0) {
            const bool fcfs_turn = A.policy == KLPM_POLICY_FCFS || (A.policy == KLPM_POLICY_KLPM && (c % A.k) == 0);
            long long slot = head;
            if (!fcfs_turn) {
                const unsigned rk = 0xffffffffu - (unsigned)(b & 0xffffffffu);
                slot = A.pinv ? (long long)__ldg(A.pinv + rk) : (long long)rk;
            }
            const int32_t qi = __ldg(A.ord + slot);
            const int32_t m = __ldcg(A.m + slot);
            const int32_t hint = __ldcg(A.hint + slot);
            const long long pos = __ldcg(A.pos + slot);
            const int32_t ntok = __ldcg(A.ntok + slot);
            const int32_t len = __ldg(A.slen + slot);
            const long long tj = __ldg(A.sorted_t + slot);
            const int32_t* x = A.tok + __ldg(A.soff + slot);
            // where the cached part ends, and what the insertion is going to allocate
            int32_t a = hint;
            int32_t a_ds = T.depth_start[a], a_sl = T.span_len[a], a_par = T.parent[a], a_ft = T.first_tok[a];   // side by side
            const int32_t below = __ldcg(T.pool + (pos + 1));       // the pool token under the cut, if there is a cut
            while (a != 0 && m <= a_ds) {
                a = a_par;
                a_ds = T.depth_start[a]; a_sl = T.span_len[a]; a_par = T.parent[a]; a_ft = T.first_tok[a];
            }
            const int32_t o = a == 0 ? 0 : m - a_ds;
            const bool mid = a != 0 && o < a_sl;
            const int32_t unc = len - m;
            const int32_t leaf_pred = unc > 0 ? (int32_t)s_st.n_nodes + (mid ? 1 : 0) : -1;
            const long long leaf_off_pred = unc > 0 ? ((s_st.pool_used + 3) & ~3LL) + (m & 3) : 0;
            // Three lanes read, side by side, what the serial insertion would otherwise wait for one after
            // the other: the tokens that key its table operations, then the first slot each will probe.
            // The reads are issued here and collected after the pick has been published.
            int32_t v = 0;
            if (lane == 0 && unc > 0) v = ntok;
            if (lane == 1 && mid) v = below;
            if (lane == 2 && mid) v = a_ft;
            unsigned long long seen = 0;
            {
                const int32_t end = mid ? (int32_t)s_st.n_nodes : a;
                unsigned long long key = 0;
                bool want = false;
                if (lane == 0) { key = make_key(end, v); want = unc > 0; }
                if (lane == 1) { key = make_key(end, v); want = mid; }
                if (lane == 2) { key = make_key(a_par, v); want = mid; }
                if (want) seen = __ldcg(&T.table[hash_key(key) & T.table_mask].key);
                for (int32_t i = lane * 32; i < unc; i += 32 * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + m + i));
            }
            if (lane == 0) {
                s_j[0] = m; s_j[1] = len; s_x = x;
                const long long now = s_bound[1];
                const long long begin = now > tj ? now : tj;
                const long long R = begin + (A.c_den + A.c_num * (long long)len) * (long long)unc;
                A.m[slot] = -1;
                long long h = head;
                if (slot == head) while (h < A.n && (h == slot || (h < adm_new && __ldcg(A.m + h) < 0))) ++h;
                RunBcast nb = s_bc;
                nb.head = h; nb.now = R; nb.admitted = adm_new;
                nb.evicted = 0;
                nb.last_valid = unc > 0; nb.last_q = qi; nb.last_m = m; nb.last_len = len;
                nb.last_leaf = leaf_pred; nb.last_pos = pos; nb.last_leaf_off = leaf_off_pred; nb.last_xm = ntok;
                s_bc = nb;
                // may the scanners start on the next decision while the tree is being updated?
                long long adm_next, now_next;
                run_bound(A, nb, &adm_next, &now_next);
                const int early = (G > 1 && T.budget == 0 && adm_next == adm_new && c + 1 < A.n) ? 1 : 0;
                s_flag[0] = early; s_flag[1] = leaf_pred;
                if (early) {
                    *A.bc = nb;
                    __threadfence();
                    atomicExch(&A.sy->seq, (unsigned long long)(c + 1));
                }
                A.order[c] = qi; A.uncached[qi] = unc; A.ttft[qi] = R - tj;
                if (A.completion) A.completion[qi] = R;
            }
            InsertPre pre;
            pre.xm = __shfl_sync(FULL_MASK, v, 0); pre.pt = __shfl_sync(FULL_MASK, v, 1); pre.ft = __shfl_sync(FULL_MASK, v, 2);
            pre.k_leaf = __shfl_sync(FULL_MASK, seen, 0); pre.k_low = __shfl_sync(FULL_MASK, seen, 1); pre.k_par = __shfl_sync(FULL_MASK, seen, 2);
            if (lane == 0) {
                insert_serial(T0, x, len, m, hint, &s_out, &pre);
                if (s_out.ok && (s_out.leaf != leaf_pred || (unc > 0 && s_out.leaf_off != leaf_off_pred))) {
                    set_status(&s_st, RT_ERR_LIMIT, 103);           // cannot happen: the prediction repeats the allocation rule
                    s_out.ok = 0;
                }
            }
        }
        __syncthreads();
        if (!s_out.ok) { ok = false; break; }
        {
            const int32_t unc = s_out.unc, m = s_j[0];
            const int32_t* x = s_x;
            int32_t* dst = T.pool + s_out.leaf_off;
            for (int32_t i = threadIdx.x; i < unc; i += blockDim.x) dst[i] = __ldg(x + m + i);
        }
        if (!s_flag[0]) __threadfence();       // published next: others may walk the tree (the early mode's readers never touch it)
        __syncthreads();
        if (threadIdx.x == 0 && !s_flag[0]) {
            s_bc.evicted = s_out.evicted;
            if (G > 1 && c + 1 < A.n) {
                *A.bc = s_bc;
                __threadfence();
                atomicExch(&A.sy->seq, (unsigned long long)(c + 1));
            }
        }
        __syncthreads();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int st_global = *(volatile int*)&gst->status;
        TreeState out = s_st;
        if (out.status == 0) { out.status = st_global; out.detail = *(volatile int*)&gst->detail; }
        *gst = out;
        if (!ok) *(volatile int32_t*)&A.bc->abort = 1;
        __threadfence();
        atomicExch(&A.sy->seq, (unsigned long long)A.n + 1);      // releases anybody still waiting
    }
}

// ------------------------------------------------------------------------------------------------
// klpm_run on a tree without a budget: the grouped loop.
//
// Without eviction the match length of a query only ever grows, and it grows exactly when a prompt is
// processed whose own match ended at the same tree position and continues with the same token
// (otherwise the processed prompt shares no more with the query than the tree already did).  So the loop
// needs no tree at all:
//   * every query -- arrived or not -- is matched once against the tree as it stands (one warp per query,
//     streaming along contiguous pool runs), which gives its match length m, the position `pos` where the
//     match ends (pool index of the last matched token) and the query token `ntok` that follows;
//   * queries with the same (pos, ntok) form a group, held as a contiguous run of a member array
//     (a bitonic sort by a 62-bit hash of the pair puts equal pairs side by side; a hash collision only
//     puts two groups into one run, and members are checked against (pos, ntok) before they are touched);
//   * when a prompt is processed its group is dissolved: every member is compared with the prompt's
//     uncached tokens, gets its new m, a position inside the prompt's new leaf and its next token, and the
//     members are regrouped by their new pairs inside the run they already occupy (they never need more
//     room: the processed query leaves).  A query in a group of one costs nothing.  Leaves created by the
//     loop get positions from a counter that starts above every real pool index;
//   * while arrivals are pending, the longest-match pick is the root of a tournament over the keys
//     (score << 32 | ~rank) of the arrived queries: 32-ary, leaves in global memory, every level above in shared
//     memory (fast_run_kernel); once everybody has arrived it is the next entry of a list of all keys sorted as they are
//     then, and the tournament only holds the queries whose key has changed since (list_run_kernel);
//   * the oldest-first pick is a cursor over a bitmap of processed slots.
// One CTA runs the whole loop: warp 0 is the sequencer, the other warps wait at a named barrier and join
// for work that is worth sharing (a large group, a large batch of arrivals).  There is no wait on another
// CTA anywhere.  The processed prompts are stored in the tree afterwards, all at once, by the concurrent
// bulk insertion: the set of node boundaries does not depend on the order of insertion.
// ------------------------------------------------------------------------------------------------
struct alignas(32) FDyn {     // what the loop changes, one 32-byte sector per slot
    long long pos;            // pool index (real or virtual) of the last matched token, -1 at the root
    int32_t m;                // match length; -1 once processed
    int32_t ntok;             // query token right after the match (meaningful while m < length)
    int32_t gstart, gcount;   // the slot's group: run [gstart, gstart + gcount) of the member array
    int32_t hint;             // trees with a budget: a node at or below the node the match ends in (walk up while m <= depth_start)
    int32_t pad;
};
struct alignas(32) FStat {    // constant during the loop; the first 16 bytes are all that charging a pick needs
    long long t;              // arrival
    int32_t len;
    int32_t ord;              // query index
    long long soff;           // offset of the query's first token
    int32_t rank;             // low key bits: rank by (tie priority, slot), or the slot itself
    int32_t pad;
};

// Trees with a budget: what the loop reads of a node, in one 32-byte sector (the tree's arrays are packed into these
// records before the loop and written back after it).  nchild < 0: evicted.
struct alignas(32) LNode { int32_t parent, depth, len, nchild; long long last, off; };

struct FastPost {
    int32_t c0; int32_t list_c;                 // first decision the charge pass after the loop charges (n: none, as after a loop that gave up); decisions made before everybody had arrived
    long long now0; int32_t head, cyc;          // the time then, the oldest unprocessed slot, decisions made mod k
    // what the loop did (rt_debug_counters): careful steps, dissolves by the whole CTA, fallback scans, slots that fell
    // back, evictions; cycles spent in tree updates, fallback scans, dissolves; list mode: windows, batches in which the two
    // orders agree and the decisions they made, batches worked out by iteration and the decisions they made, decisions
    // made one at a time; cycles spent on new windows and on decisions made one at a time
    long long counters[16];
};

struct FastArgs {
    const int32_t* tok;
    int32_t n;
    int32_t policy, k, score_mode;
    unsigned recip_k1;            // 2^32 / (k - 1) rounded up: x / (k - 1) = high half of x * recip_k1, exact while x (k - 1) < 2^32; 0 if k - 1 is 1 or larger than any x it is used for
    long long c_num, c_den, start_tick;
    int32_t* order; int32_t* uncached; int64_t* ttft; int64_t* completion;
    FDyn* dyn; FStat* stat;
    unsigned long long* key;      // slot -> key it has (or will have once arrived); 0 once processed
    int32_t* mem;                 // member array
    const long long* sorted_t;    // per slot: arrival, side by side
    int4* lcp;                    // per slot: how far its prompt agrees with a reference prompt (see lcp_kernel)
    int4* pair;                   // list mode, two per slot that starts in a group: of two, the other slot, its match length and key once this one is processed, then the same of this slot; else -2
    const int32_t* pinv;          // rank -> slot, or null
    long long* gh; int32_t* gidx; // group hashes and slots (sorted before the loop; scratch for large groups inside it)
    unsigned int* done;           // bitmap of processed slots (used when it does not fit in shared memory)
    long long vbase;              // first virtual pool index
    int32_t lb_shift;             // log2 of the number of slots per tournament leaf block
    int32_t nb;                   // number of leaf blocks
    int32_t done_in_smem;
    int32_t list_mode;            // the list mode of the loop can be used (trees without a budget)
    unsigned int* gbits;          // bitmap of slots whose group has more than one member, as the loop starts (and throughout, if the bitmaps stay in global memory)
    unsigned int* gskip;          // list mode with the bitmaps in global memory: slots whose key has changed since the sort
    int32_t bits_in_smem;         // list mode: those two bitmaps are in shared memory
    const long long* lk;          // list mode: every slot's key, largest first, stored as ~key with the top bit flipped
    const int32_t* ls;            //            and the slot it belongs to
    int32_t max_windows;          // list mode: windows after which the loop gives up (debug setting)
    const int64_t* arrival;       // per query: arrival (for the charge pass after the loop)
    struct FastPost* post;        // where list mode began, for the charge pass after the loop
    TreeState* st;
    // trees with a budget: the loop keeps the node arrays of the tree up to date itself (LRU needs them at every decision)
    int32_t lru;                  // 1: the tree has a budget
    int32_t mem_cap;              // entries of the member array (groups formed by evictions are appended behind the first n)
    TreeDev T;
    LNode* node;                  // the tree's node arrays, one record per node, while the loop runs
    int32_t* parked;              // per node: unprocessed slots whose hint is that node
    int32_t* hintc;               // per slot: the hint once more, side by side (what the scan after an eviction reads)
    int2* leaf_run;               // per node: the member run that holds every slot whose hint is that node (y < 0: no such run is known)
    long long* pk; int32_t* pi;   // set-up: (hint, slot) pairs, sorted by hint to give every node of the tree its run
    int32_t* skip;                // set by the capacity check before the loop: leave everything untouched
    // a given processing order instead of a policy (klpm_replay): decision c processes query fixed[c]; slots are the
    // queries in index order; *n_fixed decisions are made
    const int32_t* fixed;
    const int32_t* n_fixed;
};

#define KLPM_FAST_THREADS 256
#define KLPM_FAST_SORT_CAP 4096          // largest group that is regrouped exactly (sorted in shared memory)
#define KLPM_FAST_NOGROUP 0xffffffffffffffffULL

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {      // SplitMix64's finaliser
    z ^= z >> 30; z *= 0xbf58476d1ce4e5b9ULL; z ^= z >> 27; z *= 0x94d049bb133111ebULL; z ^= z >> 31;
    return z;
}
__device__ __forceinline__ unsigned long long group_hash(long long pos, int32_t ntok) {
    return mix64((unsigned long long)(pos + 2) * 0x9E3779B97F4A7C15ULL + (unsigned)ntok) >> 2;
}
__device__ __forceinline__ unsigned long long single_hash(int32_t slot) {       // a query that is fully cached never regroups
    return mix64(0xD1B54A32D192ED03ULL ^ (unsigned long long)(unsigned)slot) >> 2;
}
__device__ __forceinline__ unsigned long long fast_key(int32_t m, int32_t len, int32_t rank, int32_t score_mode) {
    unsigned hi = (unsigned)m;
    if (score_mode == 1) hi = len > 0 ? (unsigned)(((unsigned long long)(unsigned)m << 31) / (unsigned)len) : 0u;
    return ((unsigned long long)hi << 32) | (0xffffffffu - (unsigned)rank);
}
__device__ __forceinline__ FDyn ld_dyn(const FDyn* p) {
    const int4* q = reinterpret_cast<const int4*>(p);
    const int4 a = __ldcg(q), b = __ldcg(q + 1);
    FDyn d;
    d.pos = (long long)(((unsigned long long)(unsigned)a.y << 32) | (unsigned)a.x);
    d.m = a.z; d.ntok = a.w; d.gstart = b.x; d.gcount = b.y; d.hint = b.z; d.pad = 0;
    return d;
}
__device__ __forceinline__ FDyn ld_dyn_l1(const FDyn* p) {      // a plain load: served by L1 if another warp of the CTA has read it before
    const int4* q = reinterpret_cast<const int4*>(p);
    const int4 a = q[0], b = q[1];
    FDyn d;
    d.pos = (long long)(((unsigned long long)(unsigned)a.y << 32) | (unsigned)a.x);
    d.m = a.z; d.ntok = a.w; d.gstart = b.x; d.gcount = b.y; d.hint = b.z; d.pad = 0;
    return d;
}
__device__ __forceinline__ void st_dyn_state(FDyn* p, long long pos, int32_t m, int32_t ntok) {
    __stcg(reinterpret_cast<int4*>(p), make_int4((int)(unsigned)(unsigned long long)pos, (int)(unsigned)((unsigned long long)pos >> 32), m, ntok));
}
__device__ __forceinline__ void st_dyn_group(FDyn* p, int32_t gstart, int32_t gcount) {
    __stcg(reinterpret_cast<int2*>(p) + 2, make_int2(gstart, gcount));
}
__device__ __forceinline__ void st_dyn_hint(FDyn* p, int32_t hint) { __stcg(reinterpret_cast<int32_t*>(p) + 6, hint); }
__device__ __forceinline__ FStat ld_stat(const FStat* p) {
    const int4* q = reinterpret_cast<const int4*>(p);
    const int4 a = __ldg(q), b = __ldg(q + 1);
    FStat s;
    s.t = (long long)(((unsigned long long)(unsigned)a.y << 32) | (unsigned)a.x);
    s.len = a.z; s.ord = a.w;
    s.soff = (long long)(((unsigned long long)(unsigned)b.y << 32) | (unsigned)b.x);
    s.rank = b.z; s.pad = 0;
    return s;
}
__device__ __forceinline__ LNode ld_node(const LNode* p) {
    const int4* q = reinterpret_cast<const int4*>(p);
    const int4 a = q[0], b = q[1];
    LNode r;
    r.parent = a.x; r.depth = a.y; r.len = a.z; r.nchild = a.w;
    r.last = (long long)(((unsigned long long)(unsigned)b.y << 32) | (unsigned)b.x);
    r.off = (long long)(((unsigned long long)(unsigned)b.w << 32) | (unsigned)b.z);
    return r;
}
__device__ __forceinline__ void st_node(LNode* p, const LNode& r) {
    int4* q = reinterpret_cast<int4*>(p);
    q[0] = make_int4(r.parent, r.depth, r.len, r.nchild);
    q[1] = make_int4((int)(unsigned)(unsigned long long)r.last, (int)(unsigned)((unsigned long long)r.last >> 32),
                     (int)(unsigned)(unsigned long long)r.off, (int)(unsigned)((unsigned long long)r.off >> 32));
}
__device__ __forceinline__ void named_arrive(int id, int nthreads) {      // does not wait; what was written before is seen by whoever the barrier releases
    __threadfence_block();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void named_bar(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// slot -> constant record (after the slots have been ordered by arrival)
__global__ void fast_stat_kernel(const int32_t* __restrict__ ord, const long long* __restrict__ sorted_t,
                                 const int64_t* __restrict__ off, const int32_t* __restrict__ prank, int32_t n, FStat* stat) {
    const int32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int32_t qi = ord[r];
    const int64_t lo = off[qi];
    FStat s;
    s.soff = lo; s.t = sorted_t[r]; s.len = (int32_t)(off[qi + 1] - lo); s.ord = qi; s.rank = prank ? prank[r] : r; s.pad = 0;
    stat[r] = s;
}

// The hit-rate score is kept as floor(m * 2^31 / |x|) in the high half of a key.  Two different rates m/|x| and
// m'/|x'| differ by at least 1/(|x||x'|), so while every prompt is at most 46,340 tokens long (46,340^2 < 2^31)
// different rates get different quotients, equal rates equal ones, and the order of the keys is the order of the
// rates.  Longer prompts could tie where the rates do not: the status word says so.
#define KLPM_HIT_RATE_MAX_LEN 46340
__global__ void hit_rate_guard_kernel(const int64_t* __restrict__ off, int32_t n, TreeState* st) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && off[i + 1] - off[i] > KLPM_HIT_RATE_MAX_LEN) set_status(st, RT_ERR_INVALID, 109);
}

// Every slot's starting state from the record the batched match wrote for its query (MatchState): match length,
// position, next token; from those its key and the hash of its group.  One thread per slot (and per padding entry
// of the sort that follows).
__global__ void fast_state_kernel(FastArgs A, const MatchState* __restrict__ state, unsigned long long tag, long long np2) {
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= np2) return;
    if (r >= A.n) {                                                                        // padding of the sorts
        A.gh[r] = 0x7fffffffffffffffLL; A.gidx[r] = 0x7fffffff;
        if (A.lru) { A.pk[r] = 0x7fffffffffffffffLL; A.pi[r] = 0x7fffffff; }
        return;
    }
    const FStat s = ld_stat(A.stat + r);
    const int4* src = reinterpret_cast<const int4*>(state + s.ord);
    const int4 a = __ldcg(src), b = __ldcg(src + 1);
    const long long pos_in = (long long)(((unsigned long long)(unsigned)a.y << 32) | (unsigned)a.x);
    const long long node_in = (long long)(((unsigned long long)(unsigned)a.w << 32) | (unsigned)a.z);
    int32_t m = b.x, ntok = b.y;
    long long pos = pos_in;
    int32_t hint = 0;
    const unsigned long long got = ((unsigned long long)(unsigned)b.w << 32) | (unsigned)b.z;
    bool bad = got != tag || m < 0 || m > s.len;
    if (A.lru && !bad) { bad = node_in < 0 || node_in >= A.T.max_nodes; hint = (int32_t)node_in; }
    if (bad) {                                       // not the record of that match: say so and start this slot from nothing
        set_status(A.st, RT_ERR_INVALID, 110);
        m = 0; pos = -1; ntok = 0; hint = 0;
    }
    st_dyn_state(A.dyn + r, pos, m, ntok);
    if (A.lru) {
        st_dyn_hint(A.dyn + r, hint); A.hintc[r] = hint;
        const unsigned on = __activemask(), same = __match_any_sync(on, hint);      // (on an empty tree every query is parked at the root)
        if ((int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(A.parked + hint, __popc(same));
        A.pk[r] = hint; A.pi[r] = (int32_t)r;
    }
    A.key[r] = fast_key(m, s.len, s.rank, A.score_mode);
    A.gh[r] = (long long)(m < s.len ? group_hash(pos, ntok) : single_hash((int32_t)r));
    A.gidx[r] = (int32_t)r;
}

// Trees with a budget, after the sort by hint: the slots whose match ends in one node, side by side, are that node's
// run (entries n .. 2n-1 of the member array): where the loop looks when the node is evicted with queries parked in it.
__global__ void lru_parklist_kernel(FastArgs A) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    A.mem[A.n + i] = A.pi[i];
    const long long node = A.pk[i];
    if (i > 0 && A.pk[i - 1] == node) return;              // not the first of its run
    int32_t lo = i + 1, hi = A.n;                          // first index with a larger hint
    while (lo < hi) { const int32_t mid = (lo + hi) >> 1; if (A.pk[mid] <= node) lo = mid + 1; else hi = mid; }
    A.leaf_run[node] = make_int2(A.n + i, lo - i);
}

// The groups the loop starts from: slots with equal hashes, side by side in the member array (in any order).  A hash table
// counts them -- nothing needs them sorted, which took eight launches and 94 us for 32,768 slots, the three kernels take 20:
// every slot finds its entry and its number there, one slot per entry takes room in the member array, and every slot
// writes itself down.
struct GroupTable { unsigned long long* key; int32_t* cnt; int32_t* off; unsigned mask; int32_t* ent; int32_t* num; unsigned int* used; };
__device__ __forceinline__ void group_count(const FastArgs& A, const GroupTable& H, int32_t r) {
    const bool in = r < A.n;
    unsigned e = 0;
    if (in) {
        const unsigned long long h = (unsigned long long)A.gh[r];              // 62 bits
        const unsigned long long key = h + 1;                                  // 0: empty entry
        e = (unsigned)(h ^ (h >> 31)) & H.mask;
        for (unsigned probes = 0; probes <= H.mask; ++probes) {                // (at most half full: an entry is found)
            const unsigned long long old = atomicCAS(H.key + e, 0ULL, key);
            if (old == 0ULL || old == key) break;
            e = (e + 1) & H.mask;
        }
    }
    const int lane = threadIdx.x & 31;
    const unsigned same = __match_any_sync(FULL_MASK, in ? e : 0xffffffffu);
    const int lead = __ffs(same) - 1;
    int32_t at = 0;
    if (in && lane == lead) at = atomicAdd(H.cnt + e, __popc(same));
    at = __shfl_sync(FULL_MASK, at, lead) + __popc(same & ((1u << lane) - 1u));
    if (in) { H.ent[r] = (int32_t)e; H.num[r] = at; }
}
__device__ __forceinline__ void group_room(const FastArgs& A, const GroupTable& H, int32_t r) {
    const int lane = threadIdx.x & 31;
    const bool first = r < A.n && H.num[r] == 0;
    const int32_t e = first ? H.ent[r] : 0, cnt = first ? __ldcg(H.cnt + e) : 0;
    int32_t inc = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const int32_t o = __shfl_up_sync(FULL_MASK, inc, d); if (lane >= d) inc += o; }
    unsigned base = 0;
    if (lane == 31 && inc > 0) base = atomicAdd(H.used, (unsigned)inc);
    base = __shfl_sync(FULL_MASK, base, 31);
    if (first) H.off[e] = (int32_t)base + inc - cnt;
}
__device__ __forceinline__ void group_place(const FastArgs& A, const GroupTable& H, int32_t r) {
    if (r >= A.n) return;
    const int32_t e = H.ent[r], first = H.off[e], cnt = __ldcg(H.cnt + e);
    A.mem[first + H.num[r]] = r;
    st_dyn_group(A.dyn + r, first, cnt);
    if (cnt > 1) atomicOr(A.gbits + (r >> 5), 1u << (r & 31));
}
__global__ void group_count_kernel(FastArgs A, GroupTable H) { group_count(A, H, blockIdx.x * blockDim.x + threadIdx.x); }
__global__ void group_room_kernel(FastArgs A, GroupTable H) { group_room(A, H, blockIdx.x * blockDim.x + threadIdx.x); }
__global__ void fast_group_kernel(FastArgs A, GroupTable H) { group_place(A, H, blockIdx.x * blockDim.x + threadIdx.x); }
// The three, and the clearing of the table, in one launch for queues of up to a thread per slot of one CTA (four launches cost a
// queue of one prompt on a full cache 10 of 87 us, 1,000 prompts 5 of 102).
__global__ void __launch_bounds__(1024)
group_small_kernel(FastArgs A, GroupTable H) {
    for (unsigned i = threadIdx.x; i <= H.mask; i += 1024) { H.key[i] = 0ULL; H.cnt[i] = 0; }
    if (threadIdx.x == 0) *H.used = 0u;
    __syncthreads();
    group_count(A, H, threadIdx.x);
    __syncthreads();
    group_room(A, H, threadIdx.x);
    __syncthreads();
    group_place(A, H, threadIdx.x);
}

// Overlaps inside the groups the loop starts from, worked out by the whole chip before the one CTA of the loop needs them.
// Every member is compared with its group's first member (the reference): the record says whom it was compared with (-1:
// nobody, the slot is alone in its group or shares it by a hash collision only), up to which depth e the two agree, and
// the token that follows there (meaningful while e < length).  Two prompts with the same reference and different e
// overlap in the smaller e; with equal e and different next tokens, or one of them at its end, in exactly e; otherwise
// they agree beyond e and are compared from there (overlap_known).  That holds for any two prompts whatever happens to
// their groups later.  A warp takes `per` consecutive entries of the member array.
// `wanted` (null: all): per first entry of a group, whether it is looked at.  A given order (klpm_replay) that is short against the
// queue touches few groups, and the others are never dissolved.
// 120,000 prompts of 256 shared prefixes: 296 us, bound by the 0.9 GB of prefix tokens it compares; eight warps of the loop's
// CTA, which did the comparing before, took 73 ms for the same (220,000 cycles per group of a shared prefix, now 44,000).
// PAIRS: what becomes of groups of two is written down too (list mode).  An instance of its own: it takes 57 registers, the other one 48, which
// is 5 instead of 4 CTAs per SM in a kernel that lives from the loads it has in flight.
template <bool PAIRS>
__global__ void __launch_bounds__(256)
lcp_kernel(FastArgs A, int32_t per, const int32_t* __restrict__ wanted) {
    const int lane = threadIdx.x & 31;
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long i0 = w * per;
    const long long i = i0 + lane;
    int32_t r = -1, ref = -1, m = 0, len = 0, count = 0, other = -1;
    long long soff = 0;
    bool cmp = false;
    if (lane < per && i < A.n) {
        r = A.mem[i];
        const FDyn d = ld_dyn(A.dyn + r);
        if (d.gcount > 1 && (!wanted || wanted[d.gstart])) {
            count = d.gcount;
            ref = A.mem[d.gstart];
            other = ref;
            const FStat s = ld_stat(A.stat + r);
            m = d.m; len = s.len; soff = s.soff;
            if (ref != r) {
                const FDyn f = ld_dyn(A.dyn + ref);
                if (f.pos != d.pos || f.ntok != d.ntok || f.m != d.m || m >= len) ref = -1;
                else cmp = true;
            }
        }
    }
    int32_t e = len;
    for (unsigned todo = __ballot_sync(FULL_MASK, cmp); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const int32_t rf = __shfl_sync(FULL_MASK, ref, src), from = __shfl_sync(FULL_MASK, m, src), ql = __shfl_sync(FULL_MASK, len, src);
        const int32_t* q = A.tok + __shfl_sync(FULL_MASK, soff, src);
        const FStat f = ld_stat(A.stat + rf);
        const int32_t lim = (ql < f.len ? ql : f.len) - from;
        const int32_t x = from + first_mismatch<true>(q + from, A.tok + f.soff + from, lim);
        if (lane == src) e = x;
    }
    if (r >= 0) A.lcp[r] = make_int4(ref, e, e < len ? __ldg(A.tok + soff + e) : 0, 0);
    // A group of two is known completely: whoever is processed first, the other one matches e tokens from then on.  (Two slots that share
    // a run by a hash collision are no group.)
    if (!PAIRS || count < 2) return;
    if (count > 2) { A.pair[2LL * r] = make_int4(-2, 0, 0, 0); return; }
    if (other == r) return;                                 // (the other slot's lane writes both)
    if (!cmp) {
        atomicAnd(A.gbits + (r >> 5), ~(1u << (r & 31)));
        atomicAnd(A.gbits + (other >> 5), ~(1u << (other & 31)));
        return;
    }
    const FStat s = ld_stat(A.stat + r), f = ld_stat(A.stat + other);
    const unsigned long long kr = fast_key(e, s.len, s.rank, A.score_mode), kf = fast_key(e, f.len, f.rank, A.score_mode);
    const int4 mine = make_int4(other, e, (int)(unsigned)kf, (int)(unsigned)(kf >> 32)), its = make_int4(r, e, (int)(unsigned)kr, (int)(unsigned)(kr >> 32));
    A.pair[2LL * r] = mine; A.pair[2LL * r + 1] = its;
    A.pair[2LL * other] = its; A.pair[2LL * other + 1] = mine;
}
// The groups that a given order touches (see lcp_kernel).
__global__ void lcp_wanted_kernel(FastArgs A, int32_t* wanted) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= *A.n_fixed) return;
    const FDyn d = ld_dyn(A.dyn + A.fixed[p]);
    if (d.gcount > 1) wanted[d.gstart] = 1;
}
// The overlap of two prompts as far as their records tell it: true if *e is it, false if they agree at least up to *e.
__device__ __forceinline__ bool overlap_known(const int4& a, int32_t len_a, const int4& b, int32_t len_b, int32_t m, int32_t* e) {
    if (a.x < 0 || a.x != b.x) { *e = m; return false; }
    *e = a.y < b.y ? a.y : b.y;
    if (a.y != b.y || a.y >= len_a || b.y >= len_b || a.z != b.z) return true;
    if (*e < m) *e = m;                                     // (m: a depth up to which they are known to agree)
    return false;
}

// list mode: every slot's key in a form that sorts largest first (processed slots last, then the padding)
__global__ void fast_list_kernel(FastArgs A, long long np2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np2) return;
    const bool in = i < A.n, live = in && !(A.post->list_c > 0 && ((__ldcg(A.done + (i >> 5)) >> (i & 31)) & 1u));
    const_cast<long long*>(A.lk)[i] = live ? (long long)(~A.key[i] ^ 0x8000000000000000ULL) : 0x7fffffffffffffffLL;
    const_cast<int32_t*>(A.ls)[i] = in ? (int32_t)i : 0x7fffffff;
}

// Largest of the warp's 64-bit values with two hardware reductions: the high halves, then the low halves of
// the lanes that hold the largest high half.
__device__ __forceinline__ unsigned long long warp_max64r(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_max_sync(FULL_MASK, hi);
    const unsigned ml = __reduce_max_sync(FULL_MASK, hi == mh ? (unsigned)v : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

// position of the k-th set bit of w (k >= 1, at most the number of set bits)
__device__ __forceinline__ int kth_set_bit(unsigned w, int k) {
    int pos = 0;
    int cnt = __popc(w & 0xffffu); if (k > cnt) { k -= cnt; pos += 16; w >>= 16; }
    cnt = __popc(w & 0xffu);       if (k > cnt) { k -= cnt; pos += 8; w >>= 8; }
    cnt = __popc(w & 0xfu);        if (k > cnt) { k -= cnt; pos += 4; w >>= 4; }
    cnt = __popc(w & 0x3u);        if (k > cnt) { k -= cnt; pos += 2; w >>= 2; }
    if (k > (int)(w & 1u)) pos += 1;
    return pos;
}

// ---- the tournament above the leaf blocks (shared memory) ----
// t1[b] is the largest key of leaf block b among the slots the tournament holds: the arrived, unprocessed slots
// while arrivals are pending; in list mode (everybody has arrived) only those of them whose key has changed since
// the keys were sorted -- the others are picked from the sorted list.
struct FastTour {
    unsigned long long* t1;   // per leaf block (padded with zeros to a multiple of 32)
    unsigned long long* t2;   // per 32 leaf blocks (padded likewise)
    unsigned long long* t3;   // 32 entries
    unsigned int* done;       // bitmap of processed slots (shared memory), or null
    unsigned int* skip;       // bitmap of slots whose key has changed since the sort (the list passes over them), or null
    unsigned int* gb;         // bitmap of slots whose group has more than one member (shared memory), or null
    unsigned int* dirty;      // trees with a budget: bitmap of leaf blocks to recompute after a fallback (256 words, shared memory)
    int g_done, g_bits;       // the processed bitmap / the other two bitmaps live in global memory (queues too long for shared memory)
    int32_t n2;               // entries of t2 in use
    int32_t n3;               // entries of t3 in use
};
// A word of one of the loop's bitmaps: shared memory, or global memory read through L2 (other warps set bits with atomics).
__device__ __forceinline__ unsigned bm_ld(const unsigned int* p, long long i, int g) { return g ? __ldcg(p + i) : p[i]; }

// The first unprocessed slot after `head` (which is processed); n if there is none.  One warp.
__device__ __forceinline__ int32_t next_head(const unsigned int* s_done, int gdone, int32_t nwords, int32_t n, int32_t head, int lane) {
    if (head + 1 < n) {                                     // the usual cases: the next slot, or one of the next 32 to 63
        const int32_t h1 = head + 1, wi = h1 >> 5;
        const unsigned f0 = ~bm_ld(s_done, wi, gdone) & ~((1u << (h1 & 31)) - 1u);
        if (f0) { head = wi * 32 + __ffs(f0) - 1; return head > n ? n : head; }
        if (wi + 1 < nwords) {
            const unsigned f1 = ~bm_ld(s_done, wi + 1, gdone);
            if (f1) { head = (wi + 1) * 32 + __ffs(f1) - 1; return head > n ? n : head; }
        }
    }
    int32_t w0 = head >> 5;
    for (;;) {
        const int32_t wi = w0 + lane;
        unsigned w = 0u;                                      // past the end: "unprocessed", so the search stops
        if (wi < nwords) w = bm_ld(s_done, wi, gdone);
        if (wi == (head >> 5)) w |= (1u << (head & 31)) - 1u;
        const unsigned bal = __ballot_sync(FULL_MASK, w != 0xffffffffu);
        if (bal) {
            const int src = __ffs(bal) - 1;
            const unsigned fw = ~__shfl_sync(FULL_MASK, w, src);
            head = (w0 + src) * 32 + __ffs(fw) - 1;
            break;
        }
        w0 += 32;
    }
    return head > n ? n : head;
}

// Recompute the ancestors of leaf block b; returns the root.  One warp.
__device__ __forceinline__ unsigned long long tour_update(const FastTour& R, int32_t b, int lane) {
    const int32_t i2 = b >> 5;
    unsigned long long v = warp_max64r(R.t1[(i2 << 5) + lane]);
    if (lane == 0) R.t2[i2] = v;
    __syncwarp();
    const int32_t i3 = i2 >> 5;
    v = warp_max64r(R.t2[(i3 << 5) + lane]);
    if (lane == 0) R.t3[i3] = v;
    __syncwarp();
    return warp_max64r(R.t3[lane]);
}
// Leaf block b's largest key becomes v: write it and its ancestors; returns the root.  One warp; every lane
// performs the same stores, so each lane sees them in its own program order without a barrier.
__device__ __forceinline__ unsigned long long tour_set(const FastTour& R, int32_t b, unsigned long long v, int lane) {
    const int32_t i2 = b >> 5, i3 = i2 >> 5;
    const unsigned long long o1 = warp_max64r(lane == (b & 31) ? 0ULL : R.t1[(i2 << 5) + lane]);
    const unsigned long long o2 = warp_max64r(lane == (i2 & 31) ? 0ULL : R.t2[(i3 << 5) + lane]);
    const unsigned long long o3 = warp_max64r(lane == i3 ? 0ULL : R.t3[lane]);
    const unsigned long long v2 = v > o1 ? v : o1, v3 = v2 > o2 ? v2 : o2;
    R.t1[b] = v; R.t2[i2] = v2; R.t3[i3] = v3;
    return v3 > o3 ? v3 : o3;
}
// Recompute t3 and the root from t2.  One warp.
__device__ __forceinline__ unsigned long long tour_top(const FastTour& R, int lane) {
    for (int32_t i3 = 0; i3 < R.n3; ++i3) {
        const unsigned long long v = warp_max64r(R.t2[(i3 << 5) + lane]);
        if (lane == 0) R.t3[i3] = v;
    }
    __syncwarp();
    return warp_max64r(R.t3[lane]);
}
// Recompute t2 from t1.  Every warp of the CTA; the caller synchronises.
__device__ __forceinline__ void tour_mid(const FastTour& R, int warp, int nwarps, int lane) {
    for (int32_t i2 = warp; i2 < R.n2; i2 += nwarps) {
        const unsigned long long v = warp_max64r(R.t1[(i2 << 5) + lane]);
        if (lane == 0) R.t2[i2] = v;
    }
}
// has slot r been processed?  (the bitmap lives in shared memory when it fits)
__device__ __forceinline__ bool slot_done(const FastTour& R, const FastArgs& A, long long r) {
    const unsigned w = bm_ld(R.done, r >> 5, R.g_done);
    return (w >> (r & 31)) & 1u;
}
__device__ __forceinline__ void set_grouped(const FastTour& R, int32_t r, bool grouped) {
    if (!R.gb) return;
    if (grouped) atomicOr(R.gb + (r >> 5), 1u << (r & 31));
    else atomicAnd(R.gb + (r >> 5), ~(1u << (r & 31)));
}

// An entry of the member array: a slot, always.  Anything else is recorded and passed over (-1) instead of being used as an index.
__device__ __forceinline__ int32_t ld_member(const FastArgs& A, int32_t i) {
    const int32_t r = __ldcg(A.mem + i);
    if ((unsigned)r < (unsigned)A.n) return r;
    set_status(A.st, RT_ERR_LIMIT, 119);
    return -1;
}

struct FastPick {             // the prompt being processed, as its group's members need it
    int32_t slot, m, len, ntok;
    const int32_t* x;         // its tokens
    int4 lcp;                 // its record of lcp_kernel
    long long pos;
    long long vleaf;          // virtual pool index of the first token of its new leaf
    long long admitted;       // slots below this have arrived
    int32_t gstart, gcount;
    int32_t leaf;             // trees with a budget: id of its new leaf (the tied members are parked in it from now on)
};
struct FastJob { int32_t type; int32_t a0, a1; FastPick pick; };
enum { FAST_JOB_EXIT = 0, FAST_JOB_ADMIT = 1, FAST_JOB_DISSOLVE = 2, FAST_JOB_FALLBACK = 3 };

// trees with a budget: slot r's match now ends inside node `to` (it was counted for node `from`)
__device__ __forceinline__ void lru_move(const FastArgs& A, int32_t r, int32_t from, int32_t to) {
    st_dyn_hint(A.dyn + r, to);
    __stcg(A.hintc + r, to);
    atomicSub(A.parked + from, 1);
    atomicAdd(A.parked + to, 1);
}

// One member of the dissolving group per lane (r < 0: none).  Members tied with the processed prompt are
// compared with its uncached tokens and get their new state and key; every live member gets the hash of the
// group it belongs to from now on (KLPM_FAST_NOGROUP: it leaves the run).  *touched: its key grew and it
// has arrived, so its leaf block's ancestors need recomputing.  Warp-cooperative.
__device__ __forceinline__ unsigned long long fast_member(const FastArgs& A, const FastPick& P, const FastTour& R, int32_t r, int lane,
                                                          bool* touched) {
    const bool act = r >= 0 && r != P.slot;
    FDyn d; d.pos = 0; d.m = -1; d.ntok = 0; d.gstart = 0; d.gcount = 0;
    FStat s; s.soff = 0; s.t = 0; s.len = 0; s.ord = 0; s.rank = 0;
    if (act) { d = ld_dyn(A.dyn + r); s = ld_stat(A.stat + r); }
    const bool live = act && !slot_done(R, A, r);
    const bool tied = live && d.pos == P.pos && d.ntok == P.ntok && d.m == P.m && d.m < s.len;
    const int32_t* q = A.tok + s.soff;
    int32_t from = P.m;                                     // they agree at least up to here
    bool known = false;
    if (tied) known = overlap_known(__ldcg(A.lcp + r), s.len, P.lcp, P.len, P.m, &from);
    int32_t e = from - P.m;
    unsigned cm = __ballot_sync(FULL_MASK, tied && !known);
    while (cm) {
        const int src = __ffs(cm) - 1; cm &= cm - 1;
        const int32_t* qq = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)q, src);
        const int32_t ql = __shfl_sync(FULL_MASK, s.len, src);
        const int32_t f = __shfl_sync(FULL_MASK, from, src);
        const int32_t lim = (ql < P.len ? ql : P.len) - f;
        const int32_t ee = first_mismatch<true>(qq + f, P.x + f, lim);
        if (lane == src) e = f + ee - P.m;
    }
    *touched = false;
    if (tied) {
        d.m = P.m + e; d.pos = P.vleaf + e - 1; d.ntok = d.m < s.len ? __ldg(q + d.m) : 0;
        st_dyn_state(A.dyn + r, d.pos, d.m, d.ntok);
        if (A.lru) lru_move(A, r, d.hint, P.leaf);
        const unsigned long long key = fast_key(d.m, s.len, s.rank, A.score_mode);
        __stcg(A.key + r, key);
        if (R.skip) atomicOr(R.skip + (r >> 5), 1u << (r & 31));          // its entry of the sorted list is stale now
        if ((long long)r < P.admitted) { atomicMax(R.t1 + (r >> A.lb_shift), key); *touched = true; }
    }
    if (!live) return KLPM_FAST_NOGROUP;
    return d.m < s.len ? group_hash(d.pos, d.ntok) : single_hash(r);
}

// Small groups are handled by the sequencer warp alone, unless several long compares are better spread over the CTA.
__device__ __forceinline__ bool dissolve_is_small(const FastPick& P) { return P.gcount <= 32 && (P.lcp.x >= 0 || P.gcount <= 2 || P.len - P.m <= 512); }

// The sequencer warp dissolves a group of at most 32 members and regroups it inside its run; returns the tournament's root.
__device__ __forceinline__ unsigned long long dissolve_small(const FastArgs& A, const FastPick& P, const FastTour& R, unsigned long long root, int lane) {
    const int32_t r = lane < P.gcount ? ld_member(A, P.gstart + lane) : -1;
    bool touched;
    const unsigned long long h = fast_member(A, P, R, r, lane, &touched);
    int32_t rank = 0, start = 0, cnt = 0;
    for (int k2i = 0; k2i < P.gcount; ++k2i) {              // (at most 32)
        const unsigned long long hk = __shfl_sync(FULL_MASK, h, k2i);
        const bool lt = hk < h, eq = hk == h;
        start += lt; cnt += eq; rank += (lt || (eq && k2i < lane));
    }
    if (h != KLPM_FAST_NOGROUP) {
        __stcg(A.mem + P.gstart + rank, r);
        st_dyn_group(A.dyn + r, P.gstart + start, cnt);
        set_grouped(R, r, cnt > 1);
    }
    __syncwarp();
    unsigned tm = __ballot_sync(FULL_MASK, touched);
    while (tm) {
        const int src = __ffs(tm) - 1; tm &= tm - 1;
        const int32_t bb = __shfl_sync(FULL_MASK, r >> A.lb_shift, src);
        root = tour_update(R, bb, lane);
    }
    return root;
}

// sh[0..p2) / sr[0..p2) hold the group hash and the slot of cnt members (padded with KLPM_FAST_NOGROUP / -1 up to the
// power of two p2): sort them by hash and write them to the member array from `gs` on, every member with the run of
// equal hashes it is in as its group.  Every thread of the CTA calls it.
__device__ void sort_and_group(const FastArgs& A, const FastTour& R, unsigned long long* sh, int32_t* sr, int32_t cnt, int32_t p2, int32_t gs) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int32_t k = 2; k <= p2; k <<= 1)
        for (int32_t j = k >> 1; j > 0; j >>= 1) {
            for (int32_t i = tid; i < p2; i += nthr) {
                const int32_t l = i ^ j;
                if (l > i) {
                    const unsigned long long a = sh[i], b = sh[l];
                    if ((a > b) == ((i & k) == 0)) { sh[i] = b; sh[l] = a; const int32_t t = sr[i]; sr[i] = sr[l]; sr[l] = t; }
                }
            }
            __syncthreads();
        }
    for (int32_t i = tid; i < cnt; i += nthr) {
        const unsigned long long h = sh[i];
        if (h == KLPM_FAST_NOGROUP) continue;
        int32_t lo = 0, hi = i;
        while (lo < hi) { const int32_t mid = (lo + hi) >> 1; if (sh[mid] < h) lo = mid + 1; else hi = mid; }
        const int32_t first = lo;
        lo = i + 1; hi = cnt;
        while (lo < hi) { const int32_t mid = (lo + hi) >> 1; if (sh[mid] <= h) lo = mid + 1; else hi = mid; }
        const int32_t r = sr[i];
        __stcg(A.mem + gs + i, r);
        st_dyn_group(A.dyn + r, gs + first, lo - first);
        set_grouped(R, r, lo - first > 1);
    }
}

// The same for more members than the shared-memory scratch holds: A.gh[0..cnt) / A.gidx[0..cnt) hold hash and slot.  A
// bitonic sort of the arrays in global memory -- partner distances of a tile (4,096) and more one pass over global
// memory each, everything below inside shared memory tile by tile -- then the runs of equal hashes become the groups.
__device__ void sort_large_and_group(const FastArgs& A, const FastTour& R, unsigned long long* sh, int32_t* sr, int32_t cnt, int32_t gs) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    constexpr int32_t TILE = KLPM_FAST_SORT_CAP;
    int32_t p2 = TILE;
    while (p2 < cnt) p2 <<= 1;
    for (int32_t i = cnt + tid; i < p2; i += nthr) { __stcg(A.gh + i, (long long)KLPM_FAST_NOGROUP); __stcg(A.gidx + i, -1); }
    __syncthreads();
    // stages k_lo .. k_hi (or the tail of one stage) on every tile, in shared memory
    auto tiles = [&](int32_t k_lo, int32_t k_hi) {
        for (int32_t base = 0; base < p2; base += TILE) {
            for (int32_t i = tid; i < TILE; i += nthr) { sh[i] = (unsigned long long)__ldcg(A.gh + base + i); sr[i] = __ldcg(A.gidx + base + i); }
            __syncthreads();
            for (int32_t k = k_lo; k <= k_hi; k <<= 1) {
                const int32_t jmax = (k >> 1) < (TILE >> 1) ? (k >> 1) : (TILE >> 1);
                for (int32_t j = jmax; j > 0; j >>= 1) {
                    for (int32_t i = tid; i < TILE; i += nthr) {
                        const int32_t l = i ^ j;
                        if (l > i) {
                            const unsigned long long a = sh[i], b = sh[l];
                            if ((a > b) == (((base + i) & k) == 0)) { sh[i] = b; sh[l] = a; const int32_t t = sr[i]; sr[i] = sr[l]; sr[l] = t; }
                        }
                    }
                    __syncthreads();
                }
            }
            for (int32_t i = tid; i < TILE; i += nthr) { __stcg(A.gh + base + i, (long long)sh[i]); __stcg(A.gidx + base + i, sr[i]); }
            __syncthreads();
        }
    };
    tiles(2, TILE);
    for (int32_t k = TILE << 1; k <= p2; k <<= 1) {
        for (int32_t j = k >> 1; j >= TILE; j >>= 1) {
            for (int32_t i = tid; i < p2; i += nthr) {
                const int32_t l = i ^ j;
                if (l > i) {
                    const unsigned long long a = (unsigned long long)__ldcg(A.gh + i), b = (unsigned long long)__ldcg(A.gh + l);
                    if ((a > b) == ((i & k) == 0)) {
                        const int32_t ri = __ldcg(A.gidx + i), rl = __ldcg(A.gidx + l);
                        __stcg(A.gh + i, (long long)b); __stcg(A.gh + l, (long long)a); __stcg(A.gidx + i, rl); __stcg(A.gidx + l, ri);
                    }
                }
            }
            __syncthreads();
        }
        tiles(k, k);
    }
    // runs of equal hashes; nearly every member is alone, which its two neighbours show
    for (int32_t i = tid; i < cnt; i += nthr) {
        const unsigned long long h = (unsigned long long)__ldcg(A.gh + i);
        if (h == KLPM_FAST_NOGROUP) continue;
        int32_t first = i, last = i + 1;
        if (i > 0 && (unsigned long long)__ldcg(A.gh + i - 1) == h) {
            int32_t lo = 0, hi = i;
            while (lo < hi) { const int32_t mid = (lo + hi) >> 1; if ((unsigned long long)__ldcg(A.gh + mid) < h) lo = mid + 1; else hi = mid; }
            first = lo;
        }
        if (i + 1 < cnt && (unsigned long long)__ldcg(A.gh + i + 1) == h) {
            int32_t lo = i + 1, hi = cnt;
            while (lo < hi) { const int32_t mid = (lo + hi) >> 1; if ((unsigned long long)__ldcg(A.gh + mid) <= h) lo = mid + 1; else hi = mid; }
            last = lo;
        }
        const int32_t r = __ldcg(A.gidx + i);
        __stcg(A.mem + gs + i, r);
        st_dyn_group(A.dyn + r, gs + first, last - first);
        set_grouped(R, r, last - first > 1);
    }
}

// t1 of leaf block b: the largest key among its arrived (< a1), unprocessed slots.  One warp.
__device__ __forceinline__ void admit_blocks_one(const FastArgs& A, const FastTour& R, int32_t b, int32_t lo_slot, int32_t a1, int lane) {
    unsigned long long v = 0;
    for (int32_t u = lane; u < (1 << A.lb_shift); u += 32) {
        const long long r = (long long)lo_slot + u;
        if (r < a1 && !slot_done(R, A, r)) { const unsigned long long kk = __ldcg(A.key + r); if (kk > v) v = kk; }
    }
    v = warp_max64r(v);
    if (lane == 0) R.t1[b] = v;
}

// t1 of every leaf block that holds a slot of [a0, a1): the largest key among its arrived (< a1), unprocessed slots.
__device__ void admit_blocks(const FastArgs& A, const FastTour& R, int32_t a0, int32_t a1) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (a1 <= a0) return;
    const int32_t b0 = a0 >> A.lb_shift, b1 = (a1 - 1) >> A.lb_shift;
    const int32_t LB = 1 << A.lb_shift;
    for (int32_t b = b0 + warp; b <= b1; b += nwarps) {
        unsigned long long v = 0;
        for (int32_t u = lane; u < LB; u += 32) {
            const long long r = ((long long)b << A.lb_shift) + u;
            if (r < a1 && !slot_done(R, A, r)) { const unsigned long long kk = __ldcg(A.key + r); if (kk > v) v = kk; }
        }
        v = warp_max64r(v);
        if (lane == 0) R.t1[b] = v;
    }
}

// Work the whole CTA shares; every thread calls it with the same job.  Ends with t2 recomputed from t1.
template <bool LRU>
__device__ void fast_job(const FastArgs& A, const FastTour& R, const FastJob& J, unsigned long long* sh, int32_t* sr, int* s_cnt,
                         int32_t* s_memcur) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (J.type == FAST_JOB_ADMIT) {
        // slots [a0, a1) have arrived: the largest key of every leaf block they fall into
        admit_blocks(A, R, J.a0, J.a1);
    } else if (J.type == FAST_JOB_FALLBACK) {
      if constexpr (LRU) {
        // Trees with a budget: a leaf in which queries were parked has been evicted.  Every unprocessed slot whose hint
        // is a dead node walks up to the node its match ends in now; the slots that lose matched tokens that way (the
        // match ended inside an evicted leaf) end at the end of a live node's edge, get their new state and key, and
        // are grouped afresh in a run appended to the member array: everybody who falls back to one position with one
        // next token is in this batch (a query parked there before would have matched into the leaf that was there).
        if (tid == 0) *s_cnt = 0;
        for (int32_t i = tid; i < 256; i += nthr) R.dirty[i] = 0u;
        __syncthreads();
        // slots below a0 (the oldest unprocessed slot) are all processed; four hints, then four dead flags, in flight per thread
        for (int32_t r0 = J.a0 + tid; r0 < A.n; r0 += 4 * nthr) {
            int32_t hh[4];
            bool dd[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { const int32_t r = r0 + u * nthr; hh[u] = r < A.n ? __ldcg(A.hintc + r) : 0; }
#pragma unroll
            for (int u = 0; u < 4; ++u) dd[u] = hh[u] != 0 && __ldcg(&A.node[hh[u]].nchild) < 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t r = r0 + u * nthr, h = hh[u];
                if (!dd[u] || slot_done(R, A, r)) continue;
                const int32_t* dp = reinterpret_cast<const int32_t*>(A.dyn + r);
                const int32_t m0 = __ldcg(dp + 2);
                int32_t m = m0, a = h;
                while (a != 0) {
                    const LNode w = ld_node(A.node + a);
                    if (w.nchild < 0) { if (w.depth < m) m = w.depth; }
                    else if (m > w.depth) break;
                    a = w.parent;
                }
                st_dyn_hint(A.dyn + r, a);
                __stcg(A.hintc + r, a);
                atomicAdd(A.parked + a, 1);                  // (what the dead node was counted for no longer matters)
                A.leaf_run[a].y = -1;                        // slots from elsewhere are parked in a now: no one run holds them all
                if (m != m0) {
                    const FStat s = ld_stat(A.stat + r);
                    long long pos = -1;
                    if (a != 0) { const LNode w = ld_node(A.node + a); pos = w.off + (long long)(m - w.depth) - 1; }
                    const int32_t ntok = __ldg(A.tok + s.soff + m);                 // m < m0 <= length
                    st_dyn_state(A.dyn + r, pos, m, ntok);
                    __stcg(A.key + r, fast_key(m, s.len, s.rank, A.score_mode));
                    if (r < J.a1) { const int32_t b = r >> A.lb_shift; atomicOr(R.dirty + (b >> 5), 1u << (b & 31)); }
                    const int32_t k = atomicAdd(s_cnt, 1);
                    __stcg(A.gh + k, (long long)group_hash(pos, ntok));
                    __stcg(A.gidx + k, r);
                }
            }
        }
        __syncthreads();
        const int32_t F = *s_cnt, base = *s_memcur;
        __syncthreads();
        if (F > 0) {
            if ((long long)base + F > (long long)A.mem_cap) {
                if (tid == 0) set_status(A.st, RT_ERR_CAPACITY, 113);      // no room for the new groups: the results are void
            } else {
                if (tid == 0) *s_memcur = base + F;
                if (F <= KLPM_FAST_SORT_CAP) {
                    int32_t p2 = 1;
                    while (p2 < F) p2 <<= 1;
                    for (int32_t i = tid; i < p2; i += nthr) {
                        sh[i] = i < F ? (unsigned long long)__ldcg(A.gh + i) : KLPM_FAST_NOGROUP;
                        sr[i] = i < F ? __ldcg(A.gidx + i) : -1;
                    }
                    __syncthreads();
                    sort_and_group(A, R, sh, sr, F, p2, base);
                } else {
                    sort_large_and_group(A, R, sh, sr, F, base);
                }
            }
        }
        __syncthreads();
        // keys went down: the leaf blocks that hold an arrived slot which fell back are recomputed
        for (int32_t w = warp; w < 256; w += nwarps) {
            unsigned bits = R.dirty[w];
            while (bits) {
                const int32_t b = w * 32 + __ffs(bits) - 1;
                bits &= bits - 1;
                const int32_t lo_slot = b << A.lb_shift;
                admit_blocks_one(A, R, b, lo_slot, J.a1, lane);
            }
        }
      }
    } else {
        // dissolve a group of more than 32 members, or a smaller one whose members have long compares ahead
        const FastPick& P = J.pick;
        const int32_t gs = P.gstart, gc = P.gcount;
        const bool exact = gc <= KLPM_FAST_SORT_CAP;
        int32_t p2 = 1;
        while (p2 < gc) p2 <<= 1;
        if (exact) {
            // classify the members; the tied ones go on a list (A.gidx is free while the run is sorted in shared memory)
            if (tid == 0) *s_cnt = 0;
            __syncthreads();
            for (int32_t base = warp * 32; base < gc; base += nwarps * 32) {
                const int32_t i = base + lane;
                const int32_t r = i < gc ? ld_member(A, gs + i) : -1;
                const bool act = r >= 0 && r != P.slot;
                unsigned long long h = KLPM_FAST_NOGROUP;
                if (act && !slot_done(R, A, r)) {
                    const FDyn d = ld_dyn(A.dyn + r);
                    const FStat s = ld_stat(A.stat + r);
                    if (d.pos == P.pos && d.ntok == P.ntok && d.m == P.m && d.m < s.len) {
                        int32_t m2;
                        const int4 rec = __ldcg(A.lcp + r);
                        if (!overlap_known(rec, s.len, P.lcp, P.len, P.m, &m2)) __stcg(A.gidx + atomicAdd(s_cnt, 1), i);
                        else {
                            const long long pos2 = P.vleaf + (m2 - P.m) - 1;
                            const int32_t ntok2 = m2 >= s.len ? 0 : m2 == rec.y ? rec.z : __ldg(A.tok + s.soff + m2);
                            st_dyn_state(A.dyn + r, pos2, m2, ntok2);
                            if (LRU) lru_move(A, r, d.hint, P.leaf);
                            const unsigned long long key = fast_key(m2, s.len, s.rank, A.score_mode);
                            __stcg(A.key + r, key);
                            if (R.skip) atomicOr(R.skip + (r >> 5), 1u << (r & 31));
                            if ((long long)r < P.admitted) atomicMax(R.t1 + (r >> A.lb_shift), key);
                            h = m2 < s.len ? group_hash(pos2, ntok2) : single_hash(r);
                        }
                    } else h = d.m < s.len ? group_hash(d.pos, d.ntok) : single_hash(r);
                }
                if (i < gc) { sh[i] = h; sr[i] = r; }
            }
            for (int32_t i = gc + tid; i < p2; i += nthr) { sh[i] = KLPM_FAST_NOGROUP; sr[i] = -1; }
            __syncthreads();
            // one tied member per warp at a time: compare it with the processed prompt's uncached tokens
            const int32_t nt = *s_cnt;
            for (int32_t k = warp; k < nt; k += nwarps) {
                const int32_t i = __ldcg(A.gidx + k);
                const int32_t r = sr[i];
                const FStat s = ld_stat(A.stat + r);
                const int32_t* qq = A.tok + s.soff;
                int32_t from;
                overlap_known(__ldcg(A.lcp + r), s.len, P.lcp, P.len, P.m, &from);
                const int32_t lim = (s.len < P.len ? s.len : P.len) - from;
                const int32_t e = from - P.m + first_mismatch<true, 8>(qq + from, P.x + from, lim);
                if (lane == 0) {
                    const int32_t m2 = P.m + e;
                    const long long pos2 = P.vleaf + e - 1;
                    const int32_t ntok2 = m2 < s.len ? __ldg(qq + m2) : 0;
                    st_dyn_state(A.dyn + r, pos2, m2, ntok2);
                    if (LRU) lru_move(A, r, __ldcg(reinterpret_cast<const int32_t*>(A.dyn + r) + 6), P.leaf);
                    const unsigned long long key = fast_key(m2, s.len, s.rank, A.score_mode);
                    __stcg(A.key + r, key);
                    if (R.skip) atomicOr(R.skip + (r >> 5), 1u << (r & 31));
                    if ((long long)r < P.admitted) atomicMax(R.t1 + (r >> A.lb_shift), key);
                    sh[i] = m2 < s.len ? group_hash(pos2, ntok2) : single_hash(r);
                }
            }
        } else {
            for (int32_t base = warp * 32; base < gc; base += nwarps * 32) {
                const int32_t i = base + lane;
                const int32_t r = i < gc ? ld_member(A, gs + i) : -1;
                bool touched;
                const unsigned long long h = fast_member(A, P, R, r, lane, &touched);
                if (i < gc) { __stcg(A.gh + i, (long long)h); __stcg(A.gidx + i, r); }
            }
            if (tid == 0) *s_cnt = 0;
        }
        __syncthreads();
        if (exact) {
            // regroup exactly: sort the members by the hash of their new group inside the run
            sort_and_group(A, R, sh, sr, gc, p2, gs);
        } else {
            // too many for the shared-memory sort: the same regrouping with the arrays in global memory
            sort_large_and_group(A, R, sh, sr, gc, gs);
        }
    }
    __syncthreads();
    tour_mid(R, warp, nwarps, lane);
    __syncthreads();
}

// The loop while arrivals are pending: every decision is one careful step: admit who has arrived, pick from the
// tournament over all arrived slots (or the oldest slot), take the pick out of its leaf block, charge it and dissolve its
// group.  Once everybody has arrived the time of a pick no longer decides who can be picked, and list_run_kernel goes on.
// G: some of the loop's bitmaps live in global memory (queues too long for shared memory).  The instance without them
// reads its bitmaps as plain shared-memory words.
template <bool G>
__global__ void __launch_bounds__(KLPM_FAST_THREADS, 1)
fast_run_kernel(FastArgs A) {
    extern __shared__ __align__(16) unsigned char fast_smem[];
    __shared__ FastJob s_job;
    __shared__ int s_cnt;
    __shared__ int32_t s_memcur;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t n = A.n;
    if (A.list_mode && __ldg(&A.stat[n - 1].t) <= A.start_tick) {      // everybody is waiting as the loop starts: nothing to do here
        if (threadIdx.x == 0) {
            A.post->c0 = 0; A.post->list_c = 0; A.post->now0 = A.start_tick; A.post->head = 0; A.post->cyc = 0;
            for (int i = 0; i < 16; ++i) A.post->counters[i] = 0;
        }
        return;
    }
    const int32_t nb1p = (A.nb + 31) & ~31, n2 = nb1p >> 5, n2p = (n2 + 31) & ~31, n3 = n2p >> 5;
    const int32_t nwords = (n + 31) >> 5;
    FastTour R;
    R.t1 = reinterpret_cast<unsigned long long*>(fast_smem);
    R.t2 = R.t1 + nb1p;
    R.t3 = R.t2 + n2p;
    R.n2 = n2; R.n3 = n3;
    unsigned long long* sh = R.t3 + 32;
    int32_t* sr = reinterpret_cast<int32_t*>(sh + KLPM_FAST_SORT_CAP);
    unsigned int* s_bits = reinterpret_cast<unsigned int*>(sr + KLPM_FAST_SORT_CAP);
    // the bitmaps: in shared memory while they fit, in global memory (cleared / filled by the host side) otherwise
    R.g_done = A.done_in_smem ? 0 : 1;
    R.g_bits = A.bits_in_smem ? 0 : 1;
    R.done = A.done_in_smem ? s_bits : A.done;
    R.skip = nullptr;
    R.gb = !A.list_mode ? nullptr : A.bits_in_smem ? s_bits + 2 * nwords : A.gbits;
    R.dirty = nullptr;
    unsigned int* const s_done = R.done;
    if (!G) { R.g_done = 0; R.g_bits = 0; }
    const int gdone = G ? R.g_done : 0;
    for (int32_t i = threadIdx.x; i < nb1p + n2p + 32; i += blockDim.x) R.t1[i] = 0ULL;
    if (threadIdx.x == 0) s_memcur = n;
    if (A.done_in_smem) for (int32_t i = threadIdx.x; i < nwords; i += blockDim.x) s_bits[i] = 0u;
    if (A.list_mode && A.bits_in_smem) for (int32_t i = threadIdx.x; i < nwords; i += blockDim.x) R.gb[i] = __ldcg(A.gbits + i);
    __syncthreads();

    if (warp != 0) {
        for (;;) {
            named_bar(1, KLPM_FAST_THREADS);
            const FastJob J = s_job;
            if (J.type == FAST_JOB_EXIT) {
                if (J.a0) {                                 // list_run_kernel takes over: it needs the bitmaps
                    for (int32_t i = threadIdx.x - 32; i < nwords; i += KLPM_FAST_THREADS - 32) {
                        if (A.done_in_smem) __stcg(A.done + i, R.done[i]);
                        if (A.bits_in_smem) __stcg(A.gbits + i, R.gb[i]);
                    }
                }
                return;
            }
            fast_job<false>(A, R, J, sh, sr, &s_cnt, &s_memcur);
        }
    }

    // ---------------------------------------------------------------- the sequencer (warp 0)
    const long long INF = 0x7fffffffffffffffLL;
    long long now = A.start_tick;
    int32_t head = 0, admitted = 0;
    long long next_t = __ldg(&A.stat[0].t);
    unsigned long long root = 0;
    long long n_careful = 0, n_cta_dissolve = 0, cy_dissolve = 0;
    int32_t cyc = 0;                                        // c mod k
    int32_t c = 0;
    bool failed = false;

    auto advance_head = [&]() { head = next_head(s_done, gdone, nwords, n, head, lane); };
    // slot j is processed from now on (every lane performs the same shared-memory stores)
    auto mark_done = [&](int32_t j) {
        if (!gdone) s_done[j >> 5] |= 1u << (j & 31);
        else if (lane == 0) __stcg(s_done + (j >> 5), __ldcg(s_done + (j >> 5)) | (1u << (j & 31)));
        __syncwarp();
    };
    // Charge pick `slot` (Definition 2; not in a given order, whose charging is the pass after the loop), write its outputs, and let the queries tied with it match into its new
    // leaf.  The caller has taken the slot out of the tournament or the list and marked it processed.
    auto careful = [&](int32_t slot, bool charge, const FDyn& d, const FStat& s) {
        const int32_t m = d.m, len = s.len, unc = len - m;
        if (charge) {
            const long long begin = now > s.t ? now : s.t;
            const long long Rj = begin + (A.c_den + A.c_num * (long long)len) * (long long)unc;
            now = Rj;
            if (lane == 0) {
                if (A.order) A.order[c] = s.ord;
                A.uncached[s.ord] = unc; A.ttft[s.ord] = Rj - s.t;
                if (A.completion) A.completion[s.ord] = Rj;
            }
        }
        // the new leaf's positions: unique per decision, above every real pool index
        const long long vleaf = A.vbase + ((long long)c << 32);
        ++c;
        ++n_careful;
        if (unc > 0 && d.gcount > 1) {
            FastPick P;
            P.slot = slot; P.m = m; P.len = len; P.ntok = d.ntok; P.x = A.tok + s.soff; P.pos = d.pos; P.vleaf = vleaf;
            P.admitted = admitted; P.gstart = d.gstart; P.gcount = d.gcount; P.leaf = -1;
            P.lcp = __ldcg(A.lcp + slot);
            if (dissolve_is_small(P)) {
                root = dissolve_small(A, P, R, root, lane);
            } else {
                const long long t_dis = clock64();
                ++n_cta_dissolve;
                if (lane == 0) { s_job.type = FAST_JOB_DISSOLVE; s_job.pick = P; }
                __syncwarp();
                named_bar(1, KLPM_FAST_THREADS);
                const FastJob J = s_job;
                fast_job<false>(A, R, J, sh, sr, &s_cnt, &s_memcur);
                root = tour_top(R, lane);
                cy_dissolve += clock64() - t_dis;
            }
        }
    };

    // ================================================================ a given order (klpm_replay): no admission, no pick
    // A decision matters to another one only if both are in one of the starting groups, so the loop runs through the order
    // and makes the decisions of grouped slots; the charge pass does everything else.
    if (A.fixed) {
        const int32_t nfix = *reinterpret_cast<const volatile int32_t*>(A.n_fixed);
        for (int32_t c1 = 0; c1 < nfix && !failed; c1 += 128) {
            int32_t j[4]; bool g[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { const int32_t x = c1 + u * 32 + lane; j[u] = x < nfix ? __ldg(A.fixed + x) : -1; }
#pragma unroll
            for (int u = 0; u < 4; ++u) g[u] = j[u] >= 0 && ((__ldcg(A.gbits + (j[u] >> 5)) >> (j[u] & 31)) & 1u);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                for (unsigned bal = __ballot_sync(FULL_MASK, g[u]); bal; bal &= bal - 1) {
                    const int src = __ffs(bal) - 1;
                    const int32_t slot = __shfl_sync(FULL_MASK, j[u], src);      // slots are the queries in index order here
                    c = c1 + u * 32 + src;
                    mark_done(slot);
                    careful(slot, false, ld_dyn(A.dyn + slot), ld_stat(A.stat + slot));
                    __syncwarp();
                }
            }
        }
        c = n;                                               // nothing is left for the policy loops below
    }

    // ================================================================ arrivals pending: one careful step per decision
    long long tw = INF;                                     // 32 coming arrivals (lane i: slot wb + i)
    int32_t wb = 0;
    if (admitted < n) { tw = lane < n ? __ldg(A.sorted_t + lane) : INF; next_t = __shfl_sync(FULL_MASK, tw, 0); }
    while (c < n && !failed && !(A.list_mode && admitted == n)) {
        // ---- time and arrivals: idle until somebody has arrived, then admit everybody who has
        if (head == admitted && next_t > now) now = next_t;
        while (admitted < n && next_t <= now) {             // (an arrival can be the largest time there is, like the padding)
            const int off = admitted - wb;
            const int cnt = __popc(__ballot_sync(FULL_MASK, lane >= off && wb + lane < n && tw <= now));      // (arrivals are sorted)
            const int32_t a1 = admitted + cnt, ra = wb + lane;
            if (off + cnt == 32 && a1 + 64 < n && __ldg(A.sorted_t + a1 + 64) <= now) {
                // a crowd: gallop, then bisect (lane 0), and the whole CTA admits them
                long long lo = a1 + 65, hi = n;
                if (lane == 0) {
                    long long step = 1;
                    while (lo + step <= hi && __ldg(A.sorted_t + lo + step - 1) <= now) { lo += step; step <<= 1; }
                    if (lo + step < hi) hi = lo + step;
                    while (lo < hi) { const long long mid = (lo + hi) >> 1; if (__ldg(A.sorted_t + mid) <= now) lo = mid + 1; else hi = mid; }
                }
                const int32_t all = (int32_t)__shfl_sync(FULL_MASK, lo, 0);
                if (lane == 0) { s_job.type = FAST_JOB_ADMIT; s_job.a0 = admitted; s_job.a1 = all; }
                __syncwarp();
                named_bar(1, KLPM_FAST_THREADS);
                const FastJob J = s_job;
                fast_job<false>(A, R, J, sh, sr, &s_cnt, &s_memcur);
                root = tour_top(R, lane);
                admitted = all;
            } else {
                // keys only come in: every level above takes the larger of what it holds and the newcomers (one or two leaf blocks)
                const unsigned long long ak = ra >= admitted && ra < a1 ? __ldcg(A.key + ra) : 0ULL;
                const int32_t b0 = admitted >> A.lb_shift, b1 = (a1 - 1) >> A.lb_shift;
                for (int32_t bb = b0; bb <= b1; ++bb) {
                    const unsigned long long km = warp_max64r((ra >> A.lb_shift) == bb ? ak : 0ULL);
                    const unsigned long long p1 = R.t1[bb], p2 = R.t2[bb >> 5], p3 = R.t3[bb >> 10];
                    __syncwarp();
                    R.t1[bb] = km > p1 ? km : p1; R.t2[bb >> 5] = km > p2 ? km : p2; R.t3[bb >> 10] = km > p3 ? km : p3;
                    root = km > root ? km : root;
                    __syncwarp();
                }
                admitted = a1;
            }
            if (admitted >= wb + 32) {
                wb = admitted;
                tw = wb + lane < n ? __ldg(A.sorted_t + wb + lane) : INF;
            }
            next_t = __shfl_sync(FULL_MASK, tw, admitted - wb);
        }
        // ---- pick
        const bool fcfs_turn = A.policy == KLPM_POLICY_FCFS || (A.policy == KLPM_POLICY_KLPM && cyc == 0);
        if (++cyc == A.k) cyc = 0;
        int32_t slot = head;
        if (!fcfs_turn) {
            const unsigned rk = 0xffffffffu - (unsigned)(root & 0xffffffffULL);
            slot = A.pinv ? __ldg(A.pinv + rk) : (int32_t)rk;
        }
        if (slot < 0 || slot >= admitted || slot_done(R, A, slot)) { if (lane == 0) set_status(A.st, RT_ERR_LIMIT, 105); failed = true; break; }   // cannot happen
        // ---- the pick leaves its leaf block: its records and the block's keys travel together, the levels above are read meanwhile
        const int32_t b = slot >> A.lb_shift, i2 = b >> 5, i3 = i2 >> 5;
        const long long r = ((long long)b << A.lb_shift) + lane;
        const unsigned long long kk = r < n ? __ldcg(A.key + r) : 0ULL;
        const FDyn pd = ld_dyn(A.dyn + slot);
        const FStat ps = ld_stat(A.stat + slot);
        const unsigned long long x1 = lane == (b & 31) ? 0ULL : R.t1[(i2 << 5) + lane];
        const unsigned long long x2 = lane == (i2 & 31) ? 0ULL : R.t2[(i3 << 5) + lane];
        const unsigned long long x3 = lane == i3 ? 0ULL : R.t3[lane];
        const unsigned long long o1 = warp_max64r(x1), o2 = warp_max64r(x2), o3 = warp_max64r(x3);
        unsigned long long bm = 0;
        if (r < admitted && r != slot && lane < (1 << A.lb_shift) && !slot_done(R, A, r)) bm = kk;
        for (int32_t u = lane + 32; u < (1 << A.lb_shift); u += 32) {
            const long long r2 = ((long long)b << A.lb_shift) + u;
            if (r2 < admitted && r2 != slot && !slot_done(R, A, r2)) { const unsigned long long k2 = __ldcg(A.key + r2); if (k2 > bm) bm = k2; }
        }
        bm = warp_max64r(bm);
        {
            const unsigned long long v2 = bm > o1 ? bm : o1, v3 = v2 > o2 ? v2 : o2;
            R.t1[b] = bm; R.t2[i2] = v2; R.t3[i3] = v3;     // (every lane stores the same)
            root = v3 > o3 ? v3 : o3;
        }
        mark_done(slot);
        careful(slot, true, pd, ps);
        if (slot == head) advance_head();
        __syncwarp();
    }

    // ---- everybody has arrived: list_run_kernel goes on from here
    if (lane == 0) {
        A.post->c0 = A.fixed ? 0 : failed ? n : c;          // (a given order: everything is charged after the loop)
        A.post->list_c = A.fixed || failed ? n : c;
        A.post->now0 = now; A.post->head = head; A.post->cyc = cyc;
        for (int i = 8; i < 16; ++i) A.post->counters[i] = 0;
    }
    __syncwarp();
    if (lane == 0) {
        long long* cn = A.post->counters;
        cn[0] = n_careful; cn[1] = n_cta_dissolve; cn[2] = 0; cn[3] = 0; cn[4] = 0; cn[5] = 0; cn[6] = 0; cn[7] = cy_dissolve;
    }
    if (lane == 0) { s_job.type = FAST_JOB_EXIT; s_job.a0 = A.list_mode && !failed && c < n; }
    __syncwarp();
    named_bar(1, KLPM_FAST_THREADS);
}

// ------------------------------------------------------------------------------------------------
// List mode: everybody has arrived.  The time of a pick no longer decides who can be picked, so the decisions are a merge
// of two orders that are known: the oldest-first turns take the next unprocessed slot, the longest-match turns the next entry
// of the sorted key list that is unprocessed and whose key has not changed since the sort -- or the root of the
// tournament, which holds the slots whose key has changed, where that is larger.  Which turn is which is fixed by the
// policy.  One CTA goes through the two orders a window at a time (2,048 unprocessed slots, 2,048 list positions) and
// works out who takes what by iteration:
//   * a slot that only one of the two sides has in its window is taken by that side, at the turn that its rank among
//     the side's picks gives it;
//   * a slot that both sides have (a meeting) is taken by whichever reaches it first.  Given for every meeting a guess of
//     who takes it, prefix sums over one bit per slot and side give both its ranks, those both its turns, and those a new
//     guess.  Let T be the earliest turn at which a meeting whose guess has changed would be taken.  Then every decision
//     before T is final: by induction over the turns, the ranks of whoever is taken at t depend only on the guesses of
//     slots that are taken before t.  So every round settles at least one turn more, and a few settle a window;
//   * only where the two orders agree for a stretch (one match length left, ties by arrival) does a round settle just one
//     or two turns: every guess there hangs on the one before.  But then the next decisions are that common order, whoever
//     makes them: R decisions, if the unprocessed slots and the live list entries have their first R elements in common.
// Groups of two and the keys that grow in them take part in the rounds, each prompt by a thread of its own (lane_round), in queues from
// KLPM_LIST_LANE_MIN on.  Any other decision that changes a key or follows from a changed one is a step of warp 0, beside the commit of the
// batch before it: the pick's group has other members, its key sits in the tournament, or the tournament's root beats the list.  The window
// goes on after it; only a group dissolved by the whole CTA takes its memory.  Where most decisions are steps, windows are left for
// stretches in which one warp makes the decisions (list_stretch).
// Decisions are recorded as slots in `order`; the charge pass after the loop computes their outputs.
// What bounds it: the barriers and shared-memory round trips of one CTA: 1,500 cycles per round, twice that where the two orders meet a lot,
// 3,000 to 6,800 per step beside its batch, 4,000 to 13,000 per window.  klpm_run of 32,768
// waiting medium queries, k = 4: 1.00 ms in all; 2.05 with batches of up to 1,024 decisions cut at every decision that touches a group.
// It has 128 registers, which 512 threads leave it, and spills some 200 bytes around the call of list_stretch.
// G: some of the loop's bitmaps live in global memory (queues too long for shared memory).
#define KLPM_LIST_THREADS 512
#define KLPM_LIST_WIN 2048            // (4 per thread, 64 words of one bit each: two per lane of a warp)
#define KLPM_LIST_ROUNDS 16           // rounds on one state of the window before what is settled is committed
#define KLPM_LIST_AGREE 24            // stretches shorter than this are left to the rounds
#define KLPM_LIST_FAR 0x3ffffff
// When windows are left for a stretch of decisions by one warp (list_stretch), and when they are tried again.  A window is given credit, in
// units of 100 cycles: what a stretch takes for the decisions of a batch (100 cycles each, 150 where both sides have turns) less what the batch
// has taken.  Only a batch that ends at a step costs any: without steps a batch is long, or the two orders keep meeting, and then a stretch is
// the slower way (1,200 cycles a decision on 1,000 prompts of eight prefixes of one length; windows 130).
#define KLPM_LIST_CREDIT 100           // at its start
#define KLPM_LIST_CREDIT_MAX 400
#define KLPM_LIST_PASS 20              // a batch
#define KLPM_LIST_ROUND 15             // a round; twice that where both sides have turns
#define KLPM_LIST_STEP 5               // a step (beside what a stretch takes for it as well)
#define KLPM_LIST_BUILD 100            // a new window after a group that the whole CTA dissolves
#define KLPM_LIST_TRIAL 64             // decisions after which a stretch ends that has cost half as much again per decision as the windows before it
#define KLPM_LIST_STRETCH 256          // decisions of a block of a stretch; doubles while the windows after it make fewer than KLPM_LIST_STRETCH_LONG
#define KLPM_LIST_STRETCH_LONG 4096
#define KLPM_LIST_STRETCH_MAX 8192     // decisions after which windows are tried again even if most were steps
#define KLPM_LIST_CALM 48              // a block with fewer steps than one in this many ends the stretch
struct ListLane;
struct ListTaken;
struct ListWin {                      // the window, in the scratch of the sorts
    int32_t* fs;                      // unprocessed slots, oldest first
    int32_t* ls; long long* lk;       // list positions from `cur` on: slot, key as the list holds it
    unsigned* col;                    // meetings: index in fs | position << 16
    int32_t* fp; unsigned* fw;        // per bitmap word from head on: free slots before it, free slots
    uint2 *F, *L;                     // per 32 indices / positions: one bit each, taken by this side (as guessed, for a meeting); such bits before
    unsigned *LF, *LL;                // still there
    unsigned *EF, *EL;                // needs a step of its own
    unsigned* eq;                     // agreement, one bit per rank
    int32_t* cand; short* cand_p;     // slots in groups found in the window, and their list positions
    ListLane* lane; ListTaken* taken; short* unsorted; // in the place of `col` once every thread has its meetings
};
// The prompts of a group of two, and prompts whose key has grown because the other one was processed, are worked out by the same
// rounds, each by a thread of its own (see `lane_round`).
struct alignas(16) ListLane {
    unsigned long long key;           // the key it has, or will have once the other one is processed
    int32_t slot, m2;                 // m2: its match length then
    short fi, lp, jr;                 // index among the oldest-first slots, list position, first list position that its key beats (-1: not in the window)
    unsigned char kind, taken;        // kind 0: none, 1: its key has grown, 2: one of a group of two; taken: guessed to be taken with that key,
    int32_t o, A;                     // at this longest-match turn; longest-match turns that are over when the key grows
};
struct ListTaken { unsigned long long key; int32_t A, o, jr, lane; };
#define KLPM_LIST_LANES 128           // the first half for grown keys, the second for groups of two
#define KLPM_LIST_LANE_MIN 8192        // shorter queues make those decisions as steps: 1,000 queries 65 us, with lanes 121 (where between that and 32,768 the line lies best was not looked for)
#define KLPM_LIST_CAND 288
#define KLPM_LIST_TAKEN (KLPM_LIST_LANES / 2 + KLPM_LIST_LANES / 4)      // guessed to be taken with a grown key at a time, at most: every grown key, one of every group
struct ListShared {
    int32_t n_cand, n_pair, n_grown, n_taken, lane_lim;
    int4 pre[2][4];                              // records of lcp_kernel's pairs for the last four steps found on either side, on their way since then
    int32_t pre_n[2], pre_slot[2][4];
    int32_t head, cur, job, failed;
    int32_t ncol;
    int32_t tot_f, tot_l, ev_f, ev_l, ev_r;      // picks of either side in the window; ranks of the first that needs a step, of the first list entry below the root
    int32_t ix_f, ix_l, ix_r;                    // index / positions of those three
    int32_t tstar[2];
    int32_t step_f, step_l, mate_f, mate;        // what a step took (index, position) and changed (index, slot); -1: nothing
    unsigned long long root;
    int32_t w[KLPM_LIST_THREADS / 32];
    int32_t credit;                              // of the windows (KLPM_LIST_CREDIT)
    unsigned w_clock; int32_t w_c;               // when and at which decision the first of them was begun
    int32_t alone, made, stretch_len;            // 1: a stretch (list_stretch) makes the decisions for now; those of its last call; decisions of its blocks
    int32_t stretch, block, block_steps;         // decisions of the stretch so far; of its block, and those of them that touched a group or a changed key
    long long cn[16];                            // what the loop did (FastPost::counters), kept by thread 0: registers are short here
};
static_assert(KLPM_LIST_WIN * (4 + 4 + 8 + 4) + KLPM_LIST_THREADS * 8 + 9 * (KLPM_LIST_WIN / 32) * 4 + KLPM_LIST_CAND * 6 <= KLPM_FAST_SORT_CAP * 12, "a window fits the sort scratch");
static_assert(KLPM_LIST_LANES * sizeof(ListLane) + KLPM_LIST_TAKEN * (sizeof(ListTaken) + 2) <= KLPM_LIST_WIN * 4, "the lanes fit the place of the meetings");
static_assert(KLPM_LIST_CAND * 6 <= KLPM_LIST_TAKEN * sizeof(ListTaken), "the candidates' pairs fit the place of the taken");

// first set bit of a bitmap of 64 words, or -1.  One warp.
__device__ __forceinline__ int32_t list_first(const unsigned* w, int lane) {
    const unsigned a = w[2 * lane], b = w[2 * lane + 1];
    const unsigned m = __ballot_sync(FULL_MASK, (a | b) != 0u);
    if (!m) return -1;
    const int src = __ffs(m) - 1;
    const unsigned x = __shfl_sync(FULL_MASK, a, src), y = __shfl_sync(FULL_MASK, b, src);
    return src * 64 + (x ? __ffs(x) - 1 : 31 + __ffs(y));
}
// Bits before each word of a bitmap of 64 words; returns the number of set bits.  One warp.
__device__ __forceinline__ int32_t list_prefix(uint2* w, int lane, unsigned* a, unsigned* b, int32_t* before) {
    const uint4 v = reinterpret_cast<uint4*>(w)[lane];
    const int32_t ca = __popc(v.x), both = ca + __popc(v.z);
    int32_t inc = both;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const int32_t o = __shfl_up_sync(FULL_MASK, inc, d); if (lane >= d) inc += o; }
    *a = v.x; *b = v.z; *before = inc - both;
    reinterpret_cast<uint4*>(w)[lane] = make_uint4(v.x, (unsigned)(inc - both), v.z, (unsigned)(inc - both + ca));
    return __shfl_sync(FULL_MASK, inc, 31);
}
// The first of the flagged bits (fa, fb: this lane's two words of the flags, already masked by a, b): its position, and its rank among the
// bits of (a, b).  One warp; position -1: none.
__device__ __forceinline__ int32_t list_event(unsigned fa, unsigned fb, unsigned a, unsigned b, int32_t before, int lane, int32_t* at) {
    const unsigned m = __ballot_sync(FULL_MASK, (fa | fb) != 0u);
    if (!m) { *at = -1; return KLPM_LIST_FAR; }
    int32_t pos, rank;
    if (fa) { const int f = __ffs(fa) - 1; pos = 64 * lane + f; rank = before + __popc(a & ((1u << f) - 1u)); }
    else { const int f = fb ? __ffs(fb) - 1 : 0; pos = 64 * lane + 32 + f; rank = before + __popc(a) + __popc(b & ((1u << f) - 1u)); }
    const int src = __ffs(m) - 1;
    *at = __shfl_sync(FULL_MASK, pos, src);
    return __shfl_sync(FULL_MASK, rank, src);
}
// 16 bytes from global to shared memory without waiting for them
__device__ __forceinline__ void list_fetch16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void list_fetch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The largest key that the tournament holds of leaf block b: of slots that are unprocessed and whose key has changed since the sort, less
// those (`held`, per bitmap word) whose key a lane has.  One warp.
template <class Held>
__device__ __forceinline__ unsigned long long changed_block_max(const FastArgs& A, const FastTour& R, int32_t b, int32_t nwords, int lane, Held held) {
    const int32_t w0 = b << (A.lb_shift - 5), w1 = (b + 1) << (A.lb_shift - 5);
    unsigned long long v = 0;
    for (int32_t w = w0; w < w1 && w < nwords; ++w) {
        unsigned m = bm_ld(R.skip, w, R.g_bits) & ~bm_ld(R.done, w, R.g_done);
        if (m) m &= ~held(w);
        if ((m >> lane) & 1u) { const unsigned long long key = __ldcg(A.key + ((long long)w << 5) + lane); if (key > v) v = key; }
    }
    return warp_max64r(v);
}

// Shared memory of list_run_kernel as in fast_run_kernel: tournament, sort scratch (here also the window), bitmaps.
template <bool G>
__device__ __forceinline__ FastTour list_tour(const FastArgs& A, unsigned char* smem, unsigned long long** sort_keys, int32_t** sort_slots) {
    const int32_t nb1p = (A.nb + 31) & ~31, n2 = nb1p >> 5, n2p = (n2 + 31) & ~31, n3 = n2p >> 5;
    const int32_t nwords = (A.n + 31) >> 5;
    FastTour R;
    R.t1 = reinterpret_cast<unsigned long long*>(smem);
    R.t2 = R.t1 + nb1p;
    R.t3 = R.t2 + n2p;
    R.n2 = n2; R.n3 = n3;
    *sort_keys = R.t3 + 32;
    *sort_slots = reinterpret_cast<int32_t*>(*sort_keys + KLPM_FAST_SORT_CAP);
    unsigned int* s_bits = reinterpret_cast<unsigned int*>(*sort_slots + KLPM_FAST_SORT_CAP);
    R.g_done = !G || A.done_in_smem ? 0 : 1;
    R.g_bits = !G || A.bits_in_smem ? 0 : 1;
    R.done = A.done_in_smem ? s_bits : A.done;
    R.skip = A.bits_in_smem ? s_bits + nwords : A.gskip;
    R.gb = A.bits_in_smem ? s_bits + 2 * nwords : A.gbits;
    R.dirty = nullptr;
    return R;
}
// Slot j of a group of two has been processed, and `rec` (lcp_kernel's pairs) says what becomes of the other prompt: its key grows and goes
// to the tournament, whose root is returned.  One warp.
__device__ __forceinline__ unsigned long long list_dissolve_pair(const FastArgs& A, const FastTour& R, int32_t j, const int4& rec, unsigned long long root, int lane) {
    const int32_t mate = rec.x;
    const unsigned long long key = (unsigned long long)(unsigned)rec.w << 32 | (unsigned)rec.z;
    if (lane == 0) {
        __stcg(reinterpret_cast<int32_t*>(A.dyn + mate) + 2, rec.y);
        __stcg(A.key + mate, key);
        atomicOr(R.skip + (mate >> 5), 1u << (mate & 31));
        atomicAnd(R.gb + (mate >> 5), ~(1u << (mate & 31)));
        atomicAnd(R.gb + (j >> 5), ~(1u << (j & 31)));
    }
    const int32_t b = mate >> A.lb_shift;
    const unsigned long long p1 = R.t1[b], p2 = R.t2[b >> 5], p3 = R.t3[b >> 10];
    __syncwarp();
    R.t1[b] = key > p1 ? key : p1; R.t2[b >> 5] = key > p2 ? key : p2; R.t3[b >> 10] = key > p3 ? key : p3;      // (every lane stores the same)
    __syncwarp();
    return key > root ? key : root;
}
// Decision `at` took slot j of any other group (d, s: its records).  0: nothing to do; 1: dissolved, anything about the members may have
// changed; 2: left to the whole CTA, as *job.  One warp.
__device__ __forceinline__ int list_dissolve_group(const FastArgs& A, const FastTour& R, FastJob* job, int32_t j, int32_t at, const FDyn& d, const FStat& s,
                                                   unsigned long long* root, int lane) {
    if (s.len <= d.m || d.gcount <= 1) return 0;
    FastPick P;
    P.slot = j; P.m = d.m; P.len = s.len; P.ntok = d.ntok; P.x = A.tok + s.soff; P.pos = d.pos; P.vleaf = A.vbase + ((long long)at << 32);
    P.admitted = A.n; P.gstart = d.gstart; P.gcount = d.gcount; P.leaf = -1;
    P.lcp = __ldcg(A.lcp + j);
    const bool small_ = dissolve_is_small(P);
    if (small_) *root = dissolve_small(A, P, R, *root, lane);
    else if (lane == 0) { job->type = FAST_JOB_DISSOLVE; job->pick = P; }
    __syncwarp();
    return small_ ? 1 : 2;
}

// A stretch of decisions by one warp, without a window: for queues, or parts of queues, in which most decisions touch a group or a changed
// key, and where windows settle little.  Two ways, as often as each pays:
//   * warp-wide: the next 32 list entries and the next unprocessed slots side by side, interleaved as the policy says, cut before the first
//     decision that another one could have influenced (a slot in both, a group, a changed key, an entry below the tournament's root): about
//     3,000 cycles for up to 32 decisions;
//   * one decision: 900 cycles, 2,500 to 3,500 where a group is dissolved or the tournament changes (two L2 trips).
// It ends where the whole CTA is needed for a group, after a block of `len` decisions of which few were steps, and after
// KLPM_LIST_STRETCH_MAX decisions in any case.  Queues of 9,000 prompts in replicas of four: 1.45 us a decision; as steps between batches of a window
// 3 us.  (A function of its own: inside the kernel its registers would cost the rounds theirs.)
template <bool G>
__device__ __noinline__ void list_stretch(const FastArgs& __restrict__ A, ListShared& __restrict__ S, FastJob& __restrict__ job_, int32_t c, int32_t cyc) {
    extern __shared__ __align__(16) unsigned char fast_smem[];
    const int lane = threadIdx.x & 31;
    unsigned long long* sh;
    int32_t* s_H;
    const FastTour R = list_tour<G>(A, fast_smem, &sh, &s_H);
    int32_t* const s_E = s_H + 32;
    const int gdone = G ? R.g_done : 0, gbits = G ? R.g_bits : 0;
    const int32_t n = A.n, nwords = (n + 31) >> 5, k = A.k, policy = A.policy;
    const bool use_l = policy == KLPM_POLICY_LPM || (policy == KLPM_POLICY_KLPM && k >= 2);
    const long long* const lk = A.lk;
    const int32_t* const ls = A.ls;
    int32_t* const order = A.order;
    const unsigned t0 = (unsigned)clock();
    int32_t len = S.stretch_len;
    if (S.stretch == 0) {                                   // a new one
        __syncwarp();
        len = c - S.w_c >= KLPM_LIST_STRETCH_LONG ? KLPM_LIST_STRETCH : len < KLPM_LIST_STRETCH_LONG ? 2 * len : len;
        if (lane == 0) S.stretch_len = len;
        __syncwarp();
    }
    const int32_t c_in = c, before = S.stretch;
    const unsigned w_cpd = before == 0 ? (t0 - S.w_clock) / (unsigned)(c > S.w_c ? c - S.w_c : 1) : 0u;      // what the windows before it have cost per decision
    int32_t head = S.head, cur = S.cur, block = S.block, block_steps = S.block_steps, job = 0, groups = 0;
    unsigned long long root = S.root;
    bool end = false, trial = before == 0, failed = false;
    auto bit_of = [&](const unsigned* bm, int32_t slot, int g) -> unsigned { return (bm_ld(bm, slot >> 5, g) >> (slot & 31)) & 1u; };
    auto stale = [&](int32_t s) -> bool { return (((bm_ld(R.done, s >> 5, gdone) | bm_ld(R.skip, s >> 5, gbits)) >> (s & 31)) & 1u) != 0u; };
    // the list 32 entries at a time: lane l holds entry (cur & ~31) + l, the next 32 are on their way
    auto window = [&](int32_t base, long long* wk_, int32_t* ws_) {
        const long long i = (long long)base + lane;
        *wk_ = i < n ? __ldg(lk + i) : 0LL;
        *ws_ = i < n ? __ldg(ls + i) : -1;
    };
    long long wk, nk;
    int32_t ws, ns;
    window(cur & ~31, &wk, &ws);
    window((cur & ~31) + 32, &nk, &ns);
    const int32_t lane_div_k = lane / k;                    // y / k for y = 0..31, looked up by shuffle
    bool one_next = false;                                  // the last warp-wide step stopped before a decision it could not take
    int32_t wait = 0, back = 1;                             // decisions until the next warp-wide step is tried; doubles while it makes fewer than two
    // Up to 32 decisions at once: lane i makes decision c + i.  Returns how many; fewer than two: none, and nothing has changed.
    auto warp_wide = [&]() -> int32_t {
        // oldest-first turns among the next x decisions, for x = lane (f_lo) and x = lane + 1 (f_hi)
        int32_t f_lo, f_hi;
        if (policy == KLPM_POLICY_FCFS) { f_lo = lane; f_hi = lane + 1; }
        else if (policy == KLPM_POLICY_LPM) { f_lo = 0; f_hi = 0; }
        else {
            const int32_t i0 = cyc == 0 ? 0 : k - cyc;
            const int32_t y_lo = lane - i0 - 1, y_hi = lane - i0;
            const int32_t q_lo = __shfl_sync(FULL_MASK, lane_div_k, y_lo > 0 ? y_lo : 0);
            const int32_t q_hi = __shfl_sync(FULL_MASK, lane_div_k, y_hi > 0 ? y_hi : 0);
            f_lo = y_lo >= 0 ? q_lo + 1 : 0;
            f_hi = y_hi >= 0 ? q_hi + 1 : 0;
        }
        // the list entries cur .. cur + 31 that still count
        const int32_t off = (cur & 31) + lane;
        const long long k0 = __shfl_sync(FULL_MASK, wk, off & 31), k1 = __shfl_sync(FULL_MASK, nk, off & 31);
        const int32_t s0 = __shfl_sync(FULL_MASK, ws, off & 31), s1 = __shfl_sync(FULL_MASK, ns, off & 31);
        const long long kk = off < 32 ? k0 : k1;
        const int32_t es = off < 32 ? s0 : s1;
        const unsigned mask = __ballot_sync(FULL_MASK, (long long)cur + lane < n && !stale(es));
        // as many decisions as those entries allow: lane x asks whether x + 1 decisions need no more of them
        const int32_t B0 = __popc(__ballot_sync(FULL_MASK, c + lane < n && (lane + 1) - f_hi <= __popc(mask)));
        if (B0 < 2) return 0;
        const int32_t nF0 = __shfl_sync(FULL_MASK, f_hi, B0 - 1), nL0 = B0 - nF0;
        // the next nF0 unprocessed slots; limF = how many of them can be taken before one is a step
        int32_t hs = -1, hmax0 = -1, limF = nF0;
        if (nF0 > 0) {
            const int32_t w0 = head >> 5;
            const int32_t qk = lane < nF0 ? lane : nF0 - 1;           // lane q looks for the q-th unprocessed slot
            auto free_word = [&](int32_t wi) -> unsigned {            // unprocessed slots of bitmap word wi, from head on
                unsigned w = wi < nwords ? bm_ld(R.done, wi, gdone) : 0xffffffffu;
                if (wi == nwords - 1 && (n & 31)) w |= ~((1u << (n & 31)) - 1u);
                if (wi == w0) w |= (1u << (head & 31)) - 1u;
                return ~w;
            };
            const unsigned f0 = free_word(w0), f1 = free_word(w0 + 1);
            const int32_t c0 = __popc(f0);
            if (c0 + __popc(f1) >= nF0) {                             // the usual case: they are all in the first two words
                hs = qk < c0 ? w0 * 32 + kth_set_bit(f0, qk + 1) : (w0 + 1) * 32 + kth_set_bit(f1, qk - c0 + 1);
            } else {                                                  // up to 32 words: running counts, then a search per lane
                const unsigned fr = free_word(w0 + lane);
                const int32_t cnt = __popc(fr);
                int32_t inc = cnt;
#pragma unroll
                for (int dlt = 1; dlt < 32; dlt <<= 1) { const int32_t o = __shfl_up_sync(FULL_MASK, inc, dlt); if (lane >= dlt) inc += o; }
                if (__shfl_sync(FULL_MASK, inc, 31) < nF0) return 0;
                int L = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) if (__shfl_sync(FULL_MASK, inc, L + step - 1) <= qk) L += step;
                const unsigned frL = __shfl_sync(FULL_MASK, fr, L);
                const int32_t preL = __shfl_sync(FULL_MASK, inc - cnt, L);
                hs = (w0 + L) * 32 + kth_set_bit(frL, qk - preL + 1);
            }
            hmax0 = __shfl_sync(FULL_MASK, hs, nF0 - 1);
            const unsigned badH = __ballot_sync(FULL_MASK, lane < nF0 && ((((use_l ? bm_ld(R.skip, hs >> 5, gbits) : 0u) | bm_ld(R.gb, hs >> 5, gbits)) >> (hs & 31)) & 1u));
            if (badH) limF = __ffs(badH) - 1;
        }
        // limL = how many list entries can be taken before one is a step, could also be an oldest-first pick of this batch, or lies below the root
        const bool ok = (mask >> lane) & 1u;
        const int32_t rank = __popc(mask & ((1u << lane) - 1u));
        int32_t limL = nL0;
        int32_t soft = -1;                                  // slot of the entry that stops the batch, if it is only suspected of being an oldest-first pick too
        {
            const unsigned long long ek = ~((unsigned long long)kk ^ 0x8000000000000000ULL);
            const bool hard = ok && (bit_of(R.gb, es, gbits) || root > ek);
            const unsigned badE = __ballot_sync(FULL_MASK, ok && rank < nL0 && (hard || (es >= head && es <= hmax0)));
            if (badE) {
                const int src = __ffs(badE) - 1;
                limL = __popc(mask & ((1u << src) - 1u));
                if (!__shfl_sync(FULL_MASK, (int)hard, src)) soft = __shfl_sync(FULL_MASK, es, src);
            }
        }
        int32_t B = __popc(__ballot_sync(FULL_MASK, lane < B0 && f_hi <= limF && (lane + 1) - f_hi <= limL));
        if (soft >= 0 && B < B0 && B < 32) {
            // the decision after the batch (lane B's): if it is the longest-match turn that takes that entry and the
            // oldest-first picks made until then all lie before its slot, it becomes the batch's last decision
            const int32_t fl = __shfl_sync(FULL_MASK, f_lo, B), fh = __shfl_sync(FULL_MASK, f_hi, B);
            const int32_t last_h = __shfl_sync(FULL_MASK, hs, fl > 0 ? fl - 1 : 0);
            if (fh == fl && B - fl == limL && fl <= limF && (fl == 0 || last_h < soft)) { ++B; ++limL; }
        }
        if (B < 2) return 0;
        one_next = B < B0 && soft < 0;
        const int32_t nF = __shfl_sync(FULL_MASK, f_hi, B - 1), nL = B - nF;
        const int32_t hmax = nF > 0 ? __shfl_sync(FULL_MASK, hs, nF - 1) : -1;
        if (lane < nF) s_H[lane] = hs;
        int32_t consumed = 0;
        if (nL > 0) {
            consumed = kth_set_bit(mask, nL) + 1;
            if (ok && rank < nL) s_E[rank] = es;
        }
        __syncwarp();
        if (lane < B) {
            const int32_t j = f_hi > f_lo ? s_H[f_lo] : s_E[lane - f_lo];
            atomicOr(R.done + (j >> 5), 1u << (j & 31));
            order[c + lane] = j;
        }
        __syncwarp();
        if (consumed) {
            const int32_t ncur = cur + consumed;
            if ((ncur >> 5) != (cur >> 5)) { wk = nk; ws = ns; window((ncur & ~31) + 32, &nk, &ns); }
            cur = ncur;
        }
        if (nF > 0) head = next_head(R.done, gdone, nwords, n, hmax, lane);
        else if (head < n && bit_of(R.done, head, gdone)) head = next_head(R.done, gdone, nwords, n, head, lane);
        return B;
    };
    while (c < n) {
        int32_t made = 0;
        if (!one_next && wait <= 0) {
            made = warp_wide();
            if (made > 0) back = 1;
            else { wait = back; back = back < 64 ? 2 * back : 64; }
        }
        if (made == 0) {
            if (!one_next) --wait;
            one_next = false;
            made = 1;
            const bool oldest = policy == KLPM_POLICY_FCFS || (policy == KLPM_POLICY_KLPM && cyc == 0);
            int32_t j;
            bool in_tour;
            if (oldest) {
                j = head;
                in_tour = use_l && head < n && bit_of(R.skip, j, gbits) != 0u;
            } else {
                unsigned long long ek = 0;                  // next entry of the list that still counts
                int32_t es = -1;
                while (cur < n) {                           // (a window's 32 entries are examined at once: stale entries come in runs)
                    const int32_t wbase = cur & ~31;
                    const unsigned bal = __ballot_sync(FULL_MASK, lane >= (cur & 31) && (long long)wbase + lane < n && !stale(ws));
                    if (bal) {
                        const int src = __ffs(bal) - 1;
                        cur = wbase + src;
                        ek = ~((unsigned long long)__shfl_sync(FULL_MASK, wk, src) ^ 0x8000000000000000ULL);
                        es = __shfl_sync(FULL_MASK, ws, src);
                        break;
                    }
                    cur = wbase + 32; wk = nk; ws = ns; window(cur + 32, &nk, &ns);
                }
                if (cur > n) cur = n;
                in_tour = root > ek;
                if (in_tour) {
                    const unsigned rk = 0xffffffffu - (unsigned)(root & 0xffffffffULL);
                    j = A.pinv ? __ldg(A.pinv + rk) : (int32_t)rk;
                } else {
                    j = es;
                    ++cur;
                    if ((cur & 31) == 0) { wk = nk; ws = ns; window(cur + 32, &nk, &ns); }
                }
            }
            if (j < 0 || j >= n || bit_of(R.done, j, gdone)) { failed = true; break; }      // cannot happen
            const bool grouped = bit_of(R.gb, j, gbits) != 0u;
            FDyn d; FStat s; int4 rec;                      // (asked for before the tournament is brought up to date)
            if (grouped) { d = ld_dyn(A.dyn + j); s = ld_stat(A.stat + j); rec = __ldg(A.pair + 2LL * j); }
            __syncwarp();
            if (lane == 0) { atomicOr(R.done + (j >> 5), 1u << (j & 31)); order[c] = j; }
            __syncwarp();
            if (in_tour) {
                const int32_t b = j >> A.lb_shift;
                root = tour_set(R, b, changed_block_max(A, R, b, nwords, lane, [](int32_t) -> unsigned { return 0u; }), lane);
                __syncwarp();
            }
            if (j == head) head = next_head(R.done, gdone, nwords, n, j, lane);
            if (grouped) {
                ++groups;
                if (rec.x >= 0) root = list_dissolve_pair(A, R, j, rec, root, lane);
                else job = list_dissolve_group(A, R, &job_, j, c, d, s, &root, lane);
            }
            if (grouped || in_tour) ++block_steps;
        }
        c += made;
        if (policy == KLPM_POLICY_KLPM) cyc = (cyc + made) % k;
        block += made;
        if (block >= len) { end = block_steps * KLPM_LIST_CALM <= block || before + (c - c_in) >= KLPM_LIST_STRETCH_MAX; block = 0; block_steps = 0; }
        if (trial && c - c_in >= KLPM_LIST_TRIAL) {
            trial = false;
            const unsigned cy = __shfl_sync(FULL_MASK, (unsigned)clock() - t0, 0);
            if (2 * (cy / (unsigned)(c - c_in)) > 3 * w_cpd) end = true;
        }
        if (job == 2 || end) break;
    }
    if (lane == 0) {
        if (end) { S.credit = KLPM_LIST_CREDIT; S.w_clock = (unsigned)clock(); S.w_c = c; }
        if (failed) { set_status(A.st, RT_ERR_LIMIT, 107); S.failed = 1; }
        S.head = head; S.cur = cur < n ? cur : n; S.root = root; S.job = job; S.made = c - c_in; S.alone = !end;
        S.stretch = before + (c - c_in); S.block = block; S.block_steps = block_steps;
        S.cn[0] += groups; S.cn[2] += c - c_in; S.cn[13] += c - c_in; S.cn[6] += (unsigned)clock() - t0;
    }
}

template <bool G>
__global__ void __launch_bounds__(KLPM_LIST_THREADS, 1)
list_run_kernel(const __grid_constant__ FastArgs A) {
    extern __shared__ __align__(16) unsigned char fast_smem[];
    __shared__ FastJob s_job;
    __shared__ int s_cnt;
    __shared__ int32_t s_memcur;
    __shared__ ListShared S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = KLPM_LIST_THREADS / 32, WORDS = KLPM_LIST_WIN / 32, PER = KLPM_LIST_WIN / KLPM_LIST_THREADS;
    const int32_t n = A.n;
    int32_t c = A.post->list_c, cyc = A.post->cyc;
    if (c >= n) return;
    const int32_t nb1p = (A.nb + 31) & ~31, n2p = ((nb1p >> 5) + 31) & ~31;
    const int32_t nwords = (n + 31) >> 5;
    unsigned long long* sh;
    int32_t* sr;
    const FastTour R = list_tour<G>(A, fast_smem, &sh, &sr);
    const int gdone = G ? R.g_done : 0, gbits = G ? R.g_bits : 0;
    ListWin W;
    W.lk = reinterpret_cast<long long*>(sh);
    W.fs = reinterpret_cast<int32_t*>(W.lk + KLPM_LIST_WIN);
    W.ls = W.fs + KLPM_LIST_WIN;
    W.col = reinterpret_cast<unsigned*>(W.ls + KLPM_LIST_WIN);
    W.fp = reinterpret_cast<int32_t*>(W.col + KLPM_LIST_WIN);
    W.fw = reinterpret_cast<unsigned*>(W.fp + KLPM_LIST_THREADS);
    W.F = reinterpret_cast<uint2*>(W.fw + KLPM_LIST_THREADS); W.L = W.F + WORDS;
    W.LF = reinterpret_cast<unsigned*>(W.L + WORDS); W.LL = W.LF + WORDS; W.EF = W.LL + WORDS; W.EL = W.EF + WORDS; W.eq = W.EL + WORDS;
    W.cand = reinterpret_cast<int32_t*>(W.eq + WORDS); W.cand_p = reinterpret_cast<short*>(W.cand + KLPM_LIST_CAND);
    W.lane = reinterpret_cast<ListLane*>(W.col); W.taken = reinterpret_cast<ListTaken*>(W.lane + KLPM_LIST_LANES); W.unsorted = reinterpret_cast<short*>(W.taken + KLPM_LIST_TAKEN);
    for (int32_t i = tid; i < nb1p + n2p + 32; i += KLPM_LIST_THREADS) R.t1[i] = 0ULL;
    if (tid == 0) {
        s_memcur = n;
        S.head = A.post->head; S.cur = 0; S.root = 0ULL; S.failed = 0; S.job = 0; S.pre_n[0] = 0; S.pre_n[1] = 0; S.n_taken = 0;
        for (int i = 0; i < 16; ++i) S.cn[i] = 0;
        S.alone = 0; S.credit = KLPM_LIST_CREDIT; S.w_clock = (unsigned)clock(); S.w_c = c; S.stretch_len = KLPM_LIST_STRETCH / 2;
    }
    auto count = [&](int i, long long v) { if (tid == 0) S.cn[i] += v; __syncwarp(); };      // (together again at once: what follows would run for lane 0 and the others in turn)
    if (A.done_in_smem) for (int32_t i = tid; i < nwords; i += KLPM_LIST_THREADS) R.done[i] = c > 0 ? __ldcg(A.done + i) : 0u;
    for (int32_t i = tid; i < nwords; i += KLPM_LIST_THREADS) {
        R.skip[i] = 0u;                                     // (slots whose key has changed since the sort)
        if (A.bits_in_smem) R.gb[i] = __ldcg(A.gbits + i);
    }
    __syncthreads();
    auto bit_of = [&](const unsigned* bm, int32_t slot, int g) -> unsigned { return (bm_ld(bm, slot >> 5, g) >> (slot & 31)) & 1u; };
    auto stale = [&](int32_t s) -> bool { return (((bm_ld(R.done, s >> 5, gdone) | bm_ld(R.skip, s >> 5, gbits)) >> (s & 31)) & 1u) != 0u; };      // the list passes over it
    // ---- turns, counted from the next decision: the t-th oldest-first turn, the u-th longest-match turn, oldest-first turns among x decisions.
    // (a k beyond what a window holds is as good as any such k)
    const bool use_f = A.policy != KLPM_POLICY_LPM;
    const bool use_l = A.policy == KLPM_POLICY_LPM || (A.policy == KLPM_POLICY_KLPM && A.k >= 2);
    const int32_t kk = A.policy == KLPM_POLICY_KLPM ? (A.k < 8192 ? A.k : 8192) : 1;
    int32_t i0 = 0;                                         // the first oldest-first turn
    auto set_i0 = [&]() {
        if (!use_f) i0 = KLPM_LIST_FAR;
        else if (A.policy == KLPM_POLICY_FCFS || cyc == 0) i0 = 0;
        else i0 = A.k - cyc < KLPM_LIST_FAR / 2 ? A.k - cyc : KLPM_LIST_FAR / 2;
    };
    auto per_k1 = [&](int32_t u) -> int32_t { return A.k == 2 ? u : (int32_t)__umulhi((unsigned)u, A.recip_k1); };
    auto f_turn = [&](int32_t t) -> int32_t { return use_f ? i0 + t * kk : KLPM_LIST_FAR; };
    auto l_turn = [&](int32_t u) -> int32_t { return !use_l ? KLPM_LIST_FAR : u < i0 ? u : u + 1 + per_k1(u - i0); };
    auto f_count = [&](int32_t x) -> int32_t { return !use_f || x <= i0 ? 0 : (x - i0 - 1) / kk + 1; };

    // the oldest-first slots worth looking at: twice the turns that 2,048 list entries leave for them
    const int32_t most_f = use_l && A.k > 2 && 2 * KLPM_LIST_WIN / (A.k - 1) + 128 < KLPM_LIST_WIN ? 2 * KLPM_LIST_WIN / (A.k - 1) + 128 : KLPM_LIST_WIN;
    int32_t n_f = 0, n_l = 0;                               // the window: slots, list positions
    bool list_end = false;                                  // it reaches the end of the list
    int32_t w0 = 0, head0 = 0;                              // its first bitmap word and slot
    const int x = tid - 96;                                 // this thread's lane, if 0 <= x < KLPM_LIST_LANES (whole warps)
    const bool laner = x >= 0 && x < KLPM_LIST_LANES;
    int32_t sv_slot = -1, sv_m2 = 0;                        // a grown key, from one window to the next
    unsigned long long sv_key = 0;
    unsigned cv[PER], alive = 0;                            // this thread's meetings; one bit each while both sides still have the slot
#pragma unroll
    for (int r = 0; r < PER; ++r) cv[r] = 0u;
    // index of a slot among the window's oldest-first slots, or -1
    auto index_of = [&](int32_t s) -> int32_t {
        if (!use_f || n_f == 0 || s < head0 || s > W.fs[n_f - 1]) return -1;
        const int32_t wl = (s >> 5) - w0;
        const unsigned f = W.fw[wl];
        const int32_t phi = W.fp[wl] + __popc(f & ((1u << (s & 31)) - 1u));
        return ((f >> (s & 31)) & 1u) && phi < n_f ? phi : -1;
    };
    auto no_event = [&](int32_t fi, int32_t lp) {
        if (fi >= 0) atomicAnd(&W.EF[fi >> 5], ~(1u << (fi & 31)));
        if (lp >= 0) atomicAnd(&W.EL[lp >> 5], ~(1u << (lp & 31)));
    };
    auto lane_bar = [&]() { named_bar(2, KLPM_LIST_LANES); };
    // Everything about the window's slots again, after a group has been dissolved.
    auto refresh = [&]() {
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int w = warp + NW * r, i = w * 32 + lane;
            const bool hf = (W.LF[w] >> lane) & 1u, hl = (W.LL[w] >> lane) & 1u;
            const int32_t sf = hf ? W.fs[i] : 0, sl = hl ? W.ls[i] : 0;
            const bool in_f = hf && !bit_of(R.done, sf, gdone), in_l = hl && !stale(sl);
            const unsigned lf = __ballot_sync(FULL_MASK, in_f), ll = __ballot_sync(FULL_MASK, in_l);
            const unsigned ef = __ballot_sync(FULL_MASK, in_f && ((use_l ? bit_of(R.skip, sf, gbits) : 0u) | bit_of(R.gb, sf, gbits)));
            const unsigned el = __ballot_sync(FULL_MASK, in_l && bit_of(R.gb, sl, gbits));
            if (lane == 0) { W.LF[w] = lf; W.F[w].x &= lf; W.EF[w] = ef; W.LL[w] = ll; W.L[w].x &= ll; W.EL[w] = el; }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            if (!((alive >> r) & 1u)) continue;
            const int32_t i = (int32_t)(cv[r] & 0xffffu), p = (int32_t)(cv[r] >> 16);
            const bool lf = (W.LF[i >> 5] >> (i & 31)) & 1u, ll = (W.LL[p >> 5] >> (p & 31)) & 1u;
            if (lf && ll) continue;
            alive &= ~(1u << r);
            if (lf) atomicOr(&W.F[i >> 5].x, 1u << (i & 31));      // its list entry has gone stale: the oldest-first side has it alone
        }
        if (laner && W.lane[x].kind) no_event(W.lane[x].fi, W.lane[x].lp);
        __syncthreads();
    };
    // The lanes of a new window: the grown keys kept from the last one, and both prompts of the groups of two that have one in the window.
    // What finds no lane goes on as before: a grown key to the tournament, a group as an event.
    auto lanes = [&]() {
        const int32_t n_cand = S.n_cand <= KLPM_LIST_CAND && n >= KLPM_LIST_LANE_MIN ? S.n_cand : 0;      // (too many to know all positions: none)
        if (n_cand == 0 && !__syncthreads_or(sv_slot >= 0)) { if (laner) W.lane[x].kind = 0; __syncthreads(); return; }
        int32_t* const low = reinterpret_cast<int32_t*>(W.taken);              // per candidate: the smaller slot of its pair (no key is guessed to be taken yet)
        if (laner) W.lane[x].kind = 0;
        if (tid < WORDS) W.eq[tid] = 0u;
        short* const place = reinterpret_cast<short*>(low + KLPM_LIST_CAND);    // and, of the first of them, the pair's number
        int32_t mine = -1, mate = -1, lead = 0;
        int4 rec = make_int4(-2, 0, 0, 0), back = rec;
        if (tid < n_cand) {
            mine = W.cand[tid];
            rec = __ldg(A.pair + 2LL * mine); back = __ldg(A.pair + 2LL * mine + 1);
            mate = rec.x;
            low[tid] = mate < 0 ? -1 : mine < mate ? mine : mate;
        }
        __syncthreads();
        if (sv_slot >= 0 && !bit_of(R.done, sv_slot, gdone)) {
            const int32_t at = atomicAdd(&S.n_grown, 1);
            if (at < KLPM_LIST_LANES / 2) {
                ListLane l;
                l.key = sv_key; l.slot = sv_slot; l.m2 = sv_m2; l.fi = (short)index_of(sv_slot); l.lp = -1; l.jr = -1; l.o = 0; l.A = 0; l.kind = 1; l.taken = 0;
                W.lane[at] = l;
            } else {
                const int32_t b = sv_slot >> A.lb_shift;
                atomicMax(R.t1 + b, sv_key); atomicMax(R.t2 + (b >> 5), sv_key); atomicMax(R.t3 + (b >> 10), sv_key); atomicMax(&S.root, sv_key);
            }
        }
        if (mate >= 0) {
            const int32_t lo = low[tid];
            while (low[lead] != lo) ++lead;                 // (at the latest its own)
            if (lead == tid) {
                const int32_t at = atomicAdd(&S.n_pair, 1);
                place[tid] = (short)at;
                if (at < KLPM_LIST_LANES / 4) {
                    ListLane l;
                    l.lp = -1; l.jr = -1; l.o = 0; l.A = 0; l.kind = 2; l.taken = 0; l.m2 = rec.y;
                    l.slot = mine; l.fi = (short)index_of(mine); l.key = (unsigned long long)(unsigned)back.w << 32 | (unsigned)back.z;
                    W.lane[KLPM_LIST_LANES / 2 + 2 * at] = l;
                    l.slot = mate; l.fi = (short)index_of(mate); l.key = (unsigned long long)(unsigned)rec.w << 32 | (unsigned)rec.z;
                    W.lane[KLPM_LIST_LANES / 2 + 2 * at + 1] = l;
                }
            }
        }
        __syncthreads();
        if (mate >= 0 && W.cand_p[tid] >= 0 && place[lead] < KLPM_LIST_LANES / 4) {
            ListLane* const l = W.lane + KLPM_LIST_LANES / 2 + 2 * place[lead];
            l[l[0].slot == mine ? 0 : 1].lp = W.cand_p[tid];
        }
        __syncthreads();
        if (laner && W.lane[x].kind) {
            ListLane& l = W.lane[x];
            const long long rk = (long long)(~l.key ^ 0x8000000000000000ULL);      // (the list holds ~key with the top bit flipped, ascending)
            int32_t lo = 0, hi = n_l;
            while (lo < hi) { const int32_t mid = (lo + hi) >> 1; if (W.lk[mid] > rk) hi = mid; else lo = mid + 1; }
            l.jr = (short)lo;
            no_event(l.fi, l.lp);
            if (l.fi >= 0) atomicOr(&W.eq[l.fi >> 5], 1u << (l.fi & 31));
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PER; ++r) { const int32_t i = (int32_t)(cv[r] & 0xffffu); if (((alive >> r) & 1u) && ((W.eq[i >> 5] >> (i & 31)) & 1u)) alive &= ~(1u << r); }
        __syncthreads();
    };
    auto build = [&]() {
        int32_t cur = S.cur;
        const int32_t head = S.head;
        long long key_in[PER];
        int32_t slot_in[PER];
        unsigned live_l = 0;                                // which of them still count
        w0 = head >> 5; head0 = head;
        n_f = 0;
        if (use_l) {
            for (;;) {                                      // (a stretch of the list without a live entry is passed over)
                int any = 0;
                live_l = 0;
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const long long idx = (long long)cur + tid + KLPM_LIST_THREADS * r;
                    slot_in[r] = idx < n ? __ldg(A.ls + idx) : -1;
                    key_in[r] = idx < n ? __ldg(A.lk + idx) : 0LL;
                }
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const int w = warp + NW * r;
                    const bool in = slot_in[r] >= 0 && !stale(slot_in[r]);
                    if (in) live_l |= 1u << r;
                    const unsigned live = __ballot_sync(FULL_MASK, in), ev = __ballot_sync(FULL_MASK, in && bit_of(R.gb, slot_in[r], gbits));
                    if (lane == 0) { W.LL[w] = live; W.L[w].x = live; W.EL[w] = ev; }
                    any |= live != 0u;
                }
                if (__syncthreads_or(any) || (long long)cur + KLPM_LIST_WIN >= n) break;
                cur += KLPM_LIST_WIN;
            }
            n_l = n - cur < KLPM_LIST_WIN ? n - cur : KLPM_LIST_WIN;
            list_end = (long long)cur + KLPM_LIST_WIN >= n;
#pragma unroll
            for (int r = 0; r < PER; ++r) { W.ls[tid + KLPM_LIST_THREADS * r] = slot_in[r]; W.lk[tid + KLPM_LIST_THREADS * r] = key_in[r]; }
        } else {
            if (tid < WORDS) { W.LL[tid] = 0u; W.L[tid].x = 0u; W.EL[tid] = 0u; }
            n_l = 0; list_end = true;
        }
        if (use_f) {
            const int32_t wi = w0 + tid;
            unsigned w = wi < nwords ? bm_ld(R.done, wi, gdone) : 0xffffffffu;
            if (wi == nwords - 1 && (n & 31)) w |= ~((1u << (n & 31)) - 1u);
            if (wi == w0) w |= (1u << (head & 31)) - 1u;
            const unsigned fr = ~w;
            const int32_t cnt = __popc(fr);
            int32_t inc = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const int32_t o = __shfl_up_sync(FULL_MASK, inc, d); if (lane >= d) inc += o; }
            if (lane == 31) S.w[warp] = inc;
            __syncthreads();
            int32_t before = 0, all = 0;
#pragma unroll
            for (int v = 0; v < NW; ++v) { const int32_t x = S.w[v]; if (v < warp) before += x; all += x; }
            W.fp[tid] = before + inc - cnt; W.fw[tid] = fr;
            n_f = all < most_f ? all : most_f;
            __syncthreads();
            for (int32_t wl = warp; wl < KLPM_LIST_THREADS && W.fp[wl] < n_f; wl += NW) {
                const unsigned f = W.fw[wl];
                if ((f >> lane) & 1u) {
                    const int32_t rank = W.fp[wl] + __popc(f & ((1u << lane) - 1u));
                    if (rank < n_f) W.fs[rank] = (w0 + wl) * 32 + lane;
                }
            }
        } else if (tid < WORDS) { W.LF[tid] = 0u; W.F[tid].x = 0u; W.EF[tid] = 0u; }
        if (tid == 0) { S.ncol = 0; S.cur = cur; S.n_cand = 0; S.n_pair = 0; S.n_grown = 0; S.n_taken = 0; }
        __syncthreads();
        auto candidate = [&](int32_t s, int32_t pos) {
            const int32_t at = atomicAdd(&S.n_cand, 1);
            if (at < KLPM_LIST_CAND) { W.cand[at] = s; W.cand_p[at] = (short)pos; asm volatile("prefetch.global.L1 [%0];" ::"l"(A.pair + 2LL * s)); }
        };
        if (use_f) {
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int w = warp + NW * r, i = w * 32 + lane;
                const bool in = i < n_f;
                const int32_t s = in ? W.fs[i] : 0;
                const unsigned live = __ballot_sync(FULL_MASK, in);
                const unsigned ev = __ballot_sync(FULL_MASK, in && ((use_l ? bit_of(R.skip, s, gbits) : 0u) | bit_of(R.gb, s, gbits)));
                if (lane == 0) { W.LF[w] = live; W.F[w].x = live; W.EF[w] = ev; }
                if (in && bit_of(R.gb, s, gbits)) candidate(s, -1);
            }
        }
        if (use_l) {
#pragma unroll
            for (int r = 0; r < PER; ++r)
                if (((live_l >> r) & 1u) && bit_of(R.gb, slot_in[r], gbits)) candidate(slot_in[r], tid + KLPM_LIST_THREADS * r);
        }
        if (use_f && use_l && n_f > 0) {                    // the meetings
            const int32_t hmax = W.fs[n_f - 1];
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int32_t s = slot_in[r];
                bool met = ((live_l >> r) & 1u) && s >= head && s <= hmax;
                int32_t phi = 0;
                if (met) {
                    const int32_t wl = (s >> 5) - w0;       // (below KLPM_LIST_THREADS: hmax is)
                    const unsigned f = W.fw[wl];
                    phi = W.fp[wl] + __popc(f & ((1u << (s & 31)) - 1u));
                    met = ((f >> (s & 31)) & 1u) && phi < n_f;
                }
                const unsigned bal = __ballot_sync(FULL_MASK, met);
                if (bal) {
                    int32_t base = 0;
                    if (lane == __ffs(bal) - 1) base = atomicAdd(&S.ncol, __popc(bal));
                    base = __shfl_sync(FULL_MASK, base, __ffs(bal) - 1);
                    if (met) W.col[base + __popc(bal & ((1u << lane) - 1u))] = (unsigned)phi | (unsigned)(tid + KLPM_LIST_THREADS * r) << 16;
                }
            }
        }
        if (use_l) {                                        // the list behind this window, into L1 for the next one
            const long long at = (long long)cur + KLPM_LIST_WIN;
            if (tid < 128) { const long long e = at + tid * 16; if (e < n) asm volatile("prefetch.global.L1 [%0];" ::"l"(A.lk + e)); }
            else if (tid < 192) { const long long e = at + (tid - 128) * 32; if (e < n) asm volatile("prefetch.global.L1 [%0];" ::"l"(A.ls + e)); }
        }
        __syncthreads();
        const int32_t ncol = S.ncol;
        alive = 0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int32_t at = tid + KLPM_LIST_THREADS * r;
            cv[r] = at < ncol ? W.col[at] : 0u;
            if (at < ncol) alive |= 1u << r;
        }
        __syncthreads();
        lanes();
    };
    // Prefix sums of the guesses, and what ends a batch: the rank of the first pick of either side that needs a step, and of the first
    // list entry that the tournament's root beats.  The caller synchronises.
    auto ranks = [&]() {
        if (warp < 2) {
            unsigned a, b;
            int32_t before, at;
            uint2* const V = warp == 0 ? W.F : W.L;
            const unsigned* const E = warp == 0 ? W.EF : W.EL;
            const int32_t tot = list_prefix(V, lane, &a, &b, &before);
            const int32_t ev = list_event(E[2 * lane] & a, E[2 * lane + 1] & b, a, b, before, lane, &at);
            if (lane == 0) {
                if (warp == 0) { S.tot_f = tot; S.ev_f = ev; S.ix_f = at; }
                else { S.tot_l = tot; S.ev_l = ev; S.ix_l = at; }
                if (at >= 0) {
                    const int32_t slot = warp == 0 ? W.fs[at] : W.ls[at];
                    const int32_t k = S.pre_n[warp];
                    if (k == 0 || S.pre_slot[warp][(k - 1) & 3] != slot) {
                        if ((k & 3) == 0) list_fetch_wait();
                        S.pre_slot[warp][k & 3] = slot; S.pre_n[warp] = k + 1;
                        list_fetch16(&S.pre[warp][k & 3], A.pair + 2LL * slot);
                    }
                }
            }
        } else if (warp == 2) {
            // the list holds ~key with the top bit flipped, ascending: the first position with a larger value than the root's
            int32_t jr = n_l;
            const unsigned long long root = S.root;
            if (root != 0ULL && n_l > 0) {
                const long long rk = (long long)(~root ^ 0x8000000000000000ULL);
                const int32_t p = 64 * lane + 63 < n_l ? 64 * lane + 63 : n_l - 1;
                const unsigned m = __ballot_sync(FULL_MASK, W.lk[p] > rk);
                if (m) {
                    const int32_t b0 = 64 * (__ffs(m) - 1), q = b0 + lane;
                    const unsigned m0 = __ballot_sync(FULL_MASK, q < n_l && W.lk[q] > rk), m1 = __ballot_sync(FULL_MASK, q + 32 < n_l && W.lk[q + 32] > rk);
                    jr = m0 ? b0 + __ffs(m0) - 1 : m1 ? b0 + 31 + __ffs(m1) : n_l;
                }
            }
            // its picks before jr (the prefix sums are another warp's, at the same time)
            int32_t cnt = 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int32_t w = 2 * lane + u, left = jr - 32 * w;
                if (left > 0) cnt += __popc(left >= 32 ? W.L[w].x : W.L[w].x & ((1u << left) - 1u));
            }
            cnt = (int32_t)__reduce_add_sync(FULL_MASK, (unsigned)cnt);
            if (lane == 0) S.ix_r = jr;
            if (lane == 0) S.ev_r = root != 0ULL && (jr < n_l || list_end) ? cnt : KLPM_LIST_FAR;
        }
    };
    // The longest-match turn at which the list entry at position p, of rank r, is reached: a grown key that beats it goes first if it has
    // grown by then.  (They are sorted by when they grow.)
    auto ord = [&](int32_t r, int32_t p) -> int32_t {
        const int32_t nt = S.n_taken;
        for (int32_t u = 0; u < nt && W.taken[u].A <= r; ++u) r += W.taken[u].jr <= p;
        return r;
    };
    auto list_rank = [&](int32_t p) -> int32_t { const uint2 l = W.L[p >> 5]; return (int32_t)l.y + __popc(l.x & ((1u << (p & 31)) - 1u)); };
    auto l_count = [&](int32_t t) -> int32_t { return use_l ? t - f_count(t) : 0; };
    // Before the threads look at their meetings: the slots that are guessed to be taken with a grown key, by when it grows.
    auto lane_turns = [&]() {
        ListLane& l = W.lane[x];
        if (x == 0) S.n_taken = 0;
        lane_bar();
        int32_t at = -1;
        if (l.kind && l.taken) {                            // (never more than there is room for: of a group at most one has grown)
            at = atomicAdd(&S.n_taken, 1);
            W.unsorted[at] = (short)x;
        }
        lane_bar();
        const int32_t nt = S.n_taken;
        if (x == 0 && nt > S.cn[4]) S.cn[4] = nt;
        __syncwarp();
        if (at >= 0) {
            int32_t rank = 0;
            for (int32_t u = 0; u < nt; ++u) { const int32_t a = W.lane[W.unsorted[u]].A; rank += a < l.A || (a == l.A && u < at); }
            ListTaken t; t.key = l.key; t.A = l.A; t.o = l.o; t.jr = l.jr; t.lane = x;
            W.taken[rank] = t;
        }
        lane_bar();
    };
    // A lane's turns from the guesses, and its new guess.  Of a group of two, whoever is reached first is an ordinary pick of either side.
    // The other one's key grows at that moment: A longest-match turns are over by then.  It is taken before the first list entry
    // that it beats, but not before it has grown, and after the grown keys that are larger and have grown by its turn.
    // (The proof of the rounds holds for it too: its turn depends on slots that are taken before it only, and where its guess changes T is
    // no later than any turn, old or new, from which on it matters to others.)
    int32_t lane_tf = KLPM_LIST_FAR, lane_tl = KLPM_LIST_FAR, lane_o = 0, lane_A = 0;
    unsigned lane_now = 0, lane_new = 0;                    // guesses: 1 oldest-first, 2 list entry, 4 grown key
    auto lane_round = [&]() -> int32_t {
        const ListLane l = W.lane[x];
        int32_t tf = KLPM_LIST_FAR, tl = KLPM_LIST_FAR, tr = KLPM_LIST_FAR, at = 0, o = 0;
        unsigned now_ = 0;
        if (l.kind) {
            if (l.fi >= 0) { const uint2 f = W.F[l.fi >> 5]; tf = f_turn((int32_t)f.y + __popc(f.x & ((1u << (l.fi & 31)) - 1u))); if ((f.x >> (l.fi & 31)) & 1u) now_ |= 1u; }
            if (l.lp >= 0) { tl = l_turn(ord(list_rank(l.lp), l.lp)); if ((W.L[l.lp >> 5].x >> (l.lp & 31)) & 1u) now_ |= 2u; }
            if (l.taken) now_ |= 4u;
        }
        const int32_t t1 = tf < tl ? tf : tl, tm = __shfl_xor_sync(FULL_MASK, t1, 1);
        const bool grown = l.kind == 1 || (l.kind == 2 && tm < t1);
        const int32_t r0 = !l.kind || !use_l ? 0 : l.jr < n_l ? list_rank(l.jr) : S.tot_l;      // list picks before the first entry that its key beats
        if (grown && use_l && (l.jr < n_l || list_end)) {
            if (l.kind == 2) at = l_count(tm + 1);
            o = r0;
            int32_t o2 = at;
            const int32_t nt = S.n_taken;
            for (int32_t u = 0; u < nt; ++u) {
                const ListTaken t = W.taken[u];
                if (t.A > o && t.A > o2) break;
                if (t.lane == x || t.key < l.key) continue;
                if (t.A <= o) ++o;
                if (t.A <= o2 && t.o >= at) ++o2;
            }
            if (o2 > o) o = o2;
            tr = l_turn(o);
        }
        unsigned new_ = 0;
        if (l.kind) {
            const int32_t other = grown ? tr : tl;
            if (l.fi >= 0 && (tf < other || other >= KLPM_LIST_FAR)) new_ = 1u;
            else if (other < KLPM_LIST_FAR) new_ = grown ? 4u : 2u;
        }
        int32_t best = KLPM_LIST_FAR;
        if (new_ != now_ || ((new_ & 4u) && (o != l.o || at != l.A))) {
            // (with its grown key it matters to turns after it has grown, of entries that it beats)
            best = t1 < tr ? t1 : tr;
            if (new_ & 4u) { const int32_t w = l_turn(r0 > at ? r0 : at); if (w < best) best = w; }
            if (now_ & 4u) { const int32_t e = r0 > l.A ? r0 : l.A, w = l_turn(l.o < e ? l.o : e); if (w < best) best = w; }
        }
        lane_tf = tf; lane_tl = tl; lane_o = o; lane_A = at; lane_now = now_; lane_new = new_;
        return best;
    };
    auto take = [&](int32_t slot, int32_t at) {
        atomicOr(R.done + (slot >> 5), 1u << (slot & 31));
        A.order[c + at] = slot;
    };
    // Warp 0: one decision that needs a step -- the oldest slot (kind 0), the next list entry (1) or the tournament's root (2).
    // `at`: its number.  Other warps commit the batch before it at the same time.  What both change is changed by atomics.  What a step
    // reads of the bitmaps does not depend on how far the commit is: it looks at the pick and the members of its group, which are events
    // and so not in the batch, and in the pick's leaf block at slots whose key has changed.  No commit beside such a look takes or marks
    // one (a changed key is an event too, and where lanes hold some the step comes after the commit): none of the bits in motion is asked for.
    auto one_step = [&](int kind, int32_t at) {
        const unsigned t0 = (unsigned)clock();
        unsigned long long root = S.root;
        int32_t j;
        bool from_lane = false;
        if (kind == 2) {
            const unsigned rk = 0xffffffffu - (unsigned)(root & 0xffffffffULL);
            unsigned long long best = 0;                    // a grown key may be larger still
            int32_t at_lane = -1;
#pragma unroll
            for (int u = 0; u < KLPM_LIST_LANES / 32; ++u) { const ListLane& l = W.lane[32 * u + lane]; if (l.kind == 1 && l.key > best) { best = l.key; at_lane = 32 * u + lane; } }
            const unsigned long long top = warp_max64r(best);
            const bool other = top > root;
            if (other) {
                const int src = __ffs(__ballot_sync(FULL_MASK, best == top)) - 1;
                at_lane = __shfl_sync(FULL_MASK, at_lane, src);
                j = W.lane[at_lane].slot;
                __syncwarp();
                if (lane == 0) W.lane[at_lane].kind = 0;
                from_lane = true;
            } else j = A.pinv ? __ldg(A.pinv + rk) : (int32_t)rk;
        } else j = kind == 0 ? W.fs[S.ix_f] : W.ls[S.ix_l];
        if (j < 0 || j >= n || bit_of(R.done, j, gdone)) { if (lane == 0) { set_status(A.st, RT_ERR_LIMIT, 107); S.failed = 1; } return; }   // cannot happen
        const bool in_tour = (kind == 2 && !from_lane) || (kind == 0 && use_l && bit_of(R.skip, j, gbits) != 0u);      // its key changed after the sort
        const bool grouped = bit_of(R.gb, j, gbits) != 0u;
        const int32_t step_f = kind == 0 ? S.ix_f : index_of(j);
        int32_t mate_f = -1, mate_s = -1, job = 0;
        __syncwarp();
        if (lane == 0) {
            atomicOr(R.done + (j >> 5), 1u << (j & 31));
            A.order[at] = j;
        }
        __syncwarp();
        if (in_tour) {                                      // its leaf block's largest changed key, without it
            const bool with_lanes = S.n_pair > 0 || S.n_grown > 0;
            root = tour_set(R, j >> A.lb_shift, changed_block_max(A, R, j >> A.lb_shift, nwords, lane, [&](int32_t w) -> unsigned {
                if (!with_lanes) return 0u;
                unsigned m = 0;
#pragma unroll
                for (int u = 0; u < KLPM_LIST_LANES / 32; ++u) { const ListLane& l = W.lane[32 * u + lane]; if (l.kind == 1 && (l.slot >> 5) == w) m |= 1u << (l.slot & 31); }
                return __reduce_or_sync(FULL_MASK, m);
            }), lane);
            __syncwarp();
        }
        if (grouped) {
            int4 rec;
            const int last = kind < 2 ? (S.pre_n[kind] - 1) & 3 : 0;      // (found by the round before this step)
            if (kind < 2 && S.pre_slot[kind][last] == j) rec = S.pre[kind][last];
            else rec = __ldg(A.pair + 2LL * j);
            if (rec.x >= 0) {                               // one other prompt, and what becomes of it is known
                mate_s = rec.x;
                mate_f = index_of(mate_s);
                root = list_dissolve_pair(A, R, j, rec, root, lane);
            } else job = list_dissolve_group(A, R, &s_job, j, at, ld_dyn(A.dyn + j), ld_stat(A.stat + j), &root, lane);
        }
        if (lane == 0) {
            if (job == 2) S.credit -= KLPM_LIST_BUILD;
            S.cn[13] += 1; S.cn[0] += grouped; S.cn[15] += (unsigned)clock() - t0;      // (here and not where they happen: a branch of one lane before the dissolve has it run for lane 0 and the others in turn)
            S.root = root; S.job = job; S.step_f = step_f; S.step_l = kind == 1 ? S.ix_l : -1; S.mate_f = mate_f; S.mate = mate_s;
            if (step_f >= 0) { atomicAnd(&W.LF[step_f >> 5], ~(1u << (step_f & 31))); atomicAnd(&W.F[step_f >> 5].x, ~(1u << (step_f & 31))); }
            if (mate_f >= 0) {
                atomicOr(&W.F[mate_f >> 5].x, 1u << (mate_f & 31));
                if (use_l) atomicOr(&W.EF[mate_f >> 5], 1u << (mate_f & 31));
                else atomicAnd(&W.EF[mate_f >> 5], ~(1u << (mate_f & 31)));
            }
        }
    };
    // What the step leaves to do for the window, every thread: the list entries of the two slots, and their meetings.
    auto after_step = [&]() {
        const int32_t sf = S.step_f, mf = S.mate_f, ms = S.mate;
        int32_t js = -2;
        if (sf >= 0) js = W.fs[sf];
        else if (S.step_l >= 0) js = W.ls[S.step_l];
        if (use_l) {
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int32_t i = tid + KLPM_LIST_THREADS * r, s = W.ls[i];
                if (s >= 0 && (s == js || s == ms)) { atomicAnd(&W.LL[i >> 5], ~(1u << (i & 31))); atomicAnd(&W.L[i >> 5].x, ~(1u << (i & 31))); }
            }
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                const int32_t i = (int32_t)(cv[r] & 0xffffu);
                if (i == sf || i == mf) alive &= ~(1u << r);
            }
        }
        __syncthreads();
    };
    // Where the two orders stand, for the next window.
    bool built = false;                                     // there is a window
    auto leave = [&]() {
        if (warp == 0) {
            int32_t head = S.head, cur = S.cur;
            if (use_f && n_f > 0) {
                const int32_t i = list_first(W.LF, lane);
                head = i >= 0 ? W.fs[i] : next_head(R.done, gdone, nwords, n, W.fs[n_f - 1], lane);
            }
            if (use_l && n_l > 0) {
                const int32_t j = list_first(W.LL, lane);
                cur += j >= 0 ? j : n_l;
            }
            if (lane == 0) { S.head = head; S.cur = cur; }
        }
        sv_slot = -1;
        if (laner && W.lane[x].kind == 1) { sv_slot = W.lane[x].slot; sv_key = W.lane[x].key; sv_m2 = W.lane[x].m2; }
        built = false;
        __syncthreads();
    };

    bool fresh = true, agree = false;
    int32_t agree_wait = 0, agree_back = 1;                 // batches until agreement is tried again; doubles while it fails
    int32_t idle = 0;                                       // passes in a row without a decision (a new window, and then one must follow)
    while (c < n) {
        if (__builtin_expect(S.job == 2, 0)) {              // a group that the whole CTA dissolves: its sorts use the window's memory
            const unsigned t0 = (unsigned)clock();
            const FastJob J = s_job;
            fast_job<false>(A, R, J, sh, sr, &s_cnt, &s_memcur);
            if (warp == 0) { const unsigned long long r = tour_top(R, lane); if (lane == 0) { S.root = r; S.job = 0; } }
            __syncthreads();
            count(1, 1); count(7, (unsigned)clock() - t0);
        }
        if (__builtin_expect(S.alone, 0)) {
            __syncthreads();                                // (the stretch may take the flag back)
            if (warp == 0) list_stretch<G>(A, S, s_job, c, cyc);
            __syncthreads();
            // (nothing of a window is kept from before a stretch: no register has to hold any of it meanwhile)
#pragma unroll
            for (int r = 0; r < PER; ++r) cv[r] = 0u;
            alive = 0; sv_slot = -1; sv_m2 = 0; sv_key = 0; n_f = 0; n_l = 0; w0 = 0; head0 = 0; list_end = false;
            built = false; fresh = true; agree = false; agree_wait = 0; agree_back = 1; idle = 0;
            const int32_t made = S.made;
            c += made;
            if (A.policy == KLPM_POLICY_KLPM) cyc = (int32_t)(((long long)cyc + made) % A.k);
            if (S.failed) break;
            __syncthreads();
            continue;
        }
        if (++idle > 8 || (fresh && S.cn[8] >= A.max_windows)) { if (tid == 0) set_status(A.st, RT_ERR_LIMIT, 118); break; }      // cannot happen (without the debug setting)
        if (fresh) {
            const unsigned t0 = (unsigned)clock();
            if (built) leave();
            build();
            built = true;
            count(8, 1); count(14, (unsigned)clock() - t0);
            fresh = false;
        }
        set_i0();
        const int32_t left = n - c;
        int32_t B = 0, kind = -1;                           // decisions of this batch; the step that comes next (-1: none)
        int32_t rounds = 0;
        bool lanes_on = false;                              // the commit has changed lanes
        int32_t gone_f = -1, gone_l = -1;
        bool spent = false, late = false;                   // the window holds no more; the step comes after the commit
        if (agree) {
            // ---- the stretch on which both orders agree
            if (tid < WORDS) { W.F[tid].x = W.LF[tid]; W.L[tid].x = W.LL[tid]; W.eq[tid] = 0u; }
            if (tid == 0) S.lane_lim = KLPM_LIST_FAR;
            __syncthreads();
            ranks();
            __syncthreads();
            if (laner) {
                W.lane[x].taken = 0;
                if (W.lane[x].kind == 1) { const int32_t jr = W.lane[x].jr; if (jr < n_l || list_end) atomicMin(&S.lane_lim, jr < n_l ? list_rank(jr) : S.tot_l); }
            }
#pragma unroll
            for (int r = 0; r < PER; ++r) {
                if (!((alive >> r) & 1u)) continue;
                const int32_t i = (int32_t)(cv[r] & 0xffffu), p = (int32_t)(cv[r] >> 16);
                const uint2 f = W.F[i >> 5], l = W.L[p >> 5];
                const int32_t rf = (int32_t)f.y + __popc(f.x & ((1u << (i & 31)) - 1u));
                if (rf == (int32_t)l.y + __popc(l.x & ((1u << (p & 31)) - 1u))) atomicOr(W.eq + (rf >> 5), 1u << (rf & 31));
            }
            list_fetch_wait();
            __syncthreads();
            int32_t run;
            {
                const unsigned a = ~W.eq[2 * lane], b = ~W.eq[2 * lane + 1];
                const unsigned m = __ballot_sync(FULL_MASK, (a | b) != 0u);
                const int src = m ? __ffs(m) - 1 : 0;
                const unsigned x = __shfl_sync(FULL_MASK, a, src), y = __shfl_sync(FULL_MASK, b, src);
                run = !m ? KLPM_LIST_WIN : src * 64 + (x ? __ffs(x) - 1 : 31 + __ffs(y));
            }
            if (run < KLPM_LIST_AGREE) { agree = false; agree_wait = agree_back; agree_back = agree_back < 16 ? 2 * agree_back : 16; }
            else agree_back = 1;
            const int32_t e1 = S.ev_f, e2 = S.ev_l, e3 = S.ev_r;
            B = run < left ? run : left;
            if (e1 < B) B = e1;
            if (e2 < B) B = e2;
            if (e3 < B) B = e3;
            if (S.lane_lim < B) B = S.lane_lim;
            if (B > 0) {
                const bool f_next = use_f && B >= i0 && (B - i0) % kk == 0;
                if (B < left) kind = f_next ? (B == e1 ? 0 : -1) : B == e3 ? 2 : B == S.lane_lim ? -1 : B == e2 ? 1 : -1;
                spent = kind < 0 && B == run && (run == S.tot_f || run == S.tot_l);
                if (kind >= 0 && warp == 0) one_step(kind, c + B);
                else {
                    for (int w = kind >= 0 ? warp - 1 : warp; w < WORDS; w += kind >= 0 ? NW - 1 : NW) {
                        const uint2 f = W.F[w], l = W.L[w];      // (the same slots on both sides)
                        if (f.x && (int32_t)f.y < B) {
                            const int32_t rank = (int32_t)f.y + __popc(f.x & ((1u << lane) - 1u));
                            const bool mine = ((f.x >> lane) & 1u) && rank < B;
                            if (mine) take(W.fs[w * 32 + lane], rank);
                            const unsigned m = __ballot_sync(FULL_MASK, mine);
                            if (lane == 0) { atomicAnd(&W.F[w].x, ~m); atomicAnd(&W.LF[w], ~m); }
                        }
                        if (l.x && (int32_t)l.y < B) {
                            const int32_t rank = (int32_t)l.y + __popc(l.x & ((1u << lane) - 1u));
                            const unsigned m = __ballot_sync(FULL_MASK, ((l.x >> lane) & 1u) && rank < B);
                            if (lane == 0) { atomicAnd(&W.L[w].x, ~m); atomicAnd(&W.LL[w], ~m); }
                        }
                    }
                }
                count(9, 1); count(10, B);
                __syncthreads();
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const int32_t i = (int32_t)(cv[r] & 0xffffu);
                    if (((alive >> r) & 1u) && !((W.LF[i >> 5] >> (i & 31)) & 1u)) alive &= ~(1u << r);
                }
            }
        }
        if (B == 0) {
            // ---- rounds: ranks from the guesses, new guesses from the ranks
            int32_t T = 0, win = 0, ev = 0, e2 = 0, e3 = 0;
            int32_t tf[PER], tl[PER];
            unsigned own = 0;                               // bits 0-3: guessed to go to the oldest-first side, 4-7: to the list
            if (tid == 0) { S.tstar[0] = KLPM_LIST_FAR; S.tstar[1] = KLPM_LIST_FAR; }
            const bool with_lanes = S.n_pair > 0 || S.n_grown > 0;
            for (int it = 0;; ++it) {
                rounds = it + 1;
                ranks();
                __syncthreads();
                int32_t best = KLPM_LIST_FAR;
                if (with_lanes) {
                    if (laner) lane_turns();
                    __syncthreads();
                    if (laner) best = lane_round();
                }
                unsigned flip = 0;
                own = 0;
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    tf[r] = KLPM_LIST_FAR; tl[r] = KLPM_LIST_FAR;
                    if ((alive >> r) & 1u) {
                        const int32_t i = (int32_t)(cv[r] & 0xffffu), p = (int32_t)(cv[r] >> 16);
                        const unsigned bi = 1u << (i & 31), bp = 1u << (p & 31);
                        const uint2 f = W.F[i >> 5], l = W.L[p >> 5];
                        tf[r] = f_turn((int32_t)f.y + __popc(f.x & (bi - 1u)));
                        tl[r] = l_turn(ord((int32_t)l.y + __popc(l.x & (bp - 1u)), p));
                        const bool is_f = (f.x & bi) != 0u, is_l = (l.x & bp) != 0u, to_f = tf[r] < tl[r];
                        if (is_f) own |= 1u << r;
                        if (is_l) own |= 16u << r;
                        if (is_f != to_f) flip |= 1u << r;
                        if (is_l == to_f) flip |= 16u << r;
                        if ((flip >> r) & 0x11u) { const int32_t t = to_f ? tf[r] : tl[r]; if (t < best) best = t; }
                    }
                }
                best = (int32_t)__reduce_min_sync(FULL_MASK, (unsigned)best);
                if (lane == 0 && best < KLPM_LIST_FAR) atomicMin(&S.tstar[it & 1], best);
                list_fetch_wait();
                __syncthreads();
                T = S.tstar[it & 1];
                const int32_t e1 = S.ev_f < KLPM_LIST_FAR ? f_turn(S.ev_f) : KLPM_LIST_FAR;
                e2 = S.ev_l < KLPM_LIST_FAR ? l_turn(ord(S.ev_l, S.ix_l)) : KLPM_LIST_FAR;
                e3 = S.ev_r < KLPM_LIST_FAR ? l_turn(ord(S.ev_r, S.ix_r - 1)) : KLPM_LIST_FAR;      // (at the earliest)
                ev = e1 < e2 ? e1 : e2;
                if (e3 < ev) ev = e3;
                const int32_t wf = f_turn(S.tot_f), wl = l_turn(ord(S.tot_l, KLPM_LIST_WIN));
                win = wf < wl ? wf : wl;
                // (what needs a step, and what the window cannot answer any more, is only known once everything before has been settled)
                if (T > ev || T >= left || T > win || it >= KLPM_LIST_ROUNDS || (it >= 3 && T > 0 && T < 12 * it)) break;
                if (tid == 0) S.tstar[(it + 1) & 1] = KLPM_LIST_FAR;
#pragma unroll
                for (int r = 0; r < PER; ++r) {
                    const int32_t i = (int32_t)(cv[r] & 0xffffu), p = (int32_t)(cv[r] >> 16);
                    if ((flip >> r) & 1u) atomicXor(&W.F[i >> 5].x, 1u << (i & 31));
                    if ((flip >> r) & 16u) atomicXor(&W.L[p >> 5].x, 1u << (p & 31));
                }
                if (with_lanes && laner && W.lane[x].kind) {
                    ListLane& l = W.lane[x];
                    const unsigned d = lane_now ^ lane_new;
                    if (d & 1u) atomicXor(&W.F[l.fi >> 5].x, 1u << (l.fi & 31));
                    if (d & 2u) atomicXor(&W.L[l.lp >> 5].x, 1u << (l.lp & 31));
                    l.taken = lane_new >> 2; l.o = lane_o; l.A = lane_A;
                }
                __syncthreads();
            }
            if (T <= win) win = KLPM_LIST_FAR;
            B = T < ev ? T : ev;
            if (left < B) B = left;
            if (win < B) B = win;
            if (B < left && B == ev && T > ev) kind = e3 == ev ? 2 : e2 == ev ? 1 : 0;
            spent = kind < 0 && B == win;
            if (B == 0 && kind < 0 && !spent) { if (tid == 0) set_status(A.st, RT_ERR_LIMIT, 118); break; }      // cannot happen: a second round settles the first turn
            if (agree_wait > 0) --agree_wait;
            else if (use_f && use_l && T <= ev && T < left && T < 64) agree = true;      // next to nothing settled: do the orders agree?
            const bool beside = kind >= 0 && !(kind != 1 && with_lanes);      // (where a changed key is involved the step looks at the grown keys, and the commit changes those)
            late = kind >= 0 && !beside;
            lanes_on = with_lanes && B > 0;
            if (beside && warp == 0) one_step(kind, c + B);
            else if (B > 0) {
                const int32_t nfb = f_count(B), nlb = B - nfb;
                for (int w = beside ? warp - 1 : warp; w < WORDS; w += beside ? NW - 1 : NW) {
                    const uint2 f = W.F[w], l = W.L[w];
                    if (f.x && (int32_t)f.y < nfb) {
                        const int32_t rank = (int32_t)f.y + __popc(f.x & ((1u << lane) - 1u));
                        const bool mine = ((f.x >> lane) & 1u) && rank < nfb;
                        if (mine) take(W.fs[w * 32 + lane], f_turn(rank));
                        const unsigned m = __ballot_sync(FULL_MASK, mine);
                        if (lane == 0) { atomicAnd(&W.F[w].x, ~m); atomicAnd(&W.LF[w], ~m); }
                    }
                    if (l.x && (int32_t)l.y < nlb) {
                        const int32_t rank = ord((int32_t)l.y + __popc(l.x & ((1u << lane) - 1u)), w * 32 + lane);
                        const bool mine = ((l.x >> lane) & 1u) && rank < nlb;
                        if (mine) take(W.ls[w * 32 + lane], l_turn(rank));
                        const unsigned m = __ballot_sync(FULL_MASK, mine);
                        if (lane == 0) { atomicAnd(&W.L[w].x, ~m); atomicAnd(&W.LL[w], ~m); }
                    }
                }
            }
            if (B > 0) {
#pragma unroll
                for (int r = 0; r < PER; ++r) {             // the other side of a meeting that is over
                    const int32_t i = (int32_t)(cv[r] & 0xffffu), p = (int32_t)(cv[r] >> 16);
                    if (((own >> r) & 1u) && tf[r] < B) { atomicAnd(&W.LL[p >> 5], ~(1u << (p & 31))); alive &= ~(1u << r); }
                    if (((own >> r) & 16u) && tl[r] < B) { atomicAnd(&W.LF[i >> 5], ~(1u << (i & 31))); alive &= ~(1u << r); }
                }
                if (with_lanes && laner) {
                    // this lane's turn, if the batch holds it: by the guesses that the rounds ended with
                    ListLane& l = W.lane[x];
                    const int32_t nlb = l_count(B);
                    unsigned by = 0;                        // which side took it
                    if (l.kind) by = (lane_now & 1u) && lane_tf < B ? 1u : (lane_now & 2u) && lane_tl < B ? 2u : (lane_now & 4u) && l.o < nlb ? 4u : 0u;
                    const int32_t t = by == 1u ? lane_tf : by == 2u ? lane_tl : by == 4u ? l_turn(l.o) : KLPM_LIST_FAR;
                    const int32_t tm = __shfl_xor_sync(FULL_MASK, t, 1);
                    if (by) atomicAdd(reinterpret_cast<unsigned long long*>(&S.cn[3]), 1ULL);
                    if (by) {                               // its marks on the other sides go (the guesses only once everybody has read them)
                        if (by == 4u) take(l.slot, t);
                        if (by != 1u && l.fi >= 0) { atomicAnd(&W.LF[l.fi >> 5], ~(1u << (l.fi & 31))); gone_f = l.fi; }
                        if (l.lp >= 0) { atomicAnd(&W.LL[l.lp >> 5], ~(1u << (l.lp & 31))); gone_l = l.lp; }
                    }
                    if (l.kind == 2 && (by || tm < KLPM_LIST_FAR)) {      // the group is dissolved
                        atomicAnd(R.gb + (l.slot >> 5), ~(1u << (l.slot & 31)));
                        if (tm < t) {                       // the other one came first: its key has grown
                            __stcg(reinterpret_cast<int32_t*>(A.dyn + l.slot) + 2, l.m2);
                            __stcg(A.key + l.slot, l.key);
                            atomicOr(R.skip + (l.slot >> 5), 1u << (l.slot & 31));
                            if (l.lp >= 0) { atomicAnd(&W.LL[l.lp >> 5], ~(1u << (l.lp & 31))); gone_l = l.lp; }
                            l.lp = -1;
                        }
                        l.kind = by ? 0 : 1;
                    } else if (by) l.kind = 0;
                    l.o -= nlb; l.A = l.A > nlb && l.kind == 2 ? l.A - nlb : 0;
                    if (l.o < 0) l.taken = 0;
                }
                count(11, 1); count(12, B); count(5, rounds);
            }
        }
        if (B > 0 || kind >= 0) idle = 0;
        if (tid == 0) {                                     // has this been worth it?
            const int32_t credit = S.credit + (kind < 0 ? B : B - KLPM_LIST_PASS - KLPM_LIST_STEP + (use_f && use_l ? B / 2 - 2 * KLPM_LIST_ROUND * rounds : -KLPM_LIST_ROUND * rounds));
            S.credit = credit < KLPM_LIST_CREDIT_MAX ? credit : KLPM_LIST_CREDIT_MAX;
        }
        __syncwarp();
        c += B;
        if (A.policy == KLPM_POLICY_KLPM) cyc = (int32_t)(((long long)cyc + B) % A.k);
        if (c >= n) break;
        __syncthreads();
        if (lanes_on) {
            if (gone_f >= 0) atomicAnd(&W.F[gone_f >> 5].x, ~(1u << (gone_f & 31)));
            if (gone_l >= 0) atomicAnd(&W.L[gone_l >> 5].x, ~(1u << (gone_l & 31)));
            __syncthreads();
        }
        if (late) { if (warp == 0) one_step(kind, c); __syncthreads(); }
        if (kind >= 0) {
            if (S.failed) break;
            ++c;
            if (A.policy == KLPM_POLICY_KLPM && ++cyc == A.k) cyc = 0;
            if (S.job == 2) {
                refresh();
                leave();
                fresh = true;
            } else if (S.job == 1) refresh();
            else after_step();
        }
        if (spent) fresh = true;
        if (__builtin_expect(S.credit < 0, 0)) {            // windows do not pay here
            __syncthreads();
            if (built) leave();
            if (sv_slot >= 0 && !bit_of(R.done, sv_slot, gdone)) {      // a grown key goes to the tournament
                const int32_t b = sv_slot >> A.lb_shift;
                atomicMax(R.t1 + b, sv_key); atomicMax(R.t2 + (b >> 5), sv_key); atomicMax(R.t3 + (b >> 10), sv_key); atomicMax(&S.root, sv_key);
            }
            if (tid == 0) { S.alone = 1; S.stretch = 0; S.block = 0; S.block_steps = 0; }
            __syncthreads();
        }
    }
    list_fetch_wait();
    __syncthreads();
    if (tid == 0) {
        if (c < n) A.post->c0 = n;                          // gave up: the entries of `order` that were never written are no slots, and nothing is charged
        long long* cn = A.post->counters;
        for (int i = 0; i < 16; ++i) cn[i] += S.cn[i];      // (the last eight are list mode's alone)
    }
}

// The loop on a tree with a budget (and klpm_replay on one).  Every decision is a careful step, and a step has two
// halves that need little of each other, so two warps share it:
//   * warp 0 decides: admits who has arrived, picks, charges, and dissolves the pick's group;
//   * warp 1 keeps the tree: brings the node records up to date as insert_serial would -- cut the edge the match ends
//     in, stamp its node, evict least-recently-used leaves until the uncached tokens fit, add the leaf.  It keeps a
//     window of 32 clock values and who owns them in registers from one decision to the next (lane i: the owner of
//     value wbase + i, and whether it is a leaf that may go).
// While warp 1 works on decision c, warp 0 prepares decision c + 1: admission, the likely pick's records and its leaf
// block's keys are all asked for at once.  Only then does it wait for warp 1; nothing of c + 1 is committed before.  An
// eviction that shortens matches (queries parked in the evicted leaf) is handed back: warp 0 moves those queries and
// prepares the decision afresh.  A pick whose group has other members waits for its new leaf's id before the group is
// dissolved.  The other warps join for work that is worth sharing; so does warp 1, which is idle then.
// The two hand over through named barriers 2 (a job for warp 1) and 3 (its answer), helpers wait at barrier 1.
// What bounds it: the instruction streams of the two warps (4 to 7 cycles an instruction, most of it fixed-latency
// dependencies), no longer the L2 round trips.  120,000 queries on a cold cache with 93,000 evictions: 232 ms = 1.9 us a
// decision (3,800 cycles); one warp doing everything took 441 ms.  12,007 on a warm cache: 32 ms (48.6).
struct LruJob { int32_t type; int32_t hint, m, len, gstart, gcount; int32_t moved; long long vleaf; };   // moved: queries have been parked elsewhere since the last job
struct LruAnswer { int32_t failed, scan, n_small, leaf; int32_t small_v[8]; };
enum { LRU_JOB_EXIT = 0, LRU_JOB_STEP = 1, LRU_JOB_JOIN = 2 };

// Warp 1.  Returns when the loop is over; *out receives the tree's counters.
__device__ __forceinline__ void lru_tree_warp(const FastArgs& A, const FastTour& R, const LruJob* s_tj, LruAnswer* s_ta, const FastJob* s_job,
                                              unsigned long long* sh, int32_t* sr, int* s_cnt, int32_t* s_memcur, int lane) {
    const TreeDev& T = A.T;
    TreeState st = *A.st;
    const long long evictions0 = st.evictions;
    long long wbase = st.lru_cursor, wend = wbase;          // the window's clock values: [wbase, wend)
    int32_t wv = 0;                                         // this lane's owner
    bool wok = false;                                       // it is a leaf and its stamp is this clock value
    // the next leaf to go, its record, its parent's record and how many queries are parked in it: read between two jobs
    int32_t v0 = -1, pk0 = 0;
    LNode rv, rp0;
    rv.parent = 0; rv.depth = 0; rv.len = 0; rv.nchild = 0; rv.last = 0; rv.off = 0;
    rp0 = rv;
    for (;;) {
        {
            const unsigned okm = __ballot_sync(FULL_MASK, wok);
            v0 = -1;
            if (okm) {
                v0 = __shfl_sync(FULL_MASK, wv, __ffs(okm) - 1);
                rv = ld_node(A.node + v0);
                pk0 = __ldcg(A.parked + v0);
                rp0 = ld_node(A.node + rv.parent);
            }
        }
        named_bar(2, 64);
        const LruJob J = *s_tj;
        if (J.type != LRU_JOB_STEP) {
            if (J.type == LRU_JOB_EXIT) break;
            named_bar(1, KLPM_FAST_THREADS);
            const FastJob F = *s_job;
            fast_job<true>(A, R, F, sh, sr, s_cnt, s_memcur);
            continue;
        }
        LruAnswer ans;
        ans.failed = 0; ans.scan = 0; ans.n_small = 0; ans.leaf = -1;
        const int32_t unc = J.len - J.m;
        if (st.clock + 1 >= T.max_clock || st.n_nodes + 2 > T.max_nodes) {           // (the check before the loop rules this out)
            if (lane == 0) { set_status(A.st, RT_ERR_CAPACITY, 114); s_ta->failed = 1; s_ta->scan = 0; s_ta->n_small = 0; s_ta->leaf = -1; }
            __syncwarp();
            named_arrive(3, 64);
            continue;
        }
        const long long clock = ++st.clock;
        LNode ra = ld_node(A.node + J.hint);                // the node the match ends in (its hint; then up)
        if (J.moved && v0 >= 0) pk0 = __ldcg(A.parked + v0);
        if (lane == 0) atomicSub(A.parked + J.hint, 1);
        int32_t a = J.hint;
        while (a != 0 && J.m <= ra.depth) { a = ra.parent; ra = ld_node(A.node + a); }
        const int32_t o = a == 0 ? 0 : J.m - ra.depth;
        int32_t end = a;                                    // the node that ends where the match ends; its record, stored below
        LNode e = ra;
        const bool cut = a != 0 && o < ra.len;
        if (cut) {                                          // a new node takes the upper part of a's edge
            end = (int32_t)st.n_nodes++;
            ++st.live_nodes;
            e.len = o; e.nchild = 1;
            ra.parent = end; ra.depth += o; ra.len -= o; ra.off += o;
            if (lane == 0) st_node(A.node + a, ra);
        }
        if (end != 0) e.last = clock;
        if (wv == end) wok = false;                         // (the node stamped here is safe)
        __syncwarp();
        while (st.tokens_live + unc > T.budget) {
            unsigned okm = __ballot_sync(FULL_MASK, wok);
            while (!okm && wend < clock) {                  // the next 32 clock values
                wbase = wend;
                const long long cc = wbase + lane;
                wv = cc < clock ? T.clock_owner[cc] : 0;
                wend = wbase + 32 < clock ? wbase + 32 : clock;
                wok = false;
                if (wv > 0 && wv != end) { const LNode w = ld_node(A.node + wv); wok = w.nchild == 0 && w.last == cc; }
                okm = __ballot_sync(FULL_MASK, wok);
            }
            if (!okm) {
                if (lane == 0) set_status(A.st, RT_ERR_BUDGET);
                ans.failed = 1; break;
            }
            const int src = __ffs(okm) - 1;
            const int32_t victim = __shfl_sync(FULL_MASK, wv, src);
            const long long stamp = wbase + src;
            bool have_parent = victim == v0;
            if (victim != v0) { rv = ld_node(A.node + victim); pk0 = __ldcg(A.parked + victim); }
            if (cut && victim == a) { rv.parent = end; rv.len = ra.len; }      // the lower part of the edge just cut
            if (cut && rv.parent == a) have_parent = false;                    // (its parent's record has changed)
            v0 = -1;
            st.tokens_live -= rv.len;
            --st.live_nodes; ++st.evictions;
            if (pk0 > 0) {
                // Queries are parked in the evicted leaf.  If one run of the member array is known to hold every slot whose
                // hint is this leaf, warp 0 looks after them itself (up to 8 such leaves and 32 slots that fall back per
                // decision); otherwise the whole CTA scans the unprocessed slots.
                const int2 lr = __ldcg(A.leaf_run + victim);
                if (lr.y > 0 && lr.y <= 1024 && ans.n_small < 8) { if (lane == 0) s_ta->small_v[ans.n_small] = victim; ++ans.n_small; }
                else ans.scan = 1;
            }
            if (lane == src) wok = false;
            const int32_t P = rv.parent;
            if (lane == 0) A.node[victim].nchild = -1;
            if (P == end) --e.nchild;                       // (its stamp is newer)
            else {
                LNode rp = rp0;
                if (!have_parent) rp = ld_node(A.node + P);
                const int32_t nc = rp.nchild - 1;
                if (P != 0 && stamp >= rp.last) {           // the stamp goes to the parent if newer
                    rp.last = stamp;
                    if (lane == 0) { A.node[P].last = stamp; T.clock_owner[stamp] = P; }
                }
                if (lane == 0) A.node[P].nchild = nc;
                // a parent that has become a leaf may be the next to go
                if (nc == 0 && P != 0 && rp.last >= wbase && rp.last < wend && lane == (int)(rp.last - wbase)) { wv = P; wok = true; }
            }
            __syncwarp();
        }
        if (!ans.failed && unc > 0) {
            ans.leaf = (int32_t)st.n_nodes++;
            ++st.live_nodes;
            st.tokens_live += unc;
            ++e.nchild;
            if (lane == 0) {
                LNode l;
                l.parent = end; l.depth = J.m; l.len = unc; l.nchild = 0; l.last = clock; l.off = J.vleaf;
                st_node(A.node + ans.leaf, l);
                T.clock_owner[clock] = ans.leaf;
                A.leaf_run[ans.leaf] = make_int2(J.gstart, J.gcount);     // whoever gets parked in it is a member of the pick's group
            }
        } else if (end != 0 && lane == 0) T.clock_owner[clock] = end;
        if (lane == 0) {
            st_node(A.node + end, e);
            s_ta->failed = ans.failed; s_ta->scan = ans.scan; s_ta->n_small = ans.n_small; s_ta->leaf = ans.leaf;
        }
        __syncwarp();
        named_arrive(3, 64);
    }
    if (lane == 0) {                                        // the tree's counters go back (a status recorded meanwhile stays)
        st.lru_cursor = wbase;
        TreeState* S = A.st;
        S->n_nodes = st.n_nodes; S->tokens_live = st.tokens_live; S->live_nodes = st.live_nodes; S->clock = st.clock;
        S->lru_cursor = st.lru_cursor; S->evictions = st.evictions;
        A.post->counters[4] = st.evictions - evictions0;
    }
    __syncwarp();
    named_bar(1, KLPM_FAST_THREADS);                        // (the helpers are told to leave)
}

struct LruTouch { int32_t seq, join; int32_t slot0, admitted; unsigned long long root; };

// Warp 2, between the jobs of the whole CTA: reads ahead.  Each time warp 0 has committed a decision it says who is oldest
// and what the tournament's root is; one of the two is nearly always the next pick.  This warp loads their records, their
// leaf blocks' keys, the keys of the coming arrivals and then the node records that warp 1 will walk, for no other
// purpose than to have them in this SM's L1.  It decides nothing, so it may be late or wrong.  Returns when warp 0 calls
// for a job of the whole CTA (or after a bounded number of polls, after which it only takes part in such jobs).
__device__ __forceinline__ int32_t touch(const void* p) {
    int32_t v;
    asm volatile("ld.global.ca.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void lru_touch_warp(const FastArgs& A, const LruTouch* s_touch, int32_t joined, int32_t n, int32_t fixed_n, int lane) {
    int32_t seen = 0;
    for (unsigned polls = 0; polls < (1u << 28); ++polls) {
        if (*(const volatile int32_t*)&s_touch->join != joined) return;
        const int32_t seq = *(const volatile int32_t*)&s_touch->seq;
        if (seq == seen) { __nanosleep(20); continue; }
        seen = seq;
        __threadfence_block();
        int32_t a = *(const volatile int32_t*)&s_touch->slot0, b = -1;
        const int32_t adm = *(const volatile int32_t*)&s_touch->admitted;
        const unsigned long long root = *(const volatile unsigned long long*)&s_touch->root;
        if (A.fixed) {
            a = a >= 0 && a < fixed_n ? __ldg(A.fixed + a) : -1;               // (slot0 is the number of the decision here)
            if (a >= n) a = -1;
        } else if (root != 0) {
            const unsigned rk = 0xffffffffu - (unsigned)(root & 0xffffffffULL);
            if (rk < (unsigned)n) b = A.pinv ? __ldg(A.pinv + rk) : (int32_t)rk;
        }
        // lanes 0-9: the oldest, 10-19: the root's slot (state with its hint, constant record, eight sectors of its block's keys), 20-27: keys of arrivals
        const int u = lane < 10 ? lane : lane - 10;
        const int32_t s = lane < 10 ? a : b;
        const void* p = nullptr;
        if (lane < 20 && s >= 0 && s < n) {
            if (u == 0) p = reinterpret_cast<const int32_t*>(A.dyn + s) + 6;
            else if (u == 1) p = A.stat + s;
            else if (!A.fixed) {
                const long long r = (((long long)s >> A.lb_shift) << A.lb_shift) + 4 * (u - 2);
                if (r < n) p = A.key + r;
            }
        } else if (lane >= 20 && lane < 28 && !A.fixed) {
            const long long r = (long long)(adm & ~3) + 4 * (lane - 20);
            if (r < n) p = A.key + r;
        }
        int32_t v = p ? touch(p) : 0;
        // the node the match ends in is the hint's or above it
        bool chain = u == 0 && lane < 20 && p != nullptr;
#pragma unroll 1
        for (int d = 0; d < 3 && chain; ++d) {
            if (v <= 0 || v >= A.T.max_nodes) chain = false;
            else v = touch(&A.node[v].parent);
        }
        __syncwarp();
    }
}

// Trees with a budget: a match of m tokens that ended in node *a or above it, as it is now: up from *a past every node
// that has been evicted (it takes its tokens along) or cut above the match.  *a and *w: the node it ends in and its record.
__device__ __forceinline__ int32_t lru_match_now(const FastArgs& A, int32_t m, int32_t* a, LNode* w) {
    *w = ld_node(A.node + *a);
    while (*a != 0) {
        if (w->nchild < 0) { if (w->depth < m) m = w->depth; }
        else if (m > w->depth) break;
        *a = w->parent;
        *w = ld_node(A.node + *a);
    }
    return m;
}

// Warp 0: the queries parked in leaves that the last decision evicted, when known member runs hold them all.  All leaves
// are taken together: two of them, one above the other, send their queries to one group.  Returns false, nothing changed,
// if more than 32 slots lose matched tokens (the caller has the CTA scan for them); *failed if there is no room.
// Which slots lose tokens is found by the walk that moves them.  The depth of the evicted leaf alone does not tell: hints
// stay with the lower part of an edge that is cut, so a match can end above the leaf its slot is parked in, in a node
// that the same decision has evicted too.
__device__ __noinline__ bool lru_fall_back_small(const FastArgs& A, const FastTour& R, const int32_t* small_v, int n_small, int32_t admitted,
                                                 int32_t* s_memcur, unsigned long long* root, bool* failed, int lane) {
    int32_t n_fall = 0, listed = 0;
    for (int sv = 0; sv < n_small; ++sv) listed += __ldcg(A.leaf_run + small_v[sv]).y;
    for (int sv = 0; sv < n_small && listed > 32; ++sv) {   // (up to 32 slots in the runs: no need to count first)
        const int32_t v = small_v[sv];
        const int2 lr = __ldcg(A.leaf_run + v);
        for (int32_t base = 0; base < lr.y; base += 32) {
            const int32_t r = base + lane < lr.y ? ld_member(A, lr.x + base + lane) : -1;
            bool hit = r >= 0 && !slot_done(R, A, r) && __ldcg(A.hintc + r) == v;
            if (hit) {
                const int32_t m0 = __ldcg(reinterpret_cast<const int32_t*>(A.dyn + r) + 2);
                int32_t a = v;
                LNode w;
                hit = lru_match_now(A, m0, &a, &w) != m0;
            }
            const unsigned same = __match_any_sync(FULL_MASK, hit ? r : -1 - lane);       // a slot can be listed twice in a run
            if (hit && (int)(__ffs(same) - 1) != lane) hit = false;
            n_fall += __popc(__ballot_sync(FULL_MASK, hit));
        }
    }
    if (n_fall > 32) return false;
    // every member whose hint is a dead leaf walks up; those that lose tokens are collected
    int32_t f_slot = -1;                                    // lane k holds the k-th slot that fell back
    unsigned long long f_hash = KLPM_FAST_NOGROUP;
    int32_t n_f = 0;
    for (int sv = 0; sv < n_small; ++sv) {
        const int32_t v = small_v[sv];
        const int2 lr = __ldcg(A.leaf_run + v);
        for (int32_t base = 0; base < lr.y; base += 32) {
            const int32_t r = base + lane < lr.y ? ld_member(A, lr.x + base + lane) : -1;
            bool hit = r >= 0 && !slot_done(R, A, r) && __ldcg(A.hintc + r) == v;
            const unsigned same = __match_any_sync(FULL_MASK, hit ? r : -1 - lane);
            if (hit && (int)(__ffs(same) - 1) != lane) hit = false;
            bool fell = false;
            unsigned long long h = KLPM_FAST_NOGROUP;
            if (hit) {
                const int32_t m0 = __ldcg(reinterpret_cast<const int32_t*>(A.dyn + r) + 2);
                int32_t a = v;
                LNode w;
                const int32_t mm = lru_match_now(A, m0, &a, &w);
                st_dyn_hint(A.dyn + r, a);
                __stcg(A.hintc + r, a);
                atomicAdd(A.parked + a, 1);
                A.leaf_run[a].y = -1;
                if (mm != m0) {
                    const FStat fs = ld_stat(A.stat + r);
                    const long long pos = a == 0 ? -1 : w.off + (long long)(mm - w.depth) - 1;
                    const int32_t ntok = __ldg(A.tok + fs.soff + mm);
                    st_dyn_state(A.dyn + r, pos, mm, ntok);
                    __stcg(A.key + r, fast_key(mm, fs.len, fs.rank, A.score_mode));
                    h = group_hash(pos, ntok);
                    fell = true;
                }
            }
            const unsigned fb = __ballot_sync(FULL_MASK, fell);
            const int32_t my = n_f + __popc(fb & ((1u << lane) - 1u));
            for (unsigned bits = fb; bits; bits &= bits - 1) {      // hand each fallen slot to the lane that keeps it
                const int src = __ffs(bits) - 1;
                const int32_t dst = __shfl_sync(FULL_MASK, my, src);
                const int32_t rr = __shfl_sync(FULL_MASK, r, src);
                const unsigned long long hh = __shfl_sync(FULL_MASK, h, src);
                if (lane == dst) { f_slot = rr; f_hash = hh; }
            }
            n_f += __popc(fb);
            __syncwarp();
        }
    }
    if (n_f > 0) {
        // the fallen slots are grouped afresh in a run appended to the member array (ranked by shuffles)
        const int32_t base = *s_memcur;
        if ((long long)base + n_f > (long long)A.mem_cap) {
            if (lane == 0) set_status(A.st, RT_ERR_CAPACITY, 113);
            *failed = true;
        } else {
            int32_t rank = 0, start = 0, cnt = 0;
            for (int k2i = 0; k2i < n_f; ++k2i) {           // (at most 32)
                const unsigned long long hk = __shfl_sync(FULL_MASK, f_hash, k2i);
                const bool lt = hk < f_hash, eq = hk == f_hash;
                start += lt; cnt += eq; rank += (lt || (eq && k2i < lane));
            }
            if (f_slot >= 0) {
                __stcg(A.mem + base + rank, f_slot);
                st_dyn_group(A.dyn + f_slot, base + start, cnt);
            }
            __syncwarp();
            if (lane == 0) *s_memcur = base + n_f;
            __syncwarp();
            // their keys went down: the leaf blocks of the arrived ones are recomputed
            for (int k2i = 0; k2i < n_f; ++k2i) {
                const int32_t rr = __shfl_sync(FULL_MASK, f_slot, k2i);
                if (rr < admitted) {
                    const int32_t bb = rr >> A.lb_shift;
                    admit_blocks_one(A, R, bb, bb << A.lb_shift, admitted, lane);
                    __syncwarp();
                    *root = tour_update(R, bb, lane);
                }
            }
        }
    }
    return true;
}

// G: the bitmap of processed slots lives in global memory (queues too long for shared memory).
template <bool G>
__global__ void __launch_bounds__(KLPM_FAST_THREADS, 1)
lru_run_kernel(const __grid_constant__ FastArgs A) {
    extern __shared__ __align__(16) unsigned char fast_smem[];
    __shared__ FastJob s_job;
    __shared__ LruJob s_tj;
    __shared__ LruAnswer s_ta;
    __shared__ LruTouch s_touch;
    __shared__ int s_cnt;
    __shared__ int32_t s_memcur;              // first free entry of the member array
    __shared__ unsigned int s_dirty[256];
    if (*reinterpret_cast<const volatile int32_t*>(A.skip)) return;       // the capacity check said no: nothing is touched
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t n = A.n;
    const int32_t nb1p = (A.nb + 31) & ~31, n2 = nb1p >> 5, n2p = (n2 + 31) & ~31, n3 = n2p >> 5;
    const int32_t nwords = (n + 31) >> 5;
    FastTour R;
    R.t1 = reinterpret_cast<unsigned long long*>(fast_smem);
    R.t2 = R.t1 + nb1p;
    R.t3 = R.t2 + n2p;
    R.n2 = n2; R.n3 = n3;
    unsigned long long* sh = R.t3 + 32;
    int32_t* sr = reinterpret_cast<int32_t*>(sh + KLPM_FAST_SORT_CAP);
    unsigned int* s_bits = reinterpret_cast<unsigned int*>(sr + KLPM_FAST_SORT_CAP);
    R.g_done = G ? 1 : 0;
    R.g_bits = 0;
    R.done = G ? A.done : s_bits;
    R.skip = nullptr; R.gb = nullptr;
    R.dirty = s_dirty;
    for (int32_t i = threadIdx.x; i < nb1p + n2p + 32; i += blockDim.x) R.t1[i] = 0ULL;
    if (threadIdx.x == 0) { s_memcur = 2 * n; s_touch.seq = 0; s_touch.join = 0; }
    if (!G) for (int32_t i = threadIdx.x; i < nwords; i += blockDim.x) s_bits[i] = 0u;
    __syncthreads();

    const int32_t fixed_n = A.fixed ? *reinterpret_cast<const volatile int32_t*>(A.n_fixed) : 0;
    if (warp == 1) { lru_tree_warp(A, R, &s_tj, &s_ta, &s_job, sh, sr, &s_cnt, &s_memcur, lane); return; }
    if (warp > 1) {
        int32_t joined = 0;
        for (;;) {
            if (warp == 2) lru_touch_warp(A, &s_touch, joined++, n, fixed_n, lane);
            named_bar(1, KLPM_FAST_THREADS);
            const FastJob J = s_job;
            if (J.type == FAST_JOB_EXIT) return;
            fast_job<true>(A, R, J, sh, sr, &s_cnt, &s_memcur);
        }
    }

    // ---------------------------------------------------------------- warp 0
    const long long INF = 0x7fffffffffffffffLL;
    const bool fixed = A.fixed != nullptr;
    const int32_t n_dec = fixed ? fixed_n : n;
    const int LB = 1 << A.lb_shift;
    long long now = A.start_tick;
    int32_t head = 0, admitted = 0, cyc = 0, c = 0;
    unsigned long long root = 0;
    long long n_cta_dissolve = 0, n_scan = 0, cy_wait = 0, cy_scan = 0, cy_dissolve = 0;
    bool failed = false;
    bool busy = false;                                      // warp 1 works on decision c - 1
    bool moved = false;                                     // queries have been parked elsewhere since warp 1's last job
    bool regroup = false;                                   // decision c - 1's group has other members: dissolve it once its leaf is known
    FastPick P;
    P.slot = 0; P.m = 0; P.len = 0; P.ntok = 0; P.x = A.tok; P.lcp = make_int4(-1, 0, 0, 0); P.pos = 0; P.vleaf = 0; P.admitted = 0; P.gstart = 0; P.gcount = 0; P.leaf = -1;

    int32_t told = 0, joins = 0;                            // messages to warp 2
    auto cta_job = [&]() {                                  // lane 0 has filled s_job; warp 1 is idle
        if (lane == 0) { s_tj.type = LRU_JOB_JOIN; __threadfence_block(); *(volatile int32_t*)&s_touch.join = ++joins; }
        __syncwarp();
        named_arrive(2, 64);
        named_bar(1, KLPM_FAST_THREADS);
        const FastJob J = s_job;
        fast_job<true>(A, R, J, sh, sr, &s_cnt, &s_memcur);
        root = tour_top(R, lane);
    };
    // Waits for warp 1 and finishes decision c - 1: queries that fell back out of evicted leaves, then the pick's group.
    // True if anything that the next decision is prepared from may have changed.
    auto finish = [&]() -> bool {
        const long long t0 = clock64();
        named_bar(3, 64);
        cy_wait += clock64() - t0;
        busy = false;
        const int32_t n_small = s_ta.n_small;
        bool scan = s_ta.scan != 0, changed = false;
        const int32_t leaf = s_ta.leaf;
        if (s_ta.failed) { failed = true; return true; }
        if (n_small > 0 || scan) {
            changed = true; moved = true;
            if (!scan) scan = !lru_fall_back_small(A, R, s_ta.small_v, n_small, admitted, &s_memcur, &root, &failed, lane);
            if (scan) {                                     // somebody was parked in an evicted leaf
                const long long t1 = clock64();
                ++n_scan;
                if (lane == 0) { s_job.type = FAST_JOB_FALLBACK; s_job.a0 = fixed ? 0 : head; s_job.a1 = admitted; }
                cta_job();
                cy_scan += clock64() - t1;
            }
        }
        if (regroup && !failed) {
            changed = true; moved = true;
            P.leaf = leaf; P.admitted = admitted;
            P.lcp = __ldcg(A.lcp + P.slot);
            if (dissolve_is_small(P)) root = dissolve_small(A, P, R, root, lane);
            else {
                const long long t1 = clock64();
                ++n_cta_dissolve;
                if (lane == 0) { s_job.type = FAST_JOB_DISSOLVE; s_job.pick = P; }
                cta_job();
                cy_dissolve += clock64() - t1;
            }
        }
        regroup = false;
        __syncwarp();
        return changed;
    };
    auto slot_of_root = [&]() -> int32_t {
        const unsigned rk = 0xffffffffu - (unsigned)(root & 0xffffffffULL);
        return A.pinv ? __ldg(A.pinv + rk) : (int32_t)rk;
    };

    auto fcfs_next = [&]() -> bool { return A.policy == KLPM_POLICY_FCFS || (A.policy == KLPM_POLICY_KLPM && cyc == 0); };
    // warp 2 is told which slots come next: it brings what the two warps are about to read into L1
    auto tell = [&]() {
        if (lane == 0) {
            s_touch.slot0 = fixed ? c : head; s_touch.root = root; s_touch.admitted = admitted;
            __threadfence_block();
            *(volatile int32_t*)&s_touch.seq = ++told;
        }
    };
    long long tw = INF, next_t = INF;                       // 32 coming arrivals (lane i: slot wb + i); the next one
    int32_t wb = 0;
    if (!fixed) { tw = lane < n ? __ldg(A.sorted_t + lane) : INF; next_t = __shfl_sync(FULL_MASK, tw, 0); }
    tell();

    while (c < n_dec && !failed) {
        if (busy && regroup) { finish(); if (failed) break; }
        int32_t slot = 0, b = 0;
        unsigned long long bm = 0, o1 = 0, o2 = 0, o3 = 0;
        FDyn pd; FStat ps;
        if (fixed) {                                        // a given order (klpm_replay): no admission, no pick; slots are the queries in index order
            slot = __ldg(A.fixed + c);
            pd = ld_dyn_l1(A.dyn + slot);
            ps = ld_stat(A.stat + slot);
            if (busy && finish()) continue;
        } else {
            // ---- time and arrivals: idle until somebody has arrived, then admit everybody who has
            if (head == admitted && next_t > now) now = next_t;
            while (admitted < n && next_t <= now && !failed) {      // (an arrival can be the largest time there is, like the padding)
                const int off = admitted - wb;
                const int cnt = __popc(__ballot_sync(FULL_MASK, lane >= off && wb + lane < n && tw <= now));      // (arrivals are sorted)
                const int32_t a1 = admitted + cnt, ra = wb + lane;
                if (off + cnt == 32 && a1 + 64 < n && __ldg(A.sorted_t + a1 + 64) <= now) {
                    // a crowd: gallop, then bisect (lane 0), and the whole CTA admits them
                    long long lo = a1 + 65, hi = n;
                    if (lane == 0) {
                        long long step = 1;
                        while (lo + step <= hi && __ldg(A.sorted_t + lo + step - 1) <= now) { lo += step; step <<= 1; }
                        if (lo + step < hi) hi = lo + step;
                        while (lo < hi) { const long long mid = (lo + hi) >> 1; if (__ldg(A.sorted_t + mid) <= now) lo = mid + 1; else hi = mid; }
                    }
                    const int32_t all = (int32_t)__shfl_sync(FULL_MASK, lo, 0);
                    if (busy) finish();
                    if (failed) break;
                    if (lane == 0) { s_job.type = FAST_JOB_ADMIT; s_job.a0 = admitted; s_job.a1 = all; }
                    cta_job();
                    admitted = all;
                } else {
                    // keys only come in: every level above takes the larger of what it holds and the newcomers (one or two leaf blocks)
                    const unsigned long long ak = ra >= admitted && ra < a1 ? *(A.key + ra) : 0ULL;
                    const int32_t b0 = admitted >> A.lb_shift, b1 = (a1 - 1) >> A.lb_shift;
                    for (int32_t bb = b0; bb <= b1; ++bb) {
                        const unsigned long long km = warp_max64r((ra >> A.lb_shift) == bb ? ak : 0ULL);
                        const unsigned long long p1 = R.t1[bb], p2 = R.t2[bb >> 5], p3 = R.t3[bb >> 10];
                        __syncwarp();
                        R.t1[bb] = km > p1 ? km : p1; R.t2[bb >> 5] = km > p2 ? km : p2; R.t3[bb >> 10] = km > p3 ? km : p3;
                        root = km > root ? km : root;
                        __syncwarp();
                    }
                    admitted = a1;
                }
                if (admitted >= wb + 32) {
                    wb = admitted;
                    tw = wb + lane < n ? __ldg(A.sorted_t + wb + lane) : INF;
                }
                next_t = __shfl_sync(FULL_MASK, tw, admitted - wb);
            }
            if (failed) break;
            // ---- pick
            slot = fcfs_next() ? head : slot_of_root();
            if (slot < 0 || slot >= admitted || slot_done(R, A, slot)) {
                if (busy) { finish(); continue; }           // (prepared from a tournament that is being corrected)
                if (lane == 0) set_status(A.st, RT_ERR_LIMIT, 105);
                failed = true; break;                       // cannot happen
            }
            // ---- its records; its leaf block's largest key without it, and the largest beside its blocks on the levels above
            b = slot >> A.lb_shift;
            const long long r = ((long long)b << A.lb_shift) + lane;
            const unsigned long long kk = r < n ? *(A.key + r) : 0ULL;
            pd = ld_dyn_l1(A.dyn + slot);
            ps = ld_stat(A.stat + slot);
            {
                const int32_t i2 = b >> 5, i3 = i2 >> 5;
                const unsigned long long x1 = lane == (b & 31) ? 0ULL : R.t1[(i2 << 5) + lane];
                const unsigned long long x2 = lane == (i2 & 31) ? 0ULL : R.t2[(i3 << 5) + lane];
                const unsigned long long x3 = lane == i3 ? 0ULL : R.t3[lane];
                if (r < admitted && r != slot && lane < LB && !slot_done(R, A, r)) bm = kk;
                for (int32_t u = lane + 32; u < LB; u += 32) {
                    const long long r2 = ((long long)b << A.lb_shift) + u;
                    if (r2 < admitted && r2 != slot && !slot_done(R, A, r2)) { const unsigned long long k2 = *(A.key + r2); if (k2 > bm) bm = k2; }
                }
                o1 = warp_max64r(x1); o2 = warp_max64r(x2); o3 = warp_max64r(x3);
                bm = warp_max64r(bm);
            }
            // ---- nothing has been committed yet: the decision before must be finished first
            if (busy && finish()) continue;                 // (or failed: the loop ends)
            if (++cyc == A.k) cyc = 0;
            {
                const unsigned long long v2 = bm > o1 ? bm : o1, v3 = v2 > o2 ? v2 : o2;
                const int32_t i2 = b >> 5;
                R.t1[b] = bm; R.t2[i2] = v2; R.t3[i2 >> 5] = v3;       // (every lane stores the same)
                root = v3 > o3 ? v3 : o3;
            }
        }
        // ---- the pick is processed: charge it (Definition 2), hand the tree its part
        if (!G) R.done[slot >> 5] |= 1u << (slot & 31);
        else if (lane == 0) __stcg(R.done + (slot >> 5), __ldcg(R.done + (slot >> 5)) | (1u << (slot & 31)));
        const int32_t unc = ps.len - pd.m;
        const long long vleaf = A.vbase + ((long long)c << 32);               // positions in its new leaf: unique per decision, above every real pool index
        {
            const long long begin = now > ps.t ? now : ps.t;
            now = begin + (A.c_den + A.c_num * (long long)ps.len) * (long long)unc;
        }
        if (lane == 0) {
            s_tj.type = LRU_JOB_STEP; s_tj.hint = pd.hint; s_tj.m = pd.m; s_tj.len = ps.len; s_tj.gstart = pd.gstart; s_tj.gcount = pd.gcount;
            s_tj.vleaf = vleaf; s_tj.moved = moved ? 1 : 0;
        }
        moved = false;
        __syncwarp();
        named_arrive(2, 64);
        busy = true;
        if (lane == 0) {
            if (A.order) A.order[c] = ps.ord;
            A.uncached[ps.ord] = unc; A.ttft[ps.ord] = now - ps.t;
            if (A.completion) A.completion[ps.ord] = now;
        }
        ++c;
        regroup = unc > 0 && pd.gcount > 1;
        if (regroup) {
            P.slot = slot; P.m = pd.m; P.len = ps.len; P.ntok = pd.ntok; P.x = A.tok + ps.soff; P.pos = pd.pos; P.vleaf = vleaf;
            P.gstart = pd.gstart; P.gcount = pd.gcount;
        }
        __syncwarp();
        if (!fixed && slot == head) head = next_head(R.done, G ? 1 : 0, nwords, n, head, lane);
        tell();
    }
    if (busy) { named_bar(3, 64); }
    if (lane == 0) {
        A.post->c0 = n;                                     // list mode never began: nothing is left to charge
        A.post->now0 = now;
        long long* cn = A.post->counters;
        cn[0] = c; cn[1] = n_cta_dissolve; cn[2] = n_scan; cn[3] = s_memcur - 2 * n;
        cn[5] = cy_wait; cn[6] = cy_scan; cn[7] = cy_dissolve;
        for (int i = 8; i < 16; ++i) cn[i] = 0;
        s_job.type = FAST_JOB_EXIT;
        s_tj.type = LRU_JOB_EXIT;
        __threadfence_block();
        *(volatile int32_t*)&s_touch.join = ++joins;
    }
    __syncwarp();
    named_arrive(2, 64);
    named_bar(1, KLPM_FAST_THREADS);
}

// The charge pass after the loop: the decisions made in list mode, c0 .. n-1, are in `order` as slots (of a given order,
// klpm_replay, all decisions, and slots are queries).  Definition 2: R = max(R_prev, t) + cost.  As a function of R_prev
// that is x -> max(x + a, b) with a = cost, b = t + cost, and such functions compose to one of the same form, so the
// completion times are a prefix scan.  Three small kernels: per decision its uncached tokens and cost (and the query
// index put in `order`), a scan of the blocks, and the completion times and TTFTs.
#define KLPM_CHARGE_THREADS 256
struct ChargeFn { long long a, b; };
__device__ __forceinline__ ChargeFn charge_none() { ChargeFn f; f.a = 0; f.b = -0x4000000000000000LL; return f; }
__device__ __forceinline__ ChargeFn charge_then(const ChargeFn& f, const ChargeFn& g) {      // first f, then g
    ChargeFn r;
    r.a = f.a + g.a;
    const long long x = f.b + g.a;
    r.b = x > g.b ? x : g.b;
    return r;
}
__device__ __forceinline__ long long charge_at(const ChargeFn& f, long long x) { return x + f.a > f.b ? x + f.a : f.b; }
// inclusive scan over the warp
__device__ __forceinline__ ChargeFn charge_warp_scan(ChargeFn f, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        ChargeFn o;
        o.a = __shfl_up_sync(FULL_MASK, f.a, d); o.b = __shfl_up_sync(FULL_MASK, f.b, d);
        if (lane >= d) f = charge_then(o, f);
    }
    return f;
}
__device__ __forceinline__ int32_t charge_end(const FastArgs& A) { return A.fixed ? *A.n_fixed : A.n; }

// `ipt` consecutive decisions per thread: at most 1,024 blocks whatever the queue's length.
__global__ void __launch_bounds__(KLPM_CHARGE_THREADS)
charge_cost_kernel(FastArgs A, long long* cost, ChargeFn* bsum, int32_t ipt) {
    __shared__ ChargeFn s_w[KLPM_CHARGE_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * ipt;
    const long long c0 = A.post->c0;
    const int32_t end = charge_end(A);
    ChargeFn f = charge_none();
    for (int32_t u = 0; u < ipt; ++u) {
        const long long i = i0 + u, c = c0 + i;
        if (c < end) {
            const int32_t slot = A.fixed ? __ldg(A.fixed + c) : A.order[c];
            const int4 s = __ldg(reinterpret_cast<const int4*>(A.stat + slot));     // arrival, length, query index
            const int32_t len = s.z, ord = s.w, unc = len - A.dyn[slot].m;
            const long long t = (long long)(((unsigned long long)(unsigned)s.y << 32) | (unsigned)s.x);
            ChargeFn g;
            g.a = (A.c_den + A.c_num * (long long)len) * (long long)unc;
            g.b = t + g.a;
            if (A.order) A.order[c] = ord;
            A.uncached[ord] = unc;
            cost[i] = g.a;
            f = charge_then(f, g);
        }
    }
    f = charge_warp_scan(f, lane);
    if (lane == 31) s_w[warp] = f;
    __syncthreads();
    if (threadIdx.x == 0) {
        ChargeFn sum = s_w[0];
        for (int w = 1; w < KLPM_CHARGE_THREADS / 32; ++w) sum = charge_then(sum, s_w[w]);
        bsum[blockIdx.x] = sum;
    }
}
// bsum[b].a <- time at which block b's first decision may start (at most 1,024 blocks)
__global__ void __launch_bounds__(1024)
charge_scan_kernel(FastArgs A, ChargeFn* bsum, int32_t nblocks) {
    __shared__ ChargeFn s_w[32];
    const int u = threadIdx.x, lane = u & 31, warp = u >> 5;
    ChargeFn f = u < nblocks ? bsum[u] : charge_none();
    f = charge_warp_scan(f, lane);
    if (lane == 31) s_w[warp] = f;
    __syncthreads();
    if (warp == 0) { ChargeFn g = charge_warp_scan(s_w[lane], lane); __syncwarp(); s_w[lane] = g; }
    __syncthreads();
    ChargeFn before;                                        // everything before this block
    before.a = __shfl_up_sync(FULL_MASK, f.a, 1); before.b = __shfl_up_sync(FULL_MASK, f.b, 1);
    if (lane == 0) before = charge_none();
    if (warp > 0) before = charge_then(s_w[warp - 1], before);
    if (u < nblocks) bsum[u].a = charge_at(before, A.post->now0);
}
__global__ void __launch_bounds__(KLPM_CHARGE_THREADS)
charge_apply_kernel(FastArgs A, const long long* cost, const ChargeFn* bsum, int32_t ipt) {
    __shared__ ChargeFn s_w[KLPM_CHARGE_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * ipt;
    const long long c0 = A.post->c0;
    const int32_t end = charge_end(A);
    ChargeFn f = charge_none();                             // this thread's decisions
    for (int32_t u = 0; u < ipt; ++u) {
        const long long c = c0 + i0 + u;
        if (c < end) {
            ChargeFn g;
            g.a = cost[i0 + u];
            g.b = A.arrival[A.fixed ? __ldg(A.fixed + c) : A.order[c]] + g.a;
            f = charge_then(f, g);
        }
    }
    f = charge_warp_scan(f, lane);
    if (lane == 31) s_w[warp] = f;
    __syncthreads();
    long long run = bsum[blockIdx.x].a;                     // time at which this thread's first decision may start
    for (int w = 0; w < warp; ++w) run = charge_at(s_w[w], run);
    ChargeFn before;
    before.a = __shfl_up_sync(FULL_MASK, f.a, 1); before.b = __shfl_up_sync(FULL_MASK, f.b, 1);
    if (lane > 0) run = charge_at(before, run);
    for (int32_t u = 0; u < ipt; ++u) {
        const long long i = i0 + u, c = c0 + i;
        if (c < end) {
            const int32_t ord = A.fixed ? __ldg(A.fixed + c) : A.order[c];
            const long long t = A.arrival[ord];
            run = (run > t ? run : t) + cost[i];
            A.ttft[ord] = run - t;
            if (A.completion) A.completion[ord] = run;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// bulk insertion of many prompts into a tree without a budget.  The set of node boundaries a radix tree
// ends up with does not depend on the order in which prompts are stored, so prompts are inserted in
// rounds: every pending prompt is walked from the root (read-only), then at most one prompt per edge
// cuts that edge, and prompts that end at a node boundary add their leaves concurrently (the hash
// table's compare-and-swap on the key decides between prompts that want the same child).
// ------------------------------------------------------------------------------------------------
struct BulkArgs {
    const int32_t* tok; const int64_t* off;
    const int32_t* pend_in; int32_t* pend_out; unsigned int* n_out;   // walk: prompts to walk -> prompts not fully stored yet
    int32_t* pend_next; unsigned int* n_next;                          // apply: prompts that have to try again next round
    unsigned int* n_walk;                                              // walk: work counter
    int32_t* claim;                    // per node: lowest prompt index that wants to cut its edge
    int32_t* pm; int32_t* pnode; int32_t* poff;   // per prompt: where its walk ended
};

__global__ void __launch_bounds__(256)
bulk_walk_kernel(TreeDev T, BulkArgs A, unsigned n_pending) {
    const int lane = threadIdx.x & 31;
    for (;;) {                                              // prompts are handed out by a counter: their lengths differ widely
        unsigned p = 0;
        if (lane == 0) p = atomicAdd(A.n_walk, 1u);
        p = __shfl_sync(FULL_MASK, p, 0);
        if (p >= n_pending) return;
        const int32_t i = __ldg(A.pend_in + p);
        const int64_t lo = __ldg(A.off + i);
        const int32_t len = (int32_t)(__ldg(A.off + i + 1) - lo);
        // the tree has no budget, so the walk streams along contiguous pool runs (as the batched match does)
        int32_t node, off;
        const int32_t m = walk_chain(T, A.tok + lo, len, true, &node, &off);
        const bool full = node == 0 || off == __ldg(T.span_len + node);     // ends on a node boundary (or at the root)
        if (lane == 0 && !(m == len && full)) {
            A.pm[i] = m; A.pnode[i] = node; A.poff[i] = full ? -1 : off;
            if (!full) atomicMin(&A.claim[node], i);
            A.pend_out[atomicAdd(A.n_out, 1u)] = i;
        }
    }
}

// First round when a batched match of the prompts against the tree as it still is has left its records (MatchState):
// the node where each match ended is looked up from the position (end_node[] along the run), then what
// bulk_walk_kernel does after its walk.  One lane per prompt, 32 prompts of the list per warp at a time; the search
// along a run for a match that ended inside an edge is the whole warp's, one prompt after the other; the list of
// pending prompts grows by one addition per warp.
__global__ void __launch_bounds__(256)
bulk_from_state_kernel(TreeDev T, BulkArgs A, const MatchState* __restrict__ state, unsigned long long tag, unsigned n_pending) {
    const int lane = threadIdx.x & 31;
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
    const EndIndex X = end_index(T);
    for (unsigned long long p0 = (unsigned long long)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32ULL; p0 < n_pending;
         p0 += (unsigned long long)nwarps * 32ULL) {
        const unsigned long long p = p0 + lane;
        int32_t i = -1;
        if (p < n_pending) i = A.pend_in[p];                 // < 0: a replay that stopped early, not processed
        bool act = i >= 0, inside = false;
        int32_t len = 0, m = 0, node = 0, off = -1;          // off < 0: the match ends on a node boundary (or at the root)
        long long pos = -1, cend = 0;
        if (act) {
            len = (int32_t)(__ldg(A.off + i + 1) - __ldg(A.off + i));
            const int4* src = reinterpret_cast<const int4*>(state + i);
            const int4 a = __ldcg(src), b = __ldcg(src + 1);
            pos = (long long)(((unsigned long long)(unsigned)a.y << 32) | (unsigned)a.x);
            cend = (long long)(((unsigned long long)(unsigned)a.w << 32) | (unsigned)a.z);
            m = b.x;
            const unsigned long long got = ((unsigned long long)(unsigned)b.w << 32) | (unsigned)b.z;
            if (got != tag || m < 0 || m > len || pos < -1 || pos >= T.max_pool || cend < 0 || cend > T.max_pool) {
                set_status(T.st, RT_ERR_INVALID, 110);      // not a record of that match: the prompt is left out
                act = false;
            } else if (pos >= 0) {
                node = node_ending_at(X, pos, *reinterpret_cast<const volatile long long*>(&T.st->n_nodes));
                inside = node < 0;
            }
        }
        // The node of the run whose edge ends first after the match: four searches side by side, eight lanes and 32 pool
        // tokens each per step (one after the other with the whole warp: 239 us for 262,144 prompts, now 196; 32,768: 47, now 31).
        const long long n_nodes = *reinterpret_cast<const volatile long long*>(&T.st->n_nodes);
        for (unsigned im = __ballot_sync(FULL_MASK, inside); im;) {
            const int grp = lane >> 3, sub = lane & 7;
            int src = -1;                                    // the prompt (lane) this group of eight looks after
#pragma unroll
            for (int g = 0; g < 4; ++g) { if (im) { if (g == grp) src = __ffs(im) - 1; im &= im - 1; } }
            const long long gp = __shfl_sync(FULL_MASK, pos, src < 0 ? 0 : src), ge = __shfl_sync(FULL_MASK, cend, src < 0 ? 0 : src);
            long long q = ((gp + 1) & ~3LL) + 4 * sub;       // aligned: end_node has as many entries as the pool, rounded up
            int32_t found = -1;
            bool open = src >= 0;
            while (__any_sync(FULL_MASK, open)) {
                int32_t cand = -1;
                if (open && q < ge) {
                    const int4 e = __ldg(reinterpret_cast<const int4*>(X.end_node + q));
                    const int32_t ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
                    for (int u = 3; u >= 0; --u) {
                        const long long at = q + u;
                        if (ev[u] > 0 && ev[u] < n_nodes && at > gp && at < ge && __ldg(X.span_off + ev[u]) + __ldg(X.span_len + ev[u]) - 1 == at && !__ldg(X.dead + ev[u])) cand = ev[u];
                    }
                }
                const unsigned hit = (__ballot_sync(FULL_MASK, cand >= 0) >> (8 * grp)) & 0xffu;
                const int32_t first = __shfl_sync(FULL_MASK, cand, 8 * grp + (hit ? __ffs(hit) - 1 : 0));
                if (open && hit) { found = first; open = false; }
                q += 32;
                if (open && q - 4 * sub >= ge) open = false;
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {                    // hand the answers to the prompts' lanes
                const int32_t to = __shfl_sync(FULL_MASK, src, 8 * g), r = __shfl_sync(FULL_MASK, found, 8 * g);
                if (lane == to) {
                    if (r < 0) { set_status(T.st, RT_ERR_LIMIT, 111); act = false; }      // cannot happen
                    else { node = r; off = m - __ldg(T.depth_start + r); }
                }
            }
        }
        const bool pend = act && !(m == len && off < 0);
        if (pend) {
            A.pm[i] = m; A.pnode[i] = node; A.poff[i] = off;
            if (off >= 0) atomicMin(&A.claim[node], i);
        }
        const unsigned pm = __ballot_sync(FULL_MASK, pend);
        if (pm) {
            const int lead = __ffs(pm) - 1;
            unsigned base = 0;
            if (lane == lead) base = atomicAdd(A.n_out, (unsigned)__popc(pm));
            base = __shfl_sync(FULL_MASK, base, lead);
            if (pend) A.pend_out[base + __popc(pm & ((1u << lane) - 1u))] = i;
        }
    }
}

// What the apply step does for `width` pending prompts of the list (one per lane, from number p0 on): cut the edge the
// match ends in if the prompt holds the claim, add its leaf if it wins the child's table slot, or put the prompt on
// the list for the next round; then the warp copies the new leaves' tokens, one leaf after the other.  New nodes are
// numbered and pool space is taken with one addition per warp.  Tree fields are read through L2 (__ldcg): inside the
// kernel that runs all later rounds, another SM may have written them a moment ago.
__device__ __forceinline__ void bulk_apply_warp(const TreeDev& T, const BulkArgs& A, unsigned long long p0, unsigned n_apply, unsigned width, int lane,
                                                unsigned long long* s_live_nodes, unsigned long long* s_live_tokens) {
    TreeState* S = T.st;
    const unsigned lt = (1u << lane) - 1u;
    const bool act = (unsigned)lane < width && p0 + lane < n_apply;
    int32_t i = 0, len = 0, m = 0, node = 0, off = -1;
    const int32_t* x = A.tok;
    if (act) {
        i = __ldcg(A.pend_out + p0 + lane);
        const int64_t lo = __ldg(A.off + i);
        len = (int32_t)(__ldg(A.off + i + 1) - lo);
        x = A.tok + lo;
        m = __ldcg(A.pm + i); node = __ldcg(A.pnode + i); off = __ldcg(A.poff + i);
    }
    const int32_t unc = len - m;
    bool go = act, retry = false;
    int32_t end = node;
    // ---- the match ends inside node's edge: cut it, unless another prompt cuts this edge in this round
    bool cut = act && off >= 0;
    if (cut && __ldcg(A.claim + node) != i) { cut = false; go = false; retry = true; }
    const unsigned cm = __ballot_sync(FULL_MASK, cut);
    if (cm) {
        const int lead = __ffs(cm) - 1;
        unsigned long long base = 0;
        if (lane == lead) base = atomicAdd((unsigned long long*)&S->n_nodes, (unsigned long long)__popc(cm));
        base = __shfl_sync(FULL_MASK, base, lead);
        if (cut) {
            const long long u = (long long)base + __popc(cm & lt);
            A.claim[node] = 0x7fffffff;
            if (u >= T.max_nodes) { set_status(S, RT_ERR_CAPACITY); go = false; }
            else {
                atomicAdd(s_live_nodes, 1ULL);
                const int32_t par = __ldcg(T.parent + node), ds = __ldcg(T.depth_start + node), sl = __ldcg(T.span_len + node);
                const int64_t so = __ldcg(T.span_off + node);
                const int32_t t_up = __ldcg(T.pool + so), t_low = __ldcg(T.pool + so + off);
                T.parent[u] = par; T.depth_start[u] = ds; T.span_off[u] = so; T.span_len[u] = off;
                T.nchild[u] = 1; T.dead[u] = 0; T.last_access[u] = 0;
                T.first_tok[u] = t_up; T.first_tok[node] = t_low;
                long long slot = table_find(T, par, t_up);
                int64_t chain_end = so + sl;
                if (slot >= 0) { T.table[slot].child = (int32_t)u; T.table[slot].span_len = off; chain_end = __ldcg(&T.table[slot].chain_end); }
                else set_status(S, RT_ERR_LIMIT, 104);
                T.end_node[so + off - 1] = (int32_t)u;
                T.span_off[node] = so + off; T.span_len[node] = sl - off; T.depth_start[node] = ds + off;
                T.parent[node] = (int32_t)u;
                end = (int32_t)u;
                // (u, first token of the lower part) -> node : nobody else can want this key
                unsigned long long key = make_key(end, t_low);
                unsigned long long sl2 = hash_key(key) & T.table_mask;
                for (unsigned long long pr = 0; pr <= T.table_mask; ++pr) {
                    if (atomicCAS(&T.table[sl2].key, 0ULL, key) == 0ULL) {
                        T.table[sl2].child = node; T.table[sl2].span_len = sl - off; T.table[sl2].span_off = so + off;
                        T.table[sl2].chain_end = chain_end;
                        break;
                    }
                    sl2 = (sl2 + 1) & T.table_mask;
                }
            }
        }
    }
    // ---- the leaf: whoever puts the child's key into the table adds it
    long long won = -1;
    if (go && unc > 0) {
        unsigned long long key = make_key(end, __ldg(x + m));
        unsigned long long sl2 = hash_key(key) & T.table_mask;
        for (unsigned long long pr = 0; pr <= T.table_mask; ++pr) {
            unsigned long long old = atomicCAS(&T.table[sl2].key, 0ULL, key);
            if (old == 0ULL) { won = (long long)sl2; break; }
            if (old == key) { retry = true; break; }       // another prompt added that child (in this round, or it lost to it before)
            sl2 = (sl2 + 1) & T.table_mask;
        }
    }
    int64_t dst = -1;
    const unsigned wm = __ballot_sync(FULL_MASK, won >= 0);
    if (wm) {
        const long long need = won >= 0 ? (long long)unc + 6 : 0;
        long long inc = need;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const long long o = __shfl_up_sync(FULL_MASK, inc, d); if (lane >= d) inc += o; }
        const long long tot = __shfl_sync(FULL_MASK, inc, 31);
        unsigned long long nb = 0, pb = 0;
        if (lane == 0) {
            nb = atomicAdd((unsigned long long*)&S->n_nodes, (unsigned long long)__popc(wm));
            pb = atomicAdd((unsigned long long*)&S->pool_used, (unsigned long long)tot);
        }
        nb = __shfl_sync(FULL_MASK, nb, 0); pb = __shfl_sync(FULL_MASK, pb, 0);
        if (won >= 0) {
            const long long leaf = (long long)nb + __popc(wm & lt);
            const long long raw = (long long)pb + inc - need;
            const long long po = ((raw + 3) & ~3LL) + (m & 3);                  // span_off = depth_start (mod 4)
            if (leaf >= T.max_nodes || raw + unc + 6 > T.max_pool) {
                set_status(S, RT_ERR_CAPACITY);
                T.table[won].child = -1; T.table[won].span_len = 0; T.table[won].span_off = 0; T.table[won].chain_end = 0;
            } else {
                T.parent[leaf] = end; T.depth_start[leaf] = m; T.span_off[leaf] = po; T.span_len[leaf] = unc;
                T.nchild[leaf] = 0; T.dead[leaf] = 0; T.last_access[leaf] = 0;
                T.first_tok[leaf] = __ldg(x + m);
                T.table[won].child = (int32_t)leaf; T.table[won].span_len = unc; T.table[won].span_off = po;
                T.table[won].chain_end = po + unc;
                T.end_node[po + unc - 1] = (int32_t)leaf;
                atomicAdd(&T.nchild[end], 1);
                atomicAdd(s_live_tokens, (unsigned long long)unc);
                atomicAdd(s_live_nodes, 1ULL);
                dst = po;
            }
        }
    }
    const unsigned rm = __ballot_sync(FULL_MASK, retry);
    if (rm) {
        const int lead = __ffs(rm) - 1;
        unsigned base = 0;
        if (lane == lead) base = atomicAdd(A.n_next, (unsigned)__popc(rm));
        base = __shfl_sync(FULL_MASK, base, lead);
        if (retry) A.pend_next[base + __popc(rm & lt)] = i;
    }
    // ---- the new leaves' tokens: the first 128 of four leaves in flight together, the rest 512 at a time
    unsigned dm = __ballot_sync(FULL_MASK, dst >= 0);
    while (dm) {
        int32_t v[16];
        const int32_t* xs[4]; int64_t d[4]; int32_t cnt[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int src = dm ? __ffs(dm) - 1 : 0;
            cnt[g] = __shfl_sync(FULL_MASK, unc, src);
            if (!dm) cnt[g] = 0;
            dm &= dm - 1;
            d[g] = __shfl_sync(FULL_MASK, dst, src);
            xs[g] = reinterpret_cast<const int32_t*>(__shfl_sync(FULL_MASK, (unsigned long long)(x + m), src));
#pragma unroll
            for (int r = 0; r < 4; ++r) { const int32_t t = r * 32 + lane; v[4 * g + r] = t < cnt[g] ? __ldg(xs[g] + t) : 0; }
        }
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int r = 0; r < 4; ++r) { const int32_t t = r * 32 + lane; if (t < cnt[g]) T.pool[d[g] + t] = v[4 * g + r]; }
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
            const int32_t* xg = g == 0 ? xs[0] : g == 1 ? xs[1] : g == 2 ? xs[2] : xs[3];
            const int64_t dg = g == 0 ? d[0] : g == 1 ? d[1] : g == 2 ? d[2] : d[3];
            const int32_t cg = g == 0 ? cnt[0] : g == 1 ? cnt[1] : g == 2 ? cnt[2] : cnt[3];
            for (int32_t t0 = 128; t0 < cg; t0 += 512) {
#pragma unroll
                for (int r = 0; r < 16; ++r) { const int32_t t = t0 + r * 32 + lane; v[r] = t < cg ? __ldg(xg + t) : 0; }
#pragma unroll
                for (int r = 0; r < 16; ++r) { const int32_t t = t0 + r * 32 + lane; if (t < cg) T.pool[dg + t] = v[r]; }
            }
        }
    }
}

// Pending prompts per warp of the apply step: as few as keep every warp of the grid busy (their leaves' tokens are copied
// one warp after the other: 2,000 prompts with 6,000 tokens to store took 509 us at 32 per warp, now 50), at least two
// (a warp's prompts share its additions to the tree's counters), at most one per lane.
__device__ __forceinline__ unsigned bulk_width(unsigned n_apply, unsigned nwarps) {
    const unsigned w = (n_apply + nwarps - 1) / nwarps;
    return w < 2 ? 2 : w > 32 ? 32 : w;
}

__global__ void __launch_bounds__(256)
bulk_apply_kernel(TreeDev T, BulkArgs A) {
    // live nodes and live tokens are statistics only: summed per CTA here, added to the tree's counters once at the end
    __shared__ unsigned long long s_live_nodes, s_live_tokens;
    if (threadIdx.x == 0) { s_live_nodes = 0ULL; s_live_tokens = 0ULL; }
    __syncthreads();
    const unsigned n_pending = *A.n_out;
    const int lane = threadIdx.x & 31;
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
    const unsigned width = bulk_width(n_pending, nwarps);
    for (unsigned long long p0 = (unsigned long long)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * width; p0 < n_pending;
         p0 += (unsigned long long)nwarps * width)
        bulk_apply_warp(T, A, p0, n_pending, width, lane, &s_live_nodes, &s_live_tokens);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_live_nodes) atomicAdd((unsigned long long*)&T.st->live_nodes, s_live_nodes);
        if (s_live_tokens) atomicAdd((unsigned long long*)&T.st->tokens_live, s_live_tokens);
    }
}

// Every round after the first, in one cooperative kernel (no trip to the host between rounds).  A round = bring the
// pending prompts' positions up to date, grid barrier, apply, grid barrier.  A prompt is pending because it lost a
// cut to another prompt -- then the depth where its match ends has not moved, only the nodes around it have, and a
// walk up from the node it knew finds the node that holds that depth now -- or because another prompt added the
// child it wanted -- then it walks on from the node boundary it had reached, into that child (hop by hop, read
// through L2: the tokens may have been written by another SM a moment ago).  Counters alternate between rounds so
// that none is reset while somebody may still read it.  The barrier is bounded in time; when it gives up the status
// word says RT_ERR_LIMIT and every CTA returns.
struct BulkSync {
    unsigned int count, gen, abort, go;      // the barrier; whether another round follows
    unsigned int cnt_w[2], cnt_a[2];         // list lengths: positions brought up to date -> pend_b; retries -> pend_a
    unsigned int n_walk;                     // work counter of the first round's walk
    unsigned int pad[3];
};

// All threads call it.  `last` runs in one thread of the CTA that arrives last, before anybody is released.
template <typename F>
__device__ bool bulk_barrier(BulkSync* g, TreeState* st, long long limit_ns, F last) {
    __shared__ int s_ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned gen = *(volatile unsigned*)&g->gen;
        if (atomicAdd(&g->count, 1u) + 1u == gridDim.x) {
            last();
            g->count = 0;
            __threadfence();
            atomicAdd(&g->gen, 1u);
        } else {
            unsigned long long spins = 0, t0 = 0;
            while (*(volatile unsigned*)&g->gen == gen) {
                if (*(volatile unsigned*)&g->abort) { ok = 0; break; }
                if ((++spins & 1023ULL) == 0 || limit_ns == 0) {
                    unsigned long long now;
                    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
                    if (t0 == 0) t0 = now;
                    if (limit_ns == 0 || now - t0 > (unsigned long long)limit_ns || spins > (1ULL << 40)) {
                        set_status(st, RT_ERR_LIMIT, 112); atomicExch(&g->abort, 1u); ok = 0; break;
                    }
                }
            }
        }
        if (*(volatile unsigned*)&g->abort) ok = 0;
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    const bool ok = s_ok != 0;
    __syncthreads();
    return ok;
}

__global__ void __launch_bounds__(256)
bulk_rounds_kernel(TreeDev T, BulkArgs A, BulkSync* g, long long n_total, const int32_t* n_total_dev, long long limit_ns) {
    __shared__ unsigned long long s_live_nodes, s_live_tokens;
    if (threadIdx.x == 0) { s_live_nodes = 0ULL; s_live_tokens = 0ULL; }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned nwarps = (gridDim.x * blockDim.x) >> 5, warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    TreeState* S = T.st;
    unsigned count = __ldcg(&g->cnt_a[0]);                 // left pending by the first round (its kernels have completed)
    for (unsigned r = 1; count > 0; ++r) {
        const unsigned par = r & 1u;
        BulkArgs R = A;
        R.pend_in = A.pend_next; R.n_out = &g->cnt_w[par]; R.n_next = &g->cnt_a[par];
        // ---- positions of the pending prompts in the tree as it is now
        for (unsigned p = warp0; p < count; p += nwarps) {
            const int32_t i = __ldcg(R.pend_in + p);
            const int64_t lo = __ldg(A.off + i);
            const int32_t len = (int32_t)(__ldg(A.off + i + 1) - lo);
            int32_t m = __ldcg(A.pm + i), node = __ldcg(A.pnode + i), off = __ldcg(A.poff + i);
            bool full = true;
            if (off >= 0) {                                 // lost a cut: the depth m lies in `node` or in a node cut off above it
                int32_t a = node, ds = __ldcg(T.depth_start + a);
                while (a != 0 && m <= ds) { a = __ldcg(T.parent + a); ds = __ldcg(T.depth_start + a); }
                node = a; off = m - ds;
                full = a == 0 || off == __ldcg(T.span_len + a);
            }
            if (full) {                                     // on a node boundary: walk on into the child that may be there now
                const Term t = walk<false>(T, A.tok + lo, len, node, m);
                if (t.m > m) { m = t.m; node = t.node; off = t.off; full = t.full != 0; }
            }
            if (lane == 0 && !(m == len && full)) {
                A.pm[i] = m; A.pnode[i] = node; A.poff[i] = full ? -1 : off;
                if (!full) atomicMin(&A.claim[node], i);
                R.pend_out[atomicAdd(R.n_out, 1u)] = i;
            }
        }
        if (!bulk_barrier(g, S, limit_ns, [] {})) break;
        // ---- cuts and leaves
        const unsigned n_apply = __ldcg(R.n_out);
        if (blockIdx.x == 0 && threadIdx.x == 0) { g->cnt_w[par ^ 1u] = 0u; g->cnt_a[par ^ 1u] = 0u; }     // the next round's
        const unsigned width = bulk_width(n_apply, nwarps);
        for (unsigned long long p0 = (unsigned long long)warp0 * width; p0 < n_apply; p0 += (unsigned long long)nwarps * width)
            bulk_apply_warp(T, R, p0, n_apply, width, lane, &s_live_nodes, &s_live_tokens);
        if (!bulk_barrier(g, S, limit_ns, [&] {
                const bool stop = *(volatile int*)&S->status != 0 || (long long)r > 4 * n_total + 64;      // (every round stores a prompt)
                g->go = stop ? 0u : *(volatile unsigned*)&g->cnt_a[par];
            })) break;
        count = __ldcg(&g->go);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_live_nodes) atomicAdd((unsigned long long*)&S->live_nodes, s_live_nodes);
        if (s_live_tokens) atomicAdd((unsigned long long*)&S->tokens_live, s_live_tokens);
        if (blockIdx.x == 0) {                              // the logical clock advances by one per stored prompt
            if (n_total_dev) n_total = *n_total_dev;
            if (S->clock + n_total + 1 >= T.max_clock) set_status(S, RT_ERR_CAPACITY);
            else S->clock += n_total;
        }
    }
}

// Several arrays copied by one launch, 16 bytes at a time (every allocation of the library has room for the last, partial
// unit).  A rollback was eleven copies of their own, about 2 us each on a small tree.
#define KLPM_COPY_MAX 12
struct CopyList { int4* dst[KLPM_COPY_MAX]; const int4* src[KLPM_COPY_MAX]; long long end[KLPM_COPY_MAX]; int32_t n; };      // end: running sum of 16-byte units
__global__ void __launch_bounds__(512)
copy_list_kernel(CopyList L) {
    const long long step = (long long)gridDim.x * blockDim.x;
    if (L.end[L.n - 1] <= 4 * step) {                       // a small tree: all arrays at once, one latency
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < L.end[L.n - 1]; i += step) {
            int32_t a = 0;
            while (i >= L.end[a]) ++a;
            const long long at = i - (a > 0 ? L.end[a - 1] : 0);
            L.dst[a][at] = __ldcs(L.src[a] + at);
        }
        return;
    }
    long long begin = 0;
    for (int32_t a = 0; a < L.n; ++a) {                     // every array is spread over the whole grid
        const long long len = L.end[a] - begin;
        const int4* __restrict__ src = L.src[a];
        int4* __restrict__ dst = L.dst[a];
        long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        for (; i + 3 * step < len; i += 4 * step) {
            const int4 v0 = __ldcs(src + i), v1 = __ldcs(src + i + step), v2 = __ldcs(src + i + 2 * step), v3 = __ldcs(src + i + 3 * step);
            dst[i] = v0; dst[i + step] = v1; dst[i + 2 * step] = v2; dst[i + 3 * step] = v3;
        }
        for (; i < len; i += step) dst[i] = __ldcs(src + i);
        begin = L.end[a];
    }
}

__global__ void bulk_iota_kernel(int32_t* p, int32_t n) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = i;
}
__global__ void bulk_fill_kernel(int32_t* p, long long n, int32_t v) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}
// ------------------------------------------------------------------------------------------------
// Many independent small queues under the last-prompt cache (Definition 2 as printed; Section 2.1: only the
// previously processed prompt is cached).  This is the model the paper's worked example and Theorem 2 speak
// about, and a Monte-Carlo over random arrival orders (Definition 3) is thousands of such queues: one warp runs
// one queue from start to finish, so the schedule loop itself is what is data-parallel here.
// Per decision the warp looks at every prompt of its queue, 32 at a time: who has arrived, who is oldest, and --
// for a longest-match pick -- overlap(x_i, last processed prompt), computed by the whole warp for the prompts
// whose first token agrees with it.  The processed flags live in shared memory (one bit per prompt).
// ------------------------------------------------------------------------------------------------
#define KLPM_LAST_ONLY_WARPS 4
struct LastOnlyArgs {
    const int32_t* tok; const int64_t* off; const int64_t* arrival; const int64_t* prio; const int32_t* qoff;
    int32_t n_queues;
    int32_t policy, k;
    long long c_num, c_den, start_tick;
    int32_t* order; int32_t* uncached; int64_t* ttft; int64_t* completion; int32_t* n_skipped;
};

// First index in [0, n) where a and b differ, or n, for short strings: one warp-wide minimum per 128 tokens instead of
// a ballot per 32 of them.  Warp-cooperative: every lane calls it with the same arguments and gets the result.
__device__ __forceinline__ int32_t first_mismatch_short(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int32_t n, int lane) {
    for (int32_t base = 0; base < n; base += 128) {
        unsigned at = 0xffffffffu;
#pragma unroll
        for (int r = 3; r >= 0; --r) {
            const int32_t i = base + r * 32 + lane;
            if (i < n && __ldg(a + i) != __ldg(b + i)) at = (unsigned)i;
        }
        const unsigned m = __reduce_min_sync(FULL_MASK, at);
        if (m != 0xffffffffu) return (int32_t)m;
    }
    return n;
}

// A queue of at most 32 prompts (every queue of the Monte-Carlo): lane i keeps prompt i in registers from the first
// decision to the last, and the results leave in four coalesced stores at the end.
//   * The two orders a pick goes by -- (arrival, index) and (priority, arrival, index) -- are turned into ranks once, so
//     a pick is one or two warp reductions instead of a five-step tournament over 64-bit tuples.
//   * Overlaps come from one comparison per prompt instead of one or two per decision and candidate: prompts with the
//     same first token form a class, and each of them is compared once with the class's first prompt (the pivot), which
//     gives e = overlap with the pivot and the token that follows.  Two members with different e overlap in the smaller
//     one; with equal e and different next tokens in exactly e.  Only members that leave the pivot at the same place
//     with the same token (`twin`, rare) still have to be compared with each other, from e on.
// What bounds it: the issue rate (about 50 warp instructions per decision, 32 comparisons of 128 tokens); the tokens are
// read from HBM once.  65,536 queues of 32 prompts of 128 tokens: 376 us (3.1 TB/s, 5.6 G decisions/s); two passes over
// the queue and two token comparisons per decision, as longer queues still do it, took 1,482 us.
// Every warp-wide operation below is executed by all 32 lanes: lanes beyond the queue's length take part with values
// that never win.
__device__ __forceinline__ void last_only_small(const LastOnlyArgs& A, int32_t q0, int32_t n, int lane) {
    const long long INF = 0x7fffffffffffffffLL;
    const bool in = lane < n;
    long long t = INF, pr = 0;
    int32_t len = 0;
    const int32_t* x = A.tok;
    if (in) {
        t = __ldg(A.arrival + q0 + lane);
        const int64_t lo = __ldg(A.off + q0 + lane);
        len = (int32_t)(__ldg(A.off + q0 + lane + 1) - lo);
        x += lo;
        if (A.prio) pr = __ldg(A.prio + q0 + lane);
    }
    const bool full = len > 0;
    const int32_t first = full ? __ldg(x) : 0;
    const unsigned nonempty = __ballot_sync(FULL_MASK, full);
    const unsigned same = __match_any_sync(FULL_MASK, first) & nonempty;
    const int pivot = full ? __ffs(same) - 1 : 32 + lane;     // (an empty prompt is in no class)
    // ---- overlap with the class's pivot (the pivot's own is its length)
    int32_t e = len;
    for (unsigned todo = __ballot_sync(FULL_MASK, full && pivot != lane); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1, p = __shfl_sync(FULL_MASK, pivot, src);
        const int32_t* xs = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)x, src);
        const int32_t* xp = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)x, p);
        const int32_t ls = __shfl_sync(FULL_MASK, len, src), lp = __shfl_sync(FULL_MASK, len, p);
        const int32_t ee = first_mismatch_short(xs, xp, ls < lp ? ls : lp, lane);
        if (lane == src) e = ee;
    }
    const bool ended = e >= len;                              // nothing follows: agrees with the pivot to its own end
    const int32_t ntok = ended ? 0 : __ldg(x + e);
    const unsigned goes_on = __ballot_sync(FULL_MASK, !ended);
    const unsigned alike = __match_any_sync(FULL_MASK, ((unsigned long long)(unsigned)ntok << 32) | (unsigned)e) & same & goes_on;
    const bool twin = !ended && (alike & (alike - 1)) != 0;   // another member leaves the pivot at the same place with the same token
    const bool twins = __any_sync(FULL_MASK, twin);
    // ---- ranks in the two orders, the lane in the low bits: (rank << 5) | lane
    int rank_f = 0, rank_l = 0;
    const int t_hi = (int)(t >> 32), p_hi = (int)(pr >> 32);
    const int t_hi0 = __shfl_sync(FULL_MASK, t_hi, 0), p_hi0 = __shfl_sync(FULL_MASK, p_hi, 0);
    if (__all_sync(FULL_MASK, !in || (t_hi == t_hi0 && p_hi == p_hi0))) {      // the high words agree: the low ones decide
        const unsigned t32 = (unsigned)t, p32 = (unsigned)pr;
        for (int s = 0; s < n; ++s) {
            const unsigned ts = __shfl_sync(FULL_MASK, t32, s), ps = __shfl_sync(FULL_MASK, p32, s);
            const bool before = ts < t32 || (ts == t32 && s < lane);
            rank_f += before;
            rank_l += ps < p32 || (ps == p32 && before);
        }
    } else {
        for (int s = 0; s < n; ++s) {
            const long long ts = __shfl_sync(FULL_MASK, t, s), ps = __shfl_sync(FULL_MASK, pr, s);
            const bool before = ts < t || (ts == t && s < lane);
            rank_f += before;
            rank_l += ps < pr || (ps == pr && before);
        }
    }
    rank_f = rank_f << 5 | lane;
    rank_l = rank_l << 5 | lane;
    const long long cost_per = A.c_den + A.c_num * (long long)len;     // per uncached token (Definition 2)
    long long now = A.start_tick, my_R = 0;
    bool left = in, arrived = false;                          // not processed yet; everybody has arrived
    int32_t my_order = 0, my_m = 0, until_f = 0;
    int last = -1;
    for (int32_t c = 0; c < n; ++c) {
        // ---- who is waiting; if nobody, idle until the next arrival
        bool wait = left;
        if (!arrived) {                                       // (uniform)
            wait = left && t <= now;
            if (!__any_sync(FULL_MASK, wait)) {
                long long tmin = left ? t : INF;
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) { const long long o = __shfl_xor_sync(FULL_MASK, tmin, d); tmin = o < tmin ? o : tmin; }
                now = tmin;
                wait = left && t <= now;
            }
            arrived = __all_sync(FULL_MASK, wait == left);
        }
        bool fcfs_turn = A.policy == KLPM_POLICY_FCFS;
        if (A.policy == KLPM_POLICY_KLPM) { fcfs_turn = until_f == 0; until_f = fcfs_turn ? A.k - 1 : until_f - 1; }
        // ---- overlap with the prompt processed last
        int32_t score = 0;
        if (last >= 0) {
            const int32_t e_l = __shfl_sync(FULL_MASK, e, last), p_l = __shfl_sync(FULL_MASK, pivot, last);
            if (pivot == p_l) score = e < e_l ? e : e_l;
            if (twins) {                                      // (uniform)
                const int32_t n_l = __shfl_sync(FULL_MASK, ntok, last);
                const bool t_l = __shfl_sync(FULL_MASK, (int)twin, last) != 0;
                unsigned tm = __ballot_sync(FULL_MASK, wait && twin && t_l && pivot == p_l && e == e_l && ntok == n_l);
                if (tm) {                                     // they share more than e: compare from there on
                    const int32_t* xl = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)x, last);
                    const int32_t len_l = __shfl_sync(FULL_MASK, len, last);
                    for (; tm; tm &= tm - 1) {
                        const int src = __ffs(tm) - 1;
                        const int32_t* xs = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)x, src);
                        const int32_t ls = __shfl_sync(FULL_MASK, len, src);
                        const int32_t ee = e_l + first_mismatch_short(xs + e_l, xl + e_l, (ls < len_l ? ls : len_l) - e_l, lane);
                        if (lane == src) score = ee;
                    }
                }
            }
        }
        // ---- the pick: oldest, or largest overlap and then smallest (priority, arrival, index)
        unsigned r = 0xffffffffu;
        if (fcfs_turn) {
            if (wait) r = (unsigned)rank_f;
        } else {
            const unsigned best = __reduce_max_sync(FULL_MASK, wait ? (unsigned)score : 0u);
            if (wait && (unsigned)score == best) r = (unsigned)rank_l;
        }
        const int j = (int)(__reduce_min_sync(FULL_MASK, r) & 31u);     // (somebody is waiting)
        // ---- charge by Definition 2 (the pick has arrived, so it begins at once); x_j is the cached prompt now
        const long long cost = cost_per * (long long)(len - score);
        now += __shfl_sync(FULL_MASK, cost, j);
        if (lane == j) { my_m = score; my_R = now; left = false; }
        if (lane == c) my_order = j;
        last = j;
    }
    if (in) {
        A.order[q0 + lane] = my_order;
        A.uncached[q0 + lane] = len - my_m;
        A.ttft[q0 + lane] = my_R - t;
        if (A.completion) A.completion[q0 + lane] = my_R;
    }
}

__global__ void __launch_bounds__(32 * KLPM_LAST_ONLY_WARPS)
last_only_batch_kernel(LastOnlyArgs A) {
    __shared__ unsigned s_done[KLPM_LAST_ONLY_WARPS][KLPM_LAST_ONLY_MAX_QUEUE / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long r = (long long)blockIdx.x * KLPM_LAST_ONLY_WARPS + warp;
    if (r >= A.n_queues) return;
    const int32_t q0 = __ldg(A.qoff + r), n = __ldg(A.qoff + r + 1) - q0;
    if (n <= 0) return;
    if (n > KLPM_LAST_ONLY_MAX_QUEUE) {                       // too long for this entry point: left untouched, counted
        if (lane == 0 && A.n_skipped) atomicAdd(A.n_skipped, 1);
        return;
    }
    if (n <= 32) { last_only_small(A, q0, n, lane); return; }
    unsigned* done = s_done[warp];
    for (int32_t w = lane; w < KLPM_LAST_ONLY_MAX_QUEUE / 32; w += 32) done[w] = 0u;
    __syncwarp();
    const long long INF = 0x7fffffffffffffffLL;
    long long now = A.start_tick;
    int32_t last = -1, last_len = 0;                          // the cached prompt (global index) and its length
    const int32_t* last_x = nullptr;
    for (int32_t c = 0; c < n; ++c) {
        // ---- who is waiting; if nobody, idle until the next arrival
        bool any = false;
        long long tmin = INF;
        for (int32_t base = 0; base < n; base += 32) {
            const int32_t i = base + lane;
            if (i < n && !((done[i >> 5] >> (i & 31)) & 1u)) {
                const long long t = __ldg(A.arrival + q0 + i);
                any = any || t <= now;
                tmin = t < tmin ? t : tmin;
            }
        }
        any = __any_sync(FULL_MASK, any);
        if (!any) {
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) { const long long o = __shfl_xor_sync(FULL_MASK, tmin, d); tmin = o < tmin ? o : tmin; }
            now = tmin;
        }
        const bool fcfs_turn = A.policy == KLPM_POLICY_FCFS || (A.policy == KLPM_POLICY_KLPM && (c % A.k) == 0);
        // ---- the pick: best of (score desc, priority asc, arrival asc, index asc); score = 0 on an oldest-first turn,
        //      and the priority plays no part in it
        int32_t b_idx = -1, b_score = 0;
        long long b_prio = 0, b_t = 0;
        for (int32_t base = 0; base < n; base += 32) {
            const int32_t i = base + lane;
            bool waiting = false;
            long long t = 0, pr = 0;
            int32_t len = 0;
            const int32_t* x = nullptr;
            if (i < n && !((done[i >> 5] >> (i & 31)) & 1u)) {
                t = __ldg(A.arrival + q0 + i);
                waiting = t <= now;
            }
            int32_t score = 0;
            if (!fcfs_turn) {
                bool cmp = false;
                if (waiting) {
                    const int64_t lo = __ldg(A.off + q0 + i);
                    len = (int32_t)(__ldg(A.off + q0 + i + 1) - lo);
                    x = A.tok + lo;
                    if (A.prio) pr = __ldg(A.prio + q0 + i);
                    cmp = last >= 0 && len > 0 && last_len > 0 && __ldg(x) == __ldg(last_x);
                }
                unsigned cm = __ballot_sync(FULL_MASK, cmp);
                while (cm) {                                  // overlap(x_i, last): the whole warp compares one prompt at a time
                    const int src = __ffs(cm) - 1; cm &= cm - 1;
                    const int32_t* xs = (const int32_t*)__shfl_sync(FULL_MASK, (unsigned long long)x, src);
                    const int32_t ls = __shfl_sync(FULL_MASK, len, src);
                    const int32_t e = first_mismatch<true, 1>(xs, last_x, ls < last_len ? ls : last_len);
                    if (lane == src) score = e;
                }
            }
            if (waiting) {
                bool wins = b_idx < 0 || score > b_score;
                if (!wins && score == b_score) {
                    if (pr != b_prio) wins = pr < b_prio;
                    else wins = t < b_t || (t == b_t && i < b_idx);
                }
                if (wins) { b_idx = i; b_score = score; b_prio = pr; b_t = t; }
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const int32_t o_idx = __shfl_xor_sync(FULL_MASK, b_idx, d), o_score = __shfl_xor_sync(FULL_MASK, b_score, d);
            const long long o_prio = __shfl_xor_sync(FULL_MASK, b_prio, d), o_t = __shfl_xor_sync(FULL_MASK, b_t, d);
            bool wins = o_idx >= 0 && (b_idx < 0 || o_score > b_score);
            if (!wins && o_idx >= 0 && b_idx >= 0 && o_score == b_score) {
                if (o_prio != b_prio) wins = o_prio < b_prio;
                else wins = o_t < b_t || (o_t == b_t && o_idx < b_idx);
            }
            if (wins) { b_idx = o_idx; b_score = o_score; b_prio = o_prio; b_t = o_t; }
        }
        const int32_t j = b_idx;                               // somebody is waiting, so j >= 0
        if (j < 0) return;
        // ---- charge by Definition 2 against the cached prompt, then x_j is the cached prompt
        const int64_t lo = __ldg(A.off + q0 + j);
        const int32_t len = (int32_t)(__ldg(A.off + q0 + j + 1) - lo);
        const int32_t* x = A.tok + lo;
        int32_t m = 0;
        if (!fcfs_turn) m = b_score;                          // the overlap it was picked by
        else if (last >= 0) m = first_mismatch<true, 1>(x, last_x, len < last_len ? len : last_len);
        const int32_t unc = len - m;
        const long long tj = __ldg(A.arrival + q0 + j);
        const long long begin = now > tj ? now : tj;
        const long long R = begin + (A.c_den + A.c_num * (long long)len) * (long long)unc;
        if (lane == 0) {
            A.order[q0 + c] = j;
            A.uncached[q0 + j] = unc;
            A.ttft[q0 + j] = R - tj;
            if (A.completion) A.completion[q0 + j] = R;
            done[j >> 5] |= 1u << (j & 31);
        }
        __syncwarp();
        now = R; last = j; last_len = len; last_x = x;
    }
}

// ------------------------------------------------------------------------------------------------
// Trees with a budget: before and after the grouped loop.
// Before: the loop is all or nothing, so room for everything it can leave behind is checked first -- two nodes and one
// clock tick per prompt, and pool tokens for at most a budget's worth of new tokens plus three of alignment per node.
// After: the loop has kept the node arrays (parent, depth, length, children, stamps, dead flags) exact but has given
// the edges of new nodes virtual positions and has touched neither the token pool nor the child table.  Every node
// that is still alive gets its pool tokens (copied from the prompt that created its edge) and the child table is
// written afresh from the live nodes; nodes that were evicted again along the way cost nothing.
// ------------------------------------------------------------------------------------------------
struct LruInfo { long long n_nodes0; unsigned long long total_len; int32_t skip; int32_t pad; };

__global__ void lru_sum_kernel(const int64_t* __restrict__ off, int32_t n, LruInfo* info) {
    __shared__ unsigned long long s_w[8];
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long x = i < n ? (unsigned long long)(off[i + 1] - off[i]) : 0ULL;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(FULL_MASK, x, d);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_w[w];
        atomicAdd(&info->total_len, t);
    }
}
__global__ void lru_check_kernel(TreeDev T, int32_t n, LruInfo* info) {
    TreeState* S = T.st;
    long long fresh = S->tokens_live + (long long)info->total_len;
    if (fresh > T.budget) fresh = T.budget;
    const bool ok = S->n_nodes + 2LL * n <= T.max_nodes && S->clock + (long long)n + 1 < T.max_clock &&
                    S->pool_used + fresh + 6LL * n + 16 <= T.max_pool;
    info->n_nodes0 = S->n_nodes;
    info->skip = ok ? 0 : 1;
    if (!ok) set_status(S, RT_ERR_CAPACITY, 115);
}

// One warp per node created by the loop: if it is alive and its edge has a virtual position, give it room in the pool
// and copy its tokens from the prompt that created the edge (decision c = the position's high bits; the edge holds
// that prompt's tokens from the node's depth on).
__global__ void __launch_bounds__(256)
lru_tokens_kernel(TreeDev T, const int32_t* __restrict__ order, const int32_t* __restrict__ qtok, const int64_t* __restrict__ qoff,
                  long long vbase, const LruInfo* info) {
    if (info->skip) return;
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long n_end = T.st->n_nodes;
    for (long long v = info->n_nodes0 + (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5); v < n_end; v += nwarps) {
        if (T.dead[v]) continue;
        const long long so = T.span_off[v];
        if (so < vbase) continue;                           // a piece of an edge that was in the tree before: its tokens are in the pool
        const int32_t c = (int32_t)((so - vbase) >> 32), len = T.span_len[v], depth = T.depth_start[v];
        const int32_t* x = qtok + __ldg(qoff + __ldg(order + c)) + depth;
        long long base = 0;
        if (lane == 0) {
            const long long raw = (long long)atomicAdd((unsigned long long*)&T.st->pool_used, (unsigned long long)(len + 3));
            base = raw + (((long long)depth - raw) & 3LL);  // span_off = depth_start (mod 4), as everywhere
            if (raw + len + 3 > T.max_pool) { set_status(T.st, RT_ERR_CAPACITY, 116); base = -1; }      // (ruled out by the check before the loop)
        }
        base = __shfl_sync(FULL_MASK, base, 0);
        if (base < 0) continue;
        for (int32_t t = lane; t < len; t += 32) T.pool[base + t] = __ldg(x + t);
        if (lane == 0) T.span_off[v] = base;
    }
}

// Before the loop: the node arrays as records, no query parked anywhere, no member run known.  After it: the arrays from the
// records, and the child table empty.  (One launch each: a queue of one prompt pays for every launch: 101 us on a full cache with separate clears, now 87.)
__global__ void lru_pack_kernel(TreeDev T, LNode* node, int32_t* parked, int2* leaf_run, const LruInfo* info) {
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    for (long long v = first; v < T.max_nodes; v += step) { parked[v] = 0; leaf_run[v] = make_int2(-1, -1); }
    if (info->skip) return;
    const long long n = T.st->n_nodes;
    for (long long v = first; v < n; v += step) {
        LNode r;
        r.parent = T.parent[v]; r.depth = T.depth_start[v]; r.len = T.span_len[v]; r.nchild = T.dead[v] ? -1 : T.nchild[v];
        r.last = T.last_access[v]; r.off = T.span_off[v];
        st_node(node + v, r);
    }
}
__global__ void lru_unpack_kernel(TreeDev T, const LNode* __restrict__ node, const LruInfo* info) {
    if (info->skip) return;
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    const long long n = T.st->n_nodes, n16 = (long long)(T.table_mask + 1) * 2;      // (an entry is two 16-byte units)
    for (long long v = first; v < n; v += step) {
        const LNode r = ld_node(node + v);
        T.parent[v] = r.parent; T.depth_start[v] = r.depth; T.span_len[v] = r.len; T.nchild[v] = r.nchild < 0 ? 0 : r.nchild;
        T.dead[v] = r.nchild < 0; T.last_access[v] = r.last; T.span_off[v] = r.off;
    }
    int4* p = reinterpret_cast<int4*>(T.table);
    for (long long i = first; i < n16; i += step) p[i] = make_int4(0, 0, 0, 0);
}
__global__ void lru_table_kernel(TreeDev T, long long vbase, const LruInfo* info) {
    if (info->skip) return;
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < 1 || v >= T.st->n_nodes || T.dead[v]) return;
    const long long so = T.span_off[v];
    if (so >= vbase) return;                                // no room was found for it: the status word says so
    const int32_t len = T.span_len[v], ft = T.pool[so];
    T.first_tok[v] = ft;
    T.end_node[so + len - 1] = (int32_t)v;
    const unsigned long long key = make_key(T.parent[v], ft);
    unsigned long long slot = hash_key(key) & T.table_mask;
    for (unsigned long long pr = 0; pr <= T.table_mask; ++pr) {
        if (atomicCAS(&T.table[slot].key, 0ULL, key) == 0ULL) {
            T.table[slot].child = (int32_t)v; T.table[slot].span_len = len; T.table[slot].span_off = so; T.table[slot].chain_end = so + len;
            return;
        }
        slot = (slot + 1) & T.table_mask;
    }
    set_status(T.st, RT_ERR_CAPACITY, 117);
}

// batch size B: a query is finished when the last query of its bin of the processing order is
__global__ void batch_times_kernel(const int32_t* __restrict__ order, int32_t n, const int64_t* __restrict__ arrival,
                                   const int64_t* __restrict__ completion, int32_t n_queries, int32_t B, int64_t* ttft_b,
                                   int64_t* completion_b, int32_t* bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t last = (i / B + 1) * (int64_t)B - 1;
    if (last > n - 1) last = n - 1;
    const int32_t jl = __ldg(order + last), j = __ldg(order + i);
    if (jl < 0 || jl >= n_queries || j < 0 || j >= n_queries) {      // not a query: skipped, counted if the caller asked
        if (bad) atomicAdd(bad, 1);
        return;
    }
    const int64_t R = __ldg(completion + jl);
    completion_b[j] = R;
    ttft_b[j] = R - __ldg(arrival + j);
}

// klpm_replay through the grouped loop.  The order is checked first: the decisions that will be made are the entries
// before the first one that is not a query or names a query for the second time (the status word says so if there is
// one).  Slots are the queries in index order.
struct ReplayInfo { int32_t n_valid; int32_t pad; };
__global__ void replay_first_kernel(const int32_t* __restrict__ order, int32_t n_order, int32_t n_queries, int32_t* first_pos) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_order) return;
    const int32_t j = order[p];
    if (j >= 0 && j < n_queries) atomicMin(first_pos + j, p);
}
__global__ void replay_check_kernel(const int32_t* __restrict__ order, int32_t n_order, int32_t n_queries, const int64_t* __restrict__ off,
                                    const int32_t* __restrict__ first_pos, ReplayInfo* info, TreeState* st) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_order) return;
    const int32_t j = order[p];
    bool bad = j < 0 || j >= n_queries;
    if (!bad) { const int64_t len = off[j + 1] - off[j]; bad = len < 0 || len > 0x7fffffffLL || first_pos[j] < p; }
    if (bad) { atomicMin(&info->n_valid, p); set_status(st, RT_ERR_INVALID, 108); }
}
__global__ void replay_slots_kernel(const int64_t* __restrict__ arrival, int32_t n, long long* sorted_t, int32_t* ord) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { sorted_t[i] = arrival[i]; ord[i] = i; }
}
// the prompts a replay has processed, as the list the insertion after the loop works through (-1: not processed)
__global__ void replay_list_kernel(const int32_t* __restrict__ order, int32_t n_order, const ReplayInfo* info, int32_t* pend) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n_order) pend[p] = p < info->n_valid ? order[p] : -1;
}
__global__ void lru_sum_order_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ order, int32_t n_order,
                                     int32_t n_queries, LruInfo* info) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_order) return;
    const int32_t j = order[p];
    if (j >= 0 && j < n_queries) { const int64_t len = off[j + 1] - off[j]; if (len > 0) atomicAdd(&info->total_len, (unsigned long long)len); }
}

// slot order: bitonic sort of (arrival, index) pairs, padded to a power of two
// *unsorted (cleared by the host side): set if the arrivals are not in order yet -- queues mostly are, and their sort then
// has nothing to do.
__global__ void rank_init_kernel(const int64_t* __restrict__ arrival, int32_t n, long long np2, long long* key, int32_t* idx, unsigned int* unsorted) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np2) return;
    key[i] = i < n ? arrival[i] : 0x7fffffffffffffffLL;
    idx[i] = i < n ? (int32_t)i : 0x7fffffff;
    if (i + 1 < n && arrival[i] > arrival[i + 1]) *unsorted = 1u;
}
__global__ void slot_arrays_kernel(const int32_t* __restrict__ ord, const int64_t* __restrict__ off, int32_t n, long long* soff, int32_t* slen) {
    int32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int32_t qi = ord[r];
    const int64_t lo = off[qi];
    soff[r] = lo;
    slen[r] = (int32_t)(off[qi + 1] - lo);
}
__global__ void prio_init_kernel(const int64_t* __restrict__ prio, const int32_t* __restrict__ ord, int32_t n, long long np2,
                                 long long* key, int32_t* idx) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np2) return;
    key[i] = i < n ? prio[ord[i]] : 0x7fffffffffffffffLL;      // slot i holds query ord[i]
    idx[i] = i < n ? (int32_t)i : 0x7fffffff;
}
__global__ void prio_rank_kernel(const int32_t* __restrict__ pinv, int32_t n, int32_t* prank) {
    int32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) prank[pinv[r]] = r;
}
__global__ void bitonic_step_kernel(long long* key, int32_t* idx, long long np2, long long k, long long j, const unsigned int* needed) {
    if (needed && !*needed) return;
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np2) return;
    long long l = i ^ j;
    if (l > i) {
        long long ki = key[i], kl = key[l];
        int32_t ii = idx[i], il = idx[l];
        bool gt = ki > kl || (ki == kl && ii > il);
        bool up = (i & k) == 0;
        if (gt == up) { key[i] = kl; key[l] = ki; idx[i] = il; idx[l] = ii; }
    }
}

// Two steps of one stage in one pass (partner distances j and j / 2): a thread holds the four entries that differ in
// those two bits.
__global__ void bitonic_step2_kernel(long long* key, int32_t* idx, long long np2, long long k, long long j, const unsigned int* needed) {
    if (needed && !*needed) return;
    const long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= (np2 >> 2)) return;
    const long long j2 = j >> 1;
    const long long i0 = ((u & ~(j2 - 1)) << 2) | (u & (j2 - 1));      // u's bits with the two (adjacent) bit positions left out
    long long kk[4]; int32_t ii[4];
    const long long pos[4] = {i0, i0 | j2, i0 | j, i0 | j | j2};
#pragma unroll
    for (int r = 0; r < 4; ++r) { kk[r] = key[pos[r]]; ii[r] = idx[pos[r]]; }
    const bool up = (i0 & k) == 0;
    auto cx = [&](int x, int y) {
        const bool gt = kk[x] > kk[y] || (kk[x] == kk[y] && ii[x] > ii[y]);
        if (gt == up) { const long long tk = kk[x]; kk[x] = kk[y]; kk[y] = tk; const int32_t ti = ii[x]; ii[x] = ii[y]; ii[y] = ti; }
    };
    cx(0, 2); cx(1, 3);
    cx(0, 1); cx(2, 3);
#pragma unroll
    for (int r = 0; r < 4; ++r) { key[pos[r]] = kk[r]; idx[pos[r]] = ii[r]; }
}

// The steps of the same sort whose partner distance fits a tile of 4,096 pairs, done in shared memory: all stages
// k_lo .. k_hi when those are at most the tile (the start of the sort), otherwise the tail (distances below the
// tile) of the one stage k_lo = k_hi.
#define KLPM_SORT_TILE 4096
__global__ void __launch_bounds__(1024)
bitonic_tile_kernel(long long* key, int32_t* idx, long long np2, long long k_lo, long long k_hi, const unsigned int* needed) {
    if (needed && !*needed) return;
    __shared__ long long sk[KLPM_SORT_TILE];
    __shared__ int32_t si[KLPM_SORT_TILE];
    const int T = np2 < KLPM_SORT_TILE ? (int)np2 : KLPM_SORT_TILE;
    const long long base = (long long)blockIdx.x * T;
    for (int u = threadIdx.x; u < T; u += blockDim.x) { sk[u] = key[base + u]; si[u] = idx[base + u]; }
    __syncthreads();
    for (long long k = k_lo; k <= k_hi; k <<= 1) {
        const long long jmax = (k >> 1) < (long long)(T >> 1) ? (k >> 1) : (long long)(T >> 1);
        for (int j = (int)jmax; j > 0; j >>= 1) {
            for (int u = threadIdx.x; u < (T >> 1); u += blockDim.x) {
                const int i = ((u & ~(j - 1)) << 1) | (u & (j - 1)), l = i | j;      // the u-th pair at distance j
                const long long ki = sk[i], kl = sk[l];
                const int32_t ii = si[i], il = si[l];
                const bool gt = ki > kl || (ki == kl && ii > il);
                const bool up = ((base + i) & k) == 0;
                if (gt == up) { sk[i] = kl; sk[l] = ki; si[i] = il; si[l] = ii; }
            }
            __syncthreads();
        }
    }
    for (int u = threadIdx.x; u < T; u += blockDim.x) { key[base + u] = sk[u]; idx[base + u] = si[u]; }
}

// (key, idx) pairs ascending by key, then idx; np2 a power of two.  `needed` (nullable, device): 0 = they are in order already
void sort_pairs(long long* key, int32_t* idx, long long np2, cudaStream_t s, const unsigned int* needed = nullptr) {
    const long long T = np2 < KLPM_SORT_TILE ? np2 : KLPM_SORT_TILE;
    const unsigned tiles = (unsigned)(np2 / T), blocks = (unsigned)((np2 + 255) / 256);
    const unsigned blocks4 = (unsigned)(((np2 >> 2) + 255) / 256);
    if (T >= 2) bitonic_tile_kernel<<<tiles, 1024, 0, s>>>(key, idx, np2, 2, T, needed);
    for (long long k = T << 1; k <= np2; k <<= 1) {
        long long j = k >> 1;
        for (; (j >> 1) >= T; j >>= 2) bitonic_step2_kernel<<<blocks4, 256, 0, s>>>(key, idx, np2, k, j, needed);
        if (j >= T) bitonic_step_kernel<<<blocks, 256, 0, s>>>(key, idx, np2, k, j, needed);
        bitonic_tile_kernel<<<tiles, 1024, 0, s>>>(key, idx, np2, k, k, needed);
    }
}

}  // namespace

// ====================================================================================================
// host side
// ====================================================================================================
struct rt_tree {
    rt_config cfg;
    TreeDev dev;
    int device;
    cudaStream_t last_stream;
    unsigned long long* match_counter;
    // batched match: the order in which queries are taken (bucketed by first token)
    long long match_cap;    // queries the three arrays below hold
    int32_t* match_perm; unsigned short* match_bucket; unsigned int* match_hist;
    // match records (MatchState): which match call wrote the caller's, and the library's own for klpm_run without one
    unsigned long long version;        // bumped by every call that changes the tree
    unsigned long long ms_tag, ms_version;
    const void *ms_state, *ms_tok, *ms_off;
    int32_t ms_n;
    MatchState* own_state; long long own_state_cap;
    // klpm_run scratch
    long long run_cap;      // slots allocated (power of two)
    long long* run_key; int32_t* run_ord; int32_t* run_m; int32_t* run_hint; long long* run_pos;
    long long* run_soff; int32_t* run_slen; int32_t* run_ntok;
    unsigned int* run_unsorted;
    long long* run_pkey; int32_t* run_pinv; int32_t* run_prank;
    unsigned long long* run_partial; RunBcast* run_bc; RunSync* run_sy;
    // scratch of the grouped loop (trees without a budget)
    long long fast_cap;     // slots allocated (power of two)
    int4 *fast_lcp, *fast_pair; unsigned long long* grp_key;
    FDyn* fast_dyn; FStat* fast_stat; unsigned long long* fast_key_arr; int32_t* fast_mem;
    long long* fast_gh; int32_t* fast_gidx; unsigned int* fast_done;
    long long* fast_lk; int32_t* fast_ls;
    FastPost* fast_post; ChargeFn* fast_bsum;
    long long fast_mem_cap;  // entries of fast_mem
    int32_t* lru_parked; LruInfo* lru_info;     // grouped loop on a tree with a budget
    int32_t* lru_hintc; long long lru_hintc_cap;
    int2* lru_leaf_run; LNode* lru_node;
    ReplayInfo* replay_info;
    int run_path;           // which loop the last klpm_run took: 0 none yet, 1 one by one, 2 grouped
    void *run_slab, *fast_slab, *bulk_slab;   // the allocations behind the run_*, fast_* / grp_* and bulk_p* arrays
    int num_sms;
    int32_t *ins_pm, *ins_pnode, *ins_stop;   // insertion in order: matches of a part (one allocation), and whether a part ended early
    int32_t* claim;         // bulk insertion: per-node claim words (0x7fffffff when idle)
    long long bulk_cap;     // bulk insertion: prompts its per-prompt scratch holds
    int32_t *bulk_pend_a, *bulk_pend_b, *bulk_pm, *bulk_pnode, *bulk_poff;
    BulkSync* bulk_sync;
    // checkpoint (rt_checkpoint / rt_rollback): copies of everything a later call can modify
    bool ck_valid;
    int32_t *ck_parent, *ck_depth_start, *ck_span_len, *ck_nchild, *ck_clock_owner, *ck_first_tok;
    int64_t *ck_span_off, *ck_last_access;
    uint8_t* ck_dead;
    Entry* ck_table;
    TreeState* ck_st;
};

namespace {

#define CK(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) { \
    fprintf(stderr, "klpm: %s failed at %s:%d: %s\n", #call, __FILE__, __LINE__, cudaGetErrorString(e_)); return RT_ERR_CUDA; } } while (0)

template <typename P> rt_status dalloc(P** p, size_t count) {
    void* v = nullptr;
    CK(cudaMalloc(&v, count * sizeof(P) + 256));
    *p = (P*)v;
    return RT_OK;
}

void free_tree(rt_tree* t) {
    TreeDev& d = t->dev;
    cudaFree(d.parent); cudaFree(d.depth_start); cudaFree(d.span_len); cudaFree(d.nchild); cudaFree(d.first_tok);
    cudaFree(t->ck_first_tok);
    cudaFree(d.span_off); cudaFree(d.last_access); cudaFree(d.dead); cudaFree(d.clock_owner);
    cudaFree(d.table); cudaFree(d.pool); cudaFree(d.end_node); cudaFree(d.st); cudaFree(t->match_counter); cudaFree(t->run_unsorted);
    cudaFree(t->match_perm); cudaFree(t->match_bucket); cudaFree(t->match_hist); cudaFree(t->own_state);
    cudaFree(t->run_partial); cudaFree(t->run_bc); cudaFree(t->run_sy);
    cudaFree(t->lru_parked); cudaFree(t->lru_info); cudaFree(t->lru_hintc); cudaFree(t->lru_leaf_run); cudaFree(t->lru_node); cudaFree(t->replay_info);
    cudaFree(t->claim); cudaFree(t->ins_pm);
    cudaFree(t->bulk_sync);
    cudaFree(t->ck_parent); cudaFree(t->ck_depth_start); cudaFree(t->ck_span_len); cudaFree(t->ck_nchild);
    cudaFree(t->ck_clock_owner); cudaFree(t->ck_span_off); cudaFree(t->ck_last_access); cudaFree(t->ck_dead);
    cudaFree(t->ck_table); cudaFree(t->ck_st);
    cudaFree(t->run_slab); cudaFree(t->fast_slab); cudaFree(t->bulk_slab);
    delete t;
}

// One allocation for several arrays (an allocation takes 0.1 ms and more on a full device, and a first call needs thirty
// arrays).  Every part starts on a 256-byte boundary and has 256 bytes to spare.
struct SlabPart { void** p; size_t bytes; };
template <typename P> SlabPart slab_part(P** p, long long count) { SlabPart s; s.p = reinterpret_cast<void**>(p); s.bytes = (size_t)count * sizeof(P); return s; }
rt_status slab_alloc(void** slab, const SlabPart* parts, int n) {
    cudaFree(*slab);
    *slab = nullptr;
    size_t total = 0;
    for (int i = 0; i < n; ++i) { *parts[i].p = nullptr; total += ((parts[i].bytes + 255) & ~(size_t)255) + 256; }
    CK(cudaMalloc(slab, total));
    char* at = (char*)*slab;
    for (int i = 0; i < n; ++i) { *parts[i].p = at; at += ((parts[i].bytes + 255) & ~(size_t)255) + 256; }
    return RT_OK;
}

rt_status ensure_run_scratch(rt_tree* t, long long n) {
    long long np2 = 1;
    while (np2 < n) np2 <<= 1;
    if (np2 <= t->run_cap) return RT_OK;
    t->run_cap = 0;
    const SlabPart parts[] = {slab_part(&t->run_key, np2), slab_part(&t->run_ord, np2), slab_part(&t->run_m, np2), slab_part(&t->run_hint, np2),
                              slab_part(&t->run_pos, np2), slab_part(&t->run_soff, np2), slab_part(&t->run_slen, np2), slab_part(&t->run_ntok, np2),
                              slab_part(&t->run_pkey, np2), slab_part(&t->run_pinv, np2), slab_part(&t->run_prank, np2)};
    const rt_status s = slab_alloc(&t->run_slab, parts, (int)(sizeof(parts) / sizeof(parts[0])));
    if (s) return s;
    t->run_cap = np2;
    return RT_OK;
}

rt_status ensure_fast_scratch(rt_tree* t, long long n) {
    long long np2 = 1;
    while (np2 < n) np2 <<= 1;
    if (np2 <= t->fast_cap) return RT_OK;
    t->fast_cap = 0;
    // trees with a budget: groups formed by evictions are appended behind the first n entries
    t->fast_mem_cap = t->cfg.budget_tokens > 0 ? np2 + (8 * np2 > (1LL << 20) ? 8 * np2 : (1LL << 20)) : np2;
    const SlabPart parts[] = {slab_part(&t->fast_dyn, np2), slab_part(&t->fast_stat, np2), slab_part(&t->fast_key_arr, np2),
                              slab_part(&t->fast_mem, t->fast_mem_cap), slab_part(&t->fast_gh, np2), slab_part(&t->fast_gidx, np2),
                              slab_part(&t->fast_done, 3 * (np2 / 32 + 32)),      // processed bitmap, grouped bitmap, passed-over bitmap
                              slab_part(&t->fast_lk, np2), slab_part(&t->fast_ls, np2), slab_part(&t->fast_lcp, np2), slab_part(&t->fast_pair, 2 * np2),
                              slab_part(&t->grp_key, 4 * np2 + 1),                // keys, and as many counts and offsets (see run_impl)
                              slab_part(&t->fast_post, 1), slab_part(&t->fast_bsum, 1024)};
    const rt_status s = slab_alloc(&t->fast_slab, parts, (int)(sizeof(parts) / sizeof(parts[0])));
    if (s) return s;
    t->fast_cap = np2;
    return RT_OK;
}

bool params_ok(const klpm_params* p) {
    return p && p->policy >= KLPM_POLICY_FCFS && p->policy <= KLPM_POLICY_KLPM && p->k >= 1 && p->c_den >= 1 && p->c_num >= 0;
}

// Settings for tests and debugging (klpm_debug_set); process-wide, read when a call is made.
struct DebugKnobs {
    long long run_one_by_one;     // 1: trees without a budget take the one-by-one loop too
    long long fast_max_blocks;    // grouped loop: most tournament leaf blocks (0 = the built-in 8,192)
    long long fast_smem_kb;       // grouped loop: shared memory it may use (0 = the built-in 224 KB)
    long long wait_limit_ns;      // one-by-one loop: limit of a hand-over wait
    long long list_max_windows;   // grouped loop, everybody waiting: windows after which it gives up
};
DebugKnobs g_knobs = {0, 0, 0, KLPM_WAIT_LIMIT_NS, 0x7fffffffLL};

SelectScratch* g_select_scratch[64] = {nullptr};
TopkScratch* g_topk_scratch[64] = {nullptr};
StaticSelectScratch* g_select_static_addr[64] = {nullptr};   // device address of g_select_static, per device

// Many prompts at once into a tree without a budget (see the bulk kernels).  Waits for the stream once per round.
rt_status ensure_bulk_scratch(rt_tree* t, int32_t n) {
    rt_status st = RT_OK;
    if (n > t->bulk_cap) {                     // per-prompt scratch, kept for later calls
        t->bulk_cap = 0;
        const SlabPart parts[] = {slab_part(&t->bulk_pend_a, n), slab_part(&t->bulk_pend_b, n), slab_part(&t->bulk_pm, n), slab_part(&t->bulk_pnode, n),
                                  slab_part(&t->bulk_poff, n)};
        if ((st = slab_alloc(&t->bulk_slab, parts, (int)(sizeof(parts) / sizeof(parts[0]))))) return st;
        t->bulk_cap = n;
    }
    if (!t->bulk_sync && (st = dalloc(&t->bulk_sync, 1))) return st;        // list lengths, work counter, grid barrier
    return RT_OK;
}

// `state` (nullable): records of a batched match of these prompts against the tree as it is now; the first round
// then needs no walk.  Everything is enqueued on `s`; nothing waits for the device.
// `list_ready`: bulk_pend_a already holds the n prompts to store (entries < 0 are skipped) and *n_total_dev how many they are.
rt_status bulk_insert(rt_tree* t, const int32_t* d_tokens, const int64_t* d_offsets, int32_t n, cudaStream_t s,
                      const MatchState* state = nullptr, unsigned long long tag = 0, bool list_ready = false,
                      const int32_t* n_total_dev = nullptr) {
    rt_status st = ensure_bulk_scratch(t, n);
    if (st) return st;
    BulkSync* g = t->bulk_sync;
    // claim words start idle (an earlier call that ran out of capacity may have left some set)
    bulk_fill_kernel<<<(unsigned)((t->dev.max_nodes + 255) / 256), 256, 0, s>>>(t->claim, t->dev.max_nodes, 0x7fffffff);
    if (!list_ready) bulk_iota_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(t->bulk_pend_a, n);
    CK(cudaMemsetAsync(g, 0, sizeof(BulkSync), s));
    BulkArgs a;
    a.tok = d_tokens; a.off = d_offsets; a.pend_in = t->bulk_pend_a; a.pend_out = t->bulk_pend_b; a.n_out = &g->cnt_w[0];
    a.pend_next = t->bulk_pend_a; a.n_next = &g->cnt_a[0]; a.n_walk = &g->n_walk;      // the walk has consumed pend_a by the time apply refills it
    a.claim = t->claim; a.pm = t->bulk_pm; a.pnode = t->bulk_pnode; a.poff = t->bulk_poff;
    long long blocks = ((long long)n + 7) / 8;
    if (blocks > (long long)t->num_sms * 8) blocks = (long long)t->num_sms * 8;
    // the first round: every prompt from the root (or from its match record), then cuts and leaves
    if (state) bulk_from_state_kernel<<<(unsigned)blocks, 256, 0, s>>>(t->dev, a, state, tag, (unsigned)n);
    else bulk_walk_kernel<<<(unsigned)blocks, 256, 0, s>>>(t->dev, a, (unsigned)n);
    bulk_apply_kernel<<<(unsigned)blocks, 256, 0, s>>>(t->dev, a);
    CK(cudaGetLastError());
    // every later round, and the clock, in one cooperative kernel
    int per_sm = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bulk_rounds_kernel, 256, 0));
    if (per_sm < 1) return RT_ERR_CUDA;
    const unsigned grid = (unsigned)t->num_sms * (unsigned)(per_sm < 2 ? per_sm : 2);
    long long n_total = n, limit = g_knobs.wait_limit_ns;
    void* kargs[] = {(void*)&t->dev, (void*)&a, (void*)&g, (void*)&n_total, (void*)&n_total_dev, (void*)&limit};
    CK(cudaLaunchCooperativeKernel((void*)bulk_rounds_kernel, dim3(grid), dim3(256), kargs, 0, s));
    return RT_OK;
}

// Batches up to these sizes go to match_wide_kernel.  Cold caches, wide against the ordered persistent kernels:
//   with a budget (hop by hop): 32 queries 10 / 21 us, 4,736 32 / 54, 14,000 56 / 77, 48,000 140 / 159
//   without (along runs), medium tree: 32 queries 12 / 33 us, 4,736 34 / 62, 14,000 69 / 89, 48,000 184 / 187; deep edges
//   (adversarial): 32 queries 27 / 96, 4,736 111 / 153, 14,000 201 / 218, 24,000 307 / 288: there every query of a trunk
//   reads the trunk from HBM again unless they are taken together.
#define KLPM_WIDE_MAX_CHAIN 16384
#define KLPM_WIDE_MAX_HOPS 65536
static_assert(KLPM_INSERT_PART <= KLPM_WIDE_MAX_CHAIN && KLPM_INSERT_PART <= KLPM_WIDE_MAX_HOPS, "the parts of an insertion in order are matched by match_wide_kernel");
std::atomic<unsigned long long> g_match_tag{0};

// The batched match: the order in which the queries are taken, then the kernel.  `state` (nullable) receives the
// per-query records, stamped with `tag`.
rt_status launch_match(rt_tree* t, const int32_t* d_q_tokens, const int64_t* d_q_offsets, int32_t nq, int32_t* d_match_len,
                       int32_t* d_term_node, int32_t* d_term_off, MatchState* state, unsigned long long tag, cudaStream_t s,
                       int32_t in_order = 0) {
    if (nq <= (t->cfg.budget_tokens == 0 ? KLPM_WIDE_MAX_CHAIN : KLPM_WIDE_MAX_HOPS)) {
        // as many warps per query (a power of two, 8 at most) as leave every query of the batch resident at once
        const long long resident = (long long)t->num_sms * 32;
        int warps = 8;
        while (warps > 1 && (long long)nq * warps > resident) warps >>= 1;
        if (t->cfg.budget_tokens == 0) match_wide_kernel<true><<<(unsigned)nq, warps * 32, 0, s>>>(t->dev, d_q_tokens, d_q_offsets, d_match_len,
                                                                                                  d_term_node, d_term_off, state, tag, in_order, t->ins_stop);
        else match_wide_kernel<false><<<(unsigned)nq, warps * 32, 0, s>>>(t->dev, d_q_tokens, d_q_offsets, d_match_len, d_term_node,
                                                                          d_term_off, state, tag, in_order, t->ins_stop);
        CK(cudaGetLastError());
        return RT_OK;
    }
    if (nq > t->match_cap) {
        cudaFree(t->match_perm); cudaFree(t->match_bucket);
        t->match_perm = nullptr; t->match_bucket = nullptr; t->match_cap = 0;
        rt_status st;
        if ((st = dalloc(&t->match_perm, nq)) || (st = dalloc(&t->match_bucket, nq))) return st;
        t->match_cap = nq;
    }
    if (!t->match_hist) { rt_status st = dalloc(&t->match_hist, KLPM_ORDER_BUCKETS); if (st) return st; }
    const unsigned qb = (unsigned)((nq + 255) / 256);
    CK(cudaMemsetAsync(t->match_hist, 0, KLPM_ORDER_BUCKETS * sizeof(unsigned int), s));
    order_hist_kernel<<<qb, 256, 0, s>>>(d_q_tokens, d_q_offsets, nq, t->match_hist, t->match_bucket);
    order_scan_kernel<<<1, 1024, 0, s>>>(t->match_hist);
    order_scatter_kernel<<<qb, 256, 0, s>>>(t->match_bucket, nq, t->match_hist, t->match_perm);
    const int32_t* perm = t->match_perm;
    CK(cudaMemsetAsync(t->match_counter, 0, sizeof(unsigned long long), s));
    const int threads = 256, warps_per_block = threads / 32;
    long long blocks = ((long long)nq + warps_per_block - 1) / warps_per_block;
    const long long max_blocks = (long long)t->num_sms * 8;
    if (blocks > max_blocks) blocks = max_blocks;
    if (t->cfg.budget_tokens == 0) {
        if (state) match_chain_kernel<true><<<(unsigned)blocks, threads, 0, s>>>(t->dev, d_q_tokens, d_q_offsets, nq, perm, d_match_len,
                                                                               d_term_node, d_term_off, state, tag, t->match_counter);
        else match_chain_kernel<false><<<(unsigned)blocks, threads, 0, s>>>(t->dev, d_q_tokens, d_q_offsets, nq, perm, d_match_len,
                                                                            d_term_node, d_term_off, nullptr, 0ULL, t->match_counter);
    } else {
        match_batch_kernel<<<(unsigned)blocks, threads, 0, s>>>(t->dev, d_q_tokens, d_q_offsets, nq, perm, d_match_len,
                                                               d_term_node, d_term_off, state, tag, t->match_counter);
    }
    CK(cudaGetLastError());
    return RT_OK;
}

}  // namespace

extern "C" {

int32_t klpm_abi_version(void) { return KLPM_ABI_VERSION; }

rt_status rt_create(const rt_config* cfg, rt_tree** out) {
    if (!cfg || !out || cfg->max_nodes < 2 || cfg->max_pool_tokens < 1 || cfg->budget_tokens < 0 ||
        cfg->max_nodes > 0x7ffffff0LL || cfg->max_clock < 0) return RT_ERR_INVALID;
    rt_tree* t = new (std::nothrow) rt_tree();
    if (!t) return RT_ERR_CUDA;
    memset(t, 0, sizeof(*t));
    t->cfg = *cfg;
    CK(cudaGetDevice(&t->device));
    CK(cudaDeviceGetAttribute(&t->num_sms, cudaDevAttrMultiProcessorCount, t->device));
    TreeDev& d = t->dev;
    d.max_nodes = cfg->max_nodes;
    d.max_pool = cfg->max_pool_tokens;
    d.max_clock = (cfg->max_clock > 0 ? cfg->max_clock : cfg->max_nodes) + 2;
    d.budget = cfg->budget_tokens;
    unsigned long long cap = 1024;
    while (cap < 2ULL * (unsigned long long)cfg->max_nodes) cap <<= 1;
    d.table_mask = cap - 1;
    rt_status s = RT_OK;
    if ((s = dalloc(&d.parent, d.max_nodes)) || (s = dalloc(&d.depth_start, d.max_nodes)) ||
        (s = dalloc(&d.span_len, d.max_nodes)) || (s = dalloc(&d.nchild, d.max_nodes)) || (s = dalloc(&d.first_tok, d.max_nodes)) ||
        (s = dalloc(&d.span_off, d.max_nodes)) || (s = dalloc(&d.last_access, d.max_nodes)) ||
        (s = dalloc(&d.dead, d.max_nodes)) || (s = dalloc(&d.clock_owner, d.max_clock)) ||
        (s = dalloc(&d.table, cap)) || (s = dalloc(&d.pool, d.max_pool)) || (s = dalloc(&d.st, 1)) ||
        (s = dalloc(&d.end_node, d.max_pool)) ||
        (s = dalloc(&t->match_counter, 1)) || (s = dalloc(&t->run_unsorted, 1)) || (s = dalloc(&t->run_partial, 1024)) || (s = dalloc(&t->run_bc, 1)) || (s = dalloc(&t->run_sy, 1)) ||
        (s = dalloc(&t->ins_pm, 2 * KLPM_INSERT_PART + 1)) || (s = dalloc(&t->claim, d.max_nodes))) {
        free_tree(t);
        return s;
    }
    t->ins_pnode = t->ins_pm + KLPM_INSERT_PART; t->ins_stop = t->ins_pnode + KLPM_INSERT_PART;
    // root: node 0, empty edge
    cudaError_t e = cudaMemset(d.table, 0, cap * sizeof(Entry));
    if (e == cudaSuccess) e = cudaMemset(d.end_node, 0xff, d.max_pool * sizeof(int32_t) + 256);
    if (e == cudaSuccess) e = cudaMemset(d.clock_owner, 0, d.max_clock * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(d.parent, 0, sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(d.depth_start, 0, sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(d.span_len, 0, sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(d.nchild, 0, sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(d.first_tok, 0, sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(d.span_off, 0, sizeof(int64_t));
    if (e == cudaSuccess) e = cudaMemset(d.last_access, 0, sizeof(int64_t));
    if (e == cudaSuccess) e = cudaMemset(d.dead, 0, 1);
    if (e == cudaSuccess) {
        bulk_fill_kernel<<<(unsigned)((d.max_nodes + 255) / 256), 256>>>(t->claim, d.max_nodes, 0x7fffffff);
        e = cudaGetLastError();
    }
    TreeState st0;
    memset(&st0, 0, sizeof(st0));
    st0.n_nodes = 1;
    st0.lru_cursor = 1;
    if (e == cudaSuccess) e = cudaMemcpy(d.st, &st0, sizeof(st0), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        fprintf(stderr, "klpm: tree initialisation failed: %s\n", cudaGetErrorString(e));
        free_tree(t);
        return RT_ERR_CUDA;
    }
    *out = t;
    return RT_OK;
}

rt_status rt_destroy(rt_tree* tree) {
    if (!tree) return RT_ERR_INVALID;
    cudaDeviceSynchronize();
    free_tree(tree);
    return RT_OK;
}

rt_status rt_insert(rt_tree* tree, const int32_t* d_tokens, const int64_t* d_offsets, int32_t n,
                    int32_t* d_new_tokens, void* stream) {
    if (!tree || n < 0 || (n > 0 && (!d_tokens || !d_offsets))) return RT_ERR_INVALID;
    if (n == 0) return RT_OK;
    tree->version++;
    if (!d_new_tokens && tree->cfg.budget_tokens == 0 && n >= 64) {
        tree->last_stream = (cudaStream_t)stream;
        return bulk_insert(tree, d_tokens, d_offsets, n, (cudaStream_t)stream);
    }
    // one after the other, a part at a time: all matched at once against the tree as it is, then inserted in order
    cudaStream_t s = (cudaStream_t)stream;
    tree->last_stream = s;
    for (int32_t at = 0; at < n;) {
        const int32_t part = n - at < KLPM_INSERT_PART ? n - at : KLPM_INSERT_PART;
        const rt_status st = launch_match(tree, d_tokens, d_offsets + at, part, tree->ins_pm, tree->ins_pnode, nullptr, nullptr, 0ULL, s,
                                          at == 0 ? 1 : 2);
        if (st) return st;
        InsertArgs a;
        a.tok = d_tokens; a.off = d_offsets + at; a.n = part; a.new_tokens = d_new_tokens ? d_new_tokens + at : nullptr;
        a.pm = tree->ins_pm; a.pnode = tree->ins_pnode; a.stop = tree->ins_stop; a.first = at == 0;
        insert_seq_kernel<<<1, 512, 0, s>>>(tree->dev, a);
        CK(cudaGetLastError());
        at += part;
    }
    return RT_OK;
}

rt_status rt_build(const int32_t* d_tokens, const int64_t* d_offsets, int32_t n_prompts, const rt_config* cfg,
                   void* stream, rt_tree** out) {
    if (!out || n_prompts < 0) return RT_ERR_INVALID;
    rt_tree* t = nullptr;
    rt_status s = rt_create(cfg, &t);
    if (s) return s;
    s = rt_insert(t, d_tokens, d_offsets, n_prompts, nullptr, stream);
    if (s) { rt_destroy(t); return s; }
    *out = t;
    return RT_OK;
}

rt_status rt_match_batch_ex(rt_tree* tree, const int32_t* d_q_tokens, const int64_t* d_q_offsets, int32_t nq,
                            int32_t* d_match_len, int32_t* d_term_node, int32_t* d_term_off, klpm_match_state* d_state,
                            void* stream) {
    if (!tree || nq < 0 || (nq > 0 && (!d_q_tokens || !d_q_offsets || !d_match_len))) return RT_ERR_INVALID;
    if (nq == 0) return RT_OK;
    cudaStream_t s = (cudaStream_t)stream;
    tree->last_stream = s;
    unsigned long long tag = 0;
    if (d_state) {
        tag = ++g_match_tag;
        tree->ms_tag = tag; tree->ms_version = tree->version; tree->ms_state = d_state; tree->ms_tok = d_q_tokens;
        tree->ms_off = d_q_offsets; tree->ms_n = nq;
    }
    return launch_match(tree, d_q_tokens, d_q_offsets, nq, d_match_len, d_term_node, d_term_off,
                        reinterpret_cast<MatchState*>(d_state), tag, s);
}

rt_status rt_match_batch(const rt_tree* tree, const int32_t* d_q_tokens, const int64_t* d_q_offsets, int32_t nq,
                         int32_t* d_match_len, int32_t* d_term_node, int32_t* d_term_off, void* stream) {
    return rt_match_batch_ex(const_cast<rt_tree*>(tree), d_q_tokens, d_q_offsets, nq, d_match_len, d_term_node, d_term_off,
                             nullptr, stream);
}

rt_status rt_stats(rt_tree* tree, int64_t* n_nodes, int64_t* n_tokens, int64_t* clock, int64_t* evictions, int64_t* pool_used) {
    if (!tree) return RT_ERR_INVALID;
    CK(cudaStreamSynchronize(tree->last_stream));
    TreeState st;
    CK(cudaMemcpy(&st, tree->dev.st, sizeof(st), cudaMemcpyDeviceToHost));
    if (n_nodes) *n_nodes = st.live_nodes;
    if (n_tokens) *n_tokens = st.tokens_live;
    if (clock) *clock = st.clock;
    if (evictions) *evictions = st.evictions;
    if (pool_used) *pool_used = st.pool_used;
    return RT_OK;
}

rt_status rt_clone(rt_tree* tree, void* stream, rt_tree** out) {
    if (!tree || !out) return RT_ERR_INVALID;
    rt_tree* c = nullptr;
    rt_status s = rt_create(&tree->cfg, &c);
    if (s) return s;
    const TreeDev& a = tree->dev;
    TreeDev& b = c->dev;
    const unsigned long long cap = a.table_mask + 1;
    cudaStream_t st = (cudaStream_t)stream;
    tree->last_stream = st;
    c->last_stream = st;
    const cudaMemcpyKind k = cudaMemcpyDeviceToDevice;
    cudaError_t e = cudaMemcpyAsync(b.parent, a.parent, a.max_nodes * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.depth_start, a.depth_start, a.max_nodes * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.span_len, a.span_len, a.max_nodes * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.nchild, a.nchild, a.max_nodes * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.first_tok, a.first_tok, a.max_nodes * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.span_off, a.span_off, a.max_nodes * sizeof(int64_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.last_access, a.last_access, a.max_nodes * sizeof(int64_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.dead, a.dead, a.max_nodes, k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.clock_owner, a.clock_owner, a.max_clock * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.table, a.table, cap * sizeof(Entry), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.pool, a.pool, a.max_pool * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.end_node, a.end_node, a.max_pool * sizeof(int32_t), k, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.st, a.st, sizeof(TreeState), k, st);
    if (e != cudaSuccess) {
        fprintf(stderr, "klpm: rt_clone failed: %s\n", cudaGetErrorString(e));
        cudaStreamSynchronize(st);
        free_tree(c);
        return RT_ERR_CUDA;
    }
    *out = c;
    return RT_OK;
}

// Everything a later call can modify, from the tree to its checkpoint or back.
static rt_status copy_checkpoint(rt_tree* t, bool back, cudaStream_t s) {
    TreeDev& d = t->dev;
    const size_t cap = (size_t)d.table_mask + 1, nodes = (size_t)d.max_nodes;
    CopyList L;
    L.n = 0;
    long long total = 0;
    auto add = [&](void* tree_side, void* kept, size_t bytes) {
        L.dst[L.n] = reinterpret_cast<int4*>(back ? tree_side : kept);
        L.src[L.n] = reinterpret_cast<const int4*>(back ? kept : tree_side);
        total += (long long)((bytes + 15) / 16);
        L.end[L.n++] = total;
    };
    add(d.table, t->ck_table, cap * sizeof(Entry));
    add(d.parent, t->ck_parent, nodes * sizeof(int32_t));
    add(d.depth_start, t->ck_depth_start, nodes * sizeof(int32_t));
    add(d.span_len, t->ck_span_len, nodes * sizeof(int32_t));
    add(d.nchild, t->ck_nchild, nodes * sizeof(int32_t));
    add(d.first_tok, t->ck_first_tok, nodes * sizeof(int32_t));
    add(d.span_off, t->ck_span_off, nodes * sizeof(int64_t));
    add(d.last_access, t->ck_last_access, nodes * sizeof(int64_t));
    add(d.dead, t->ck_dead, nodes);
    add(d.clock_owner, t->ck_clock_owner, (size_t)d.max_clock * sizeof(int32_t));
    add(d.st, t->ck_st, sizeof(TreeState));
    long long blocks = (total + 512 * 4 - 1) / (512 * 4);
    if (blocks > (long long)t->num_sms * 4) blocks = (long long)t->num_sms * 4;
    copy_list_kernel<<<(unsigned)blocks, 512, 0, s>>>(L);
    CK(cudaGetLastError());
    return RT_OK;
}

rt_status rt_checkpoint(rt_tree* tree, void* stream) {
    if (!tree) return RT_ERR_INVALID;
    TreeDev& d = tree->dev;
    const unsigned long long cap = d.table_mask + 1;
    rt_status s = RT_OK;
    if (!tree->ck_parent) {
        if ((s = dalloc(&tree->ck_parent, d.max_nodes)) || (s = dalloc(&tree->ck_depth_start, d.max_nodes)) ||
            (s = dalloc(&tree->ck_span_len, d.max_nodes)) || (s = dalloc(&tree->ck_nchild, d.max_nodes)) ||
            (s = dalloc(&tree->ck_first_tok, d.max_nodes)) ||
            (s = dalloc(&tree->ck_span_off, d.max_nodes)) || (s = dalloc(&tree->ck_last_access, d.max_nodes)) ||
            (s = dalloc(&tree->ck_dead, d.max_nodes)) || (s = dalloc(&tree->ck_clock_owner, d.max_clock)) ||
            (s = dalloc(&tree->ck_table, cap)) || (s = dalloc(&tree->ck_st, 1))) return s;
    }
    cudaStream_t st = (cudaStream_t)stream;
    tree->last_stream = st;
    if ((s = copy_checkpoint(tree, false, st))) return s;
    tree->ck_valid = true;
    return RT_OK;
}

rt_status rt_rollback(rt_tree* tree, void* stream) {
    if (!tree || !tree->ck_valid) return RT_ERR_INVALID;
    tree->version++;
    cudaStream_t st = (cudaStream_t)stream;
    tree->last_stream = st;
    return copy_checkpoint(tree, true, st);
}

rt_status rt_status_detail(rt_tree* tree, int32_t* detail) {
    if (!tree || !detail) return RT_ERR_INVALID;
    CK(cudaStreamSynchronize(tree->last_stream));
    TreeState st;
    CK(cudaMemcpy(&st, tree->dev.st, sizeof(st), cudaMemcpyDeviceToHost));
    *detail = st.detail;
    return RT_OK;
}

rt_status rt_sync_status(rt_tree* tree, void* stream) {
    if (!tree) return RT_ERR_INVALID;
    CK(cudaStreamSynchronize((cudaStream_t)stream));
    TreeState st;
    CK(cudaMemcpy(&st, tree->dev.st, sizeof(st), cudaMemcpyDeviceToHost));
    return (rt_status)st.status;
}

static unsigned small_threads(int32_t nq) { const unsigned w = ((unsigned)nq + 31) / 32; return (w < 1 ? 1 : w > 32 ? 32 : w) * 32; }
static rt_status select_small(const int32_t* d_match_len, const int64_t* d_arrival, const uint8_t* d_waiting, int32_t nq,
                              int64_t pick_counter, const klpm_params* params, int32_t* d_pick, void* stream) {
    const bool fcfs_turn = params->policy == KLPM_POLICY_FCFS || (params->policy == KLPM_POLICY_KLPM && pick_counter % params->k == 0);
    cudaStream_t s = (cudaStream_t)stream;
    if (fcfs_turn) select_small_kernel<false><<<1, small_threads(nq), 0, s>>>(d_match_len, d_arrival, d_waiting, nq, 1, d_pick);
    else select_small_kernel<true><<<1, small_threads(nq), 0, s>>>(d_match_len, d_arrival, d_waiting, nq, 1, d_pick);
    CK(cudaGetLastError());
    return RT_OK;
}

rt_status klpm_select(const int32_t* d_match_len, const int64_t* d_arrival, const uint8_t* d_waiting, int32_t nq,
                      int64_t pick_counter, const klpm_params* params, int32_t* d_pick, void* stream) {
    if (!params_ok(params) || nq < 0 || !d_pick || pick_counter < 0 ||
        (nq > 0 && (!d_match_len || !d_arrival || !d_waiting))) return RT_ERR_INVALID;
    if (nq <= KLPM_SELECT_SMALL) return select_small(d_match_len, d_arrival, d_waiting, nq, pick_counter, params, d_pick, stream);
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return RT_ERR_INVALID;
    if (!g_select_scratch[dev]) {
        SelectScratch* p = nullptr;
        CK(cudaMalloc((void**)&p, sizeof(SelectScratch)));
        CK(cudaMemset(p, 0, sizeof(SelectScratch)));
        g_select_scratch[dev] = p;
    }
    const bool fcfs_turn = params->policy == KLPM_POLICY_FCFS ||
                           (params->policy == KLPM_POLICY_KLPM && pick_counter % params->k == 0);
    long long blocks = ((long long)nq + 2047) / 2048;
    if (blocks < 1) blocks = 1;
    if (blocks > 1024) blocks = 1024;
    cudaStream_t s = (cudaStream_t)stream;
    if (fcfs_turn) select_kernel<false><<<(unsigned)blocks, 512, 0, s>>>(d_match_len, d_arrival, d_waiting, nq, d_pick, g_select_scratch[dev]);
    else select_kernel<true><<<(unsigned)blocks, 512, 0, s>>>(d_match_len, d_arrival, d_waiting, nq, d_pick, g_select_scratch[dev]);
    CK(cudaGetLastError());
    return RT_OK;
}

rt_status klpm_select_topk(const int32_t* d_match_len, const int64_t* d_arrival, const uint8_t* d_waiting, int32_t nq,
                           int32_t kk, int32_t* d_out, void* stream) {
    if (nq < 0 || kk < 1 || kk > KLPM_TOPK_MAX || !d_out || (nq > 0 && (!d_match_len || !d_arrival || !d_waiting))) return RT_ERR_INVALID;
    if (nq <= KLPM_SELECT_SMALL) {
        select_small_kernel<true><<<1, small_threads(nq), 0, (cudaStream_t)stream>>>(d_match_len, d_arrival, d_waiting, nq, kk, d_out);
        CK(cudaGetLastError());
        return RT_OK;
    }
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return RT_ERR_INVALID;
    if (!g_topk_scratch[dev]) {
        TopkScratch* p = nullptr;
        CK(cudaMalloc((void**)&p, sizeof(TopkScratch)));
        CK(cudaMemset(p, 0, sizeof(TopkScratch)));
        g_topk_scratch[dev] = p;
    }
    long long blocks = ((long long)nq + 4095) / 4096;
    if (blocks < 1) blocks = 1;
    if (blocks > KLPM_TOPK_BLOCKS) blocks = KLPM_TOPK_BLOCKS;
    select_topk_kernel<<<(unsigned)blocks, 512, 0, (cudaStream_t)stream>>>(d_match_len, d_arrival, d_waiting, nq, kk, d_out,
                                                                            g_topk_scratch[dev]);
    CK(cudaGetLastError());
    return RT_OK;
}

rt_status klpm_select_noalloc(const int32_t* d_match_len, const int64_t* d_arrival, const uint8_t* d_waiting, int32_t nq,
                              int64_t pick_counter, const klpm_params* params, int32_t* d_pick, void* stream) {
    if (!params_ok(params) || nq < 0 || !d_pick || pick_counter < 0 ||
        (nq > 0 && (!d_match_len || !d_arrival || !d_waiting))) return RT_ERR_INVALID;
    if (nq > KLPM_SELECT_NOALLOC_MAX_QUERIES) {
        fprintf(stderr, "klpm_select_noalloc: nq = %d is above the fixed-scratch limit of %d queries; "
                        "use klpm_select for larger queues\n", nq, KLPM_SELECT_NOALLOC_MAX_QUERIES);
        return RT_ERR_TOO_LARGE;
    }
    if (nq <= KLPM_SELECT_SMALL) return select_small(d_match_len, d_arrival, d_waiting, nq, pick_counter, params, d_pick, stream);
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return RT_ERR_INVALID;
    if (!g_select_static_addr[dev]) {
        // In host code the array's name only stands for the symbol; the kernel needs its device address.
        StaticSelectScratch* p = nullptr;
        CK(cudaGetSymbolAddress((void**)&p, g_select_static));
        if (!p) return RT_ERR_CUDA;
        g_select_static_addr[dev] = p;
    }
    StaticSelectScratch* sc = g_select_static_addr[dev];
    cudaStream_t s = (cudaStream_t)stream;
    // the arrival counter must start at zero whatever an earlier call left behind
    CK(cudaMemsetAsync(&sc->ticket, 0, sizeof(unsigned int), s));
    const bool fcfs_turn = params->policy == KLPM_POLICY_FCFS ||
                           (params->policy == KLPM_POLICY_KLPM && pick_counter % params->k == 0);
    long long blocks = ((long long)nq + 2047) / 2048;
    if (blocks < 1) blocks = 1;
    if (blocks > KLPM_SELECT_NOALLOC_BLOCKS) blocks = KLPM_SELECT_NOALLOC_BLOCKS;
    if (fcfs_turn) select_static_kernel<false><<<(unsigned)blocks, 512, 0, s>>>(d_match_len, d_arrival, d_waiting, nq, d_pick, sc);
    else select_static_kernel<true><<<(unsigned)blocks, 512, 0, s>>>(d_match_len, d_arrival, d_waiting, nq, d_pick, sc);
    CK(cudaGetLastError());
    return RT_OK;
}

static rt_status run_impl(rt_tree* tree, const int32_t* d_q_tokens, const int64_t* d_q_offsets, const int64_t* d_arrival,
                          int32_t n, const klpm_params* params, const int64_t* d_tie_priority, int32_t score_mode,
                          const klpm_match_state* d_match_state, int32_t* d_order, int32_t* d_uncached, int64_t* d_ttft,
                          int64_t* d_completion, const int32_t* d_fixed, int32_t n_fixed, void* stream);

rt_status klpm_replay(rt_tree* tree, const int32_t* d_order, int32_t n_order, const int32_t* d_q_tokens,
                      const int64_t* d_q_offsets, const int64_t* d_arrival, int32_t n_queries, const klpm_params* params,
                      int32_t* d_uncached, int64_t* d_ttft, int64_t* d_completion, void* stream) {
    if (!tree || !params_ok(params) || n_order < 0 || n_queries < 0 ||
        (n_order > 0 && (!d_order || !d_q_tokens || !d_q_offsets || !d_arrival || !d_uncached || !d_ttft))) return RT_ERR_INVALID;
    if (n_order == 0) return RT_OK;
    // The same loop as klpm_run with the order given instead of picked (every query's match state is kept, a processed
    // prompt re-matches its group only, the tree is written once at the end).  The debug setting run_one_by_one keeps
    // the plain form: one CTA that walks, charges and stores one prompt after the other on the tree itself.
    if (!g_knobs.run_one_by_one && n_queries > 0)
        return run_impl(tree, d_q_tokens, d_q_offsets, d_arrival, n_queries, params, nullptr, 0, nullptr, nullptr, d_uncached, d_ttft,
                        d_completion, d_order, n_order, stream);
    tree->version++;
    SeqArgs a;
    memset(&a, 0, sizeof(a));
    a.tok = d_q_tokens; a.off = d_q_offsets; a.arrival = d_arrival; a.order = d_order; a.n = n_order; a.n_queries = n_queries;
    a.c_num = params->c_num; a.c_den = params->c_den; a.start_tick = params->start_tick;
    a.uncached = d_uncached; a.ttft = d_ttft; a.completion = d_completion;
    tree->last_stream = (cudaStream_t)stream;
    sequential_kernel<<<1, 1024, 0, (cudaStream_t)stream>>>(tree->dev, a);
    CK(cudaGetLastError());
    return RT_OK;
}

rt_status klpm_batch_times(const int32_t* d_order, int32_t n_order, const int64_t* d_arrival, const int64_t* d_completion,
                           int32_t n_queries, int32_t batch_size, int64_t* d_ttft_b, int64_t* d_completion_b,
                           int32_t* d_n_skipped, void* stream) {
    if (n_order < 0 || n_queries < 0 || batch_size < 1 ||
        (n_order > 0 && (!d_order || !d_arrival || !d_completion || !d_ttft_b || !d_completion_b))) return RT_ERR_INVALID;
    if (d_n_skipped) CK(cudaMemsetAsync(d_n_skipped, 0, sizeof(int32_t), (cudaStream_t)stream));
    if (n_order == 0) return RT_OK;
    batch_times_kernel<<<(unsigned)((n_order + 255) / 256), 256, 0, (cudaStream_t)stream>>>(d_order, n_order, d_arrival, d_completion,
                                                                                           n_queries, batch_size, d_ttft_b,
                                                                                           d_completion_b, d_n_skipped);
    CK(cudaGetLastError());
    return RT_OK;
}

// klpm_run_ex, and klpm_replay when d_fixed (a processing order of n_fixed entries) is given: then d_order is null,
// no decision is taken by a policy, and only the prompts of the order are charged and stored.
static rt_status run_impl(rt_tree* tree, const int32_t* d_q_tokens, const int64_t* d_q_offsets, const int64_t* d_arrival,
                          int32_t n, const klpm_params* params, const int64_t* d_tie_priority, int32_t score_mode,
                          const klpm_match_state* d_match_state, int32_t* d_order, int32_t* d_uncached, int64_t* d_ttft,
                          int64_t* d_completion, const int32_t* d_fixed, int32_t n_fixed, void* stream) {
    if (!tree || !params_ok(params) || n < 0 || score_mode < 0 || score_mode > 1 ||
        (n > 0 && (!d_q_tokens || !d_q_offsets || !d_arrival || (!d_order && !d_fixed) || !d_uncached || !d_ttft))) return RT_ERR_INVALID;
    if (n == 0) return RT_OK;
    // records of a batched match are only good for the queries they were written for and the tree as it was then
    if (d_match_state && (tree->ms_state != (const void*)d_match_state || tree->ms_n != n || tree->ms_tok != (const void*)d_q_tokens ||
                          tree->ms_off != (const void*)d_q_offsets || tree->ms_version != tree->version)) return RT_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    tree->last_stream = s;
    tree->version++;
    rt_status st = ensure_run_scratch(tree, n);
    if (st) return st;
    long long np2 = 1;
    while (np2 < n) np2 <<= 1;
    // A tree without a budget takes the grouped loop (unless the debug setting run_one_by_one is on).
    const bool grouped = !g_knobs.run_one_by_one;
    const bool lru = tree->cfg.budget_tokens > 0;
    // slots = queries ordered by (arrival, index); for a given order, the queries in index order
    if (d_fixed) {
        replay_slots_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d_arrival, n, tree->run_key, tree->run_ord);
        CK(cudaGetLastError());
    } else {
        unsigned blocks = (unsigned)((np2 + 255) / 256);
        CK(cudaMemsetAsync(tree->run_unsorted, 0, sizeof(unsigned int), s));
        rank_init_kernel<<<blocks, 256, 0, s>>>(d_arrival, n, np2, tree->run_key, tree->run_ord, tree->run_unsorted);
        sort_pairs(tree->run_key, tree->run_ord, np2, s, tree->run_unsorted);
        if (!grouped) slot_arrays_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tree->run_ord, d_q_offsets, n, tree->run_soff, tree->run_slen);
        if (score_mode == 1) hit_rate_guard_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d_q_offsets, n, tree->dev.st);
        if (d_tie_priority) {        // rank of every slot by (priority, slot)
            prio_init_kernel<<<blocks, 256, 0, s>>>(d_tie_priority, tree->run_ord, n, np2, tree->run_pkey, tree->run_pinv);
            sort_pairs(tree->run_pkey, tree->run_pinv, np2, s);
            prio_rank_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tree->run_pinv, n, tree->run_prank);
        }
        CK(cudaGetLastError());
    }
    if (grouped) {
        FastArgs f;
        memset(&f, 0, sizeof(f));
        st = ensure_fast_scratch(tree, n);
        if (st) return st;
        st = ensure_bulk_scratch(tree, d_fixed && n_fixed > n ? n_fixed : n);
        if (st) return st;
        if (d_fixed) {
            // which entries of the order will be processed: those before the first that is not a query or comes twice
            if (!tree->replay_info && (st = dalloc(&tree->replay_info, 1))) return st;
            const unsigned fb = (unsigned)((n_fixed + 255) / 256);
            bulk_fill_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tree->bulk_pm, n, 0x7fffffff);
            bulk_fill_kernel<<<1, 1, 0, s>>>(&tree->replay_info->n_valid, 1, n_fixed);
            replay_first_kernel<<<fb, 256, 0, s>>>(d_fixed, n_fixed, n, tree->bulk_pm);
            replay_check_kernel<<<fb, 256, 0, s>>>(d_fixed, n_fixed, n, d_q_offsets, tree->bulk_pm, tree->replay_info, tree->dev.st);
            f.fixed = d_fixed; f.n_fixed = &tree->replay_info->n_valid;
        }
        if (lru) {
            if (!tree->lru_parked && (st = dalloc(&tree->lru_parked, tree->dev.max_nodes))) return st;
            if (!tree->lru_info && (st = dalloc(&tree->lru_info, 1))) return st;
            if (n > tree->lru_hintc_cap) {
                cudaFree(tree->lru_hintc);
                tree->lru_hintc = nullptr; tree->lru_hintc_cap = 0;
                if ((st = dalloc(&tree->lru_hintc, n))) return st;
                tree->lru_hintc_cap = n;
            }
            f.hintc = tree->lru_hintc;
            if (!tree->lru_leaf_run && (st = dalloc(&tree->lru_leaf_run, tree->dev.max_nodes))) return st;
            f.leaf_run = tree->lru_leaf_run;
            if (!tree->lru_node && (st = dalloc(&tree->lru_node, tree->dev.max_nodes))) return st;
            f.node = tree->lru_node;
            f.pk = tree->fast_lk; f.pi = tree->fast_ls;      // (the key list of list mode is not used on these trees)
            f.lru = 1; f.T = tree->dev; f.parked = tree->lru_parked; f.skip = &tree->lru_info->skip;
            f.mem_cap = (int32_t)(tree->fast_mem_cap < 0x7fffffffLL ? tree->fast_mem_cap : 0x7fffffffLL);
            // all or nothing: is there room for whatever the loop can leave behind?
            CK(cudaMemsetAsync(tree->lru_info, 0, sizeof(LruInfo), s));
            if (d_fixed) lru_sum_order_kernel<<<(unsigned)((n_fixed + 255) / 256), 256, 0, s>>>(d_q_offsets, d_fixed, n_fixed, n, tree->lru_info);
            else lru_sum_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d_q_offsets, n, tree->lru_info);
            lru_check_kernel<<<1, 1, 0, s>>>(tree->dev, d_fixed ? n_fixed : n, tree->lru_info);
            lru_pack_kernel<<<(unsigned)tree->num_sms * 8, 256, 0, s>>>(tree->dev, tree->lru_node, tree->lru_parked, tree->lru_leaf_run, tree->lru_info);
        }
        f.tok = d_q_tokens; f.n = n; f.policy = params->policy; f.k = params->k; f.score_mode = score_mode;
        f.recip_k1 = params->k > 2 && params->k <= 4096 ? (unsigned)(((1ULL << 32) + (unsigned long long)(params->k - 2)) / (unsigned long long)(params->k - 1)) : 0u;
        f.c_num = params->c_num; f.c_den = params->c_den; f.start_tick = params->start_tick;
        f.order = d_order; f.uncached = d_uncached; f.ttft = d_ttft; f.completion = d_completion;
        f.dyn = tree->fast_dyn; f.stat = tree->fast_stat; f.key = tree->fast_key_arr; f.mem = tree->fast_mem;
        f.lcp = tree->fast_lcp; f.pair = tree->fast_pair; f.sorted_t = tree->run_key;
        f.pinv = d_tie_priority ? tree->run_pinv : nullptr;
        f.gh = tree->fast_gh; f.gidx = tree->fast_gidx; f.done = tree->fast_done;
        f.arrival = d_arrival; f.post = tree->fast_post;
        f.vbase = tree->dev.max_pool + 16;
        f.st = tree->dev.st;
        // Every query is matched once against the tree as it stands: by the caller's batched match if it kept the
        // records (rt_match_batch_ex), by the same kernel here otherwise.
        const MatchState* state = reinterpret_cast<const MatchState*>(d_match_state);
        unsigned long long tag = tree->ms_tag;
        if (!state) {
            if (n > tree->own_state_cap) {
                cudaFree(tree->own_state);
                tree->own_state = nullptr; tree->own_state_cap = 0;
                if ((st = dalloc(&tree->own_state, n))) return st;
                tree->own_state_cap = n;
            }
            tag = ++g_match_tag;
            st = launch_match(tree, d_q_tokens, d_q_offsets, n, nullptr, nullptr, nullptr, tree->own_state, tag, s);
            if (st) return st;
            state = tree->own_state;
        }
        fast_stat_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tree->run_ord, tree->run_key, d_q_offsets,
                                                                     d_tie_priority ? tree->run_prank : nullptr, n, f.stat);
        fast_state_kernel<<<(unsigned)((np2 + 255) / 256), 256, 0, s>>>(f, state, tag, np2);
        CK(cudaGetLastError());
        // Leaf blocks of 32 slots while at most 8,192 of them are needed, larger ones beyond (queues above 262,144).
        // Two debug settings shrink the limits so that small queues can exercise the large-queue layout:
        // fast_max_blocks (leaf blocks) and fast_smem_kb (shared memory the loop may use).
        long long max_blocks = 8192;
        size_t smem_max = 224 * 1024;
        if (g_knobs.fast_max_blocks >= 1 && g_knobs.fast_max_blocks < max_blocks) max_blocks = g_knobs.fast_max_blocks;
        if (g_knobs.fast_smem_kb >= 1 && (size_t)g_knobs.fast_smem_kb * 1024 < smem_max) smem_max = (size_t)g_knobs.fast_smem_kb * 1024;
        int lbs = 5;
        while ((((long long)n + (1LL << lbs) - 1) >> lbs) > max_blocks) ++lbs;
        f.lb_shift = lbs;
        f.nb = (int32_t)(((long long)n + (1LL << lbs) - 1) >> lbs);
        const long long nb1p = (f.nb + 31) & ~31, n2p = ((nb1p >> 5) + 31) & ~31;
        const long long nwords = ((long long)n + 31) >> 5;
        size_t smem = (size_t)(nb1p + n2p + 32) * 8 + (size_t)KLPM_FAST_SORT_CAP * 12;
        f.done_in_smem = smem + (size_t)nwords * 4 <= smem_max ? 1 : 0;
        if (f.done_in_smem) smem += (size_t)nwords * 4;
        // list mode (trees without a budget) needs two more bitmaps: in shared memory while they fit, in global memory beyond
        f.list_mode = (lru || d_fixed) ? 0 : 1;
        f.max_windows = (int32_t)g_knobs.list_max_windows;
        f.bits_in_smem = (f.list_mode && f.done_in_smem && smem + (size_t)nwords * 8 <= smem_max) ? 1 : 0;
        if (f.bits_in_smem) smem += (size_t)nwords * 8;
        f.gbits = tree->fast_done + (np2 / 32 + 32);
        f.gskip = tree->fast_done + 2 * (np2 / 32 + 32);
        const unsigned nblk = (unsigned)((n + 255) / 256), pblk = (unsigned)((np2 + 255) / 256);
        CK(cudaMemsetAsync(f.done, 0, (size_t)(3 * (np2 / 32 + 32)) * sizeof(unsigned int), s));
        // groups: queries whose match ends at the same position and continues with the same token
        GroupTable H;
        H.key = tree->grp_key; H.cnt = reinterpret_cast<int32_t*>(H.key + 2 * np2); H.off = H.cnt + 2 * np2; H.used = reinterpret_cast<unsigned int*>(H.off + 2 * np2);
        H.mask = (unsigned)(2 * np2 - 1); H.ent = tree->run_slen; H.num = tree->run_m;
        if (n <= 1024) group_small_kernel<<<1, 1024, 0, s>>>(f, H);
        else {
            CK(cudaMemsetAsync(H.key, 0, (size_t)(4 * np2 + 1) * sizeof(unsigned long long), s));
            group_count_kernel<<<nblk, 256, 0, s>>>(f, H);
            group_room_kernel<<<nblk, 256, 0, s>>>(f, H);
            fast_group_kernel<<<nblk, 256, 0, s>>>(f, H);
        }
        if (n > 1) {   // (a queue of one has no overlaps); one prompt per warp while that keeps every warp resident, up to 32 beyond
            long long per = (long long)n / ((long long)tree->num_sms * 32);
            per = per < 1 ? 1 : per > 32 ? 32 : per;
            const long long warps = ((long long)n + per - 1) / per;
            // An order of less than an eighth of the queue marks its groups first.  16 entries that share nothing out of 120,000
            // queries with shared prefixes: 475 us with the marks, 785 without; from an eighth on the order's own steps cost more.
            int32_t* wanted = nullptr;
            if (d_fixed && n_fixed < n / 8) {
                wanted = tree->run_hint;
                CK(cudaMemsetAsync(wanted, 0, (size_t)n * sizeof(int32_t), s));
                lcp_wanted_kernel<<<(unsigned)((n_fixed + 255) / 256), 256, 0, s>>>(f, wanted);
            }
            if (f.list_mode) lcp_kernel<true><<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(f, (int32_t)per, wanted);
            else lcp_kernel<false><<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(f, (int32_t)per, wanted);
        }
        if (lru) {                   // per node of the tree: the slots parked in it as the loop starts
            sort_pairs(f.pk, f.pi, np2, s);
            lru_parklist_kernel<<<nblk, 256, 0, s>>>(f);
        }
        f.lk = tree->fast_lk; f.ls = tree->fast_ls;
        // list mode: all keys as they are once everybody has arrived, largest first
        auto sort_keys = [&]() {
            fast_list_kernel<<<pblk, 256, 0, s>>>(f, np2);
            sort_pairs(tree->fast_lk, tree->fast_ls, np2, s);
        };
        CK(cudaGetLastError());
        if (lru && f.done_in_smem) {
            CK(cudaFuncSetAttribute(lru_run_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            lru_run_kernel<false><<<1, KLPM_FAST_THREADS, smem, s>>>(f);
        } else if (lru) {
            CK(cudaFuncSetAttribute(lru_run_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            lru_run_kernel<true><<<1, KLPM_FAST_THREADS, smem, s>>>(f);
        } else if (f.done_in_smem && (f.bits_in_smem || !f.list_mode)) {
            CK(cudaFuncSetAttribute(fast_run_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            fast_run_kernel<false><<<1, KLPM_FAST_THREADS, smem, s>>>(f);
            if (f.list_mode) {
                sort_keys();
                CK(cudaFuncSetAttribute(list_run_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
                list_run_kernel<false><<<1, KLPM_LIST_THREADS, smem, s>>>(f);
            }
        } else {
            CK(cudaFuncSetAttribute(fast_run_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            fast_run_kernel<true><<<1, KLPM_FAST_THREADS, smem, s>>>(f);
            if (f.list_mode) {
                sort_keys();
                CK(cudaFuncSetAttribute(list_run_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
                list_run_kernel<true><<<1, KLPM_LIST_THREADS, smem, s>>>(f);
            }
        }
        if (!lru) {                  // the decisions made in list mode are charged here (none if list mode never began), or a given order
            const long long nc = d_fixed ? n_fixed : n;
            const int32_t ipt = (int32_t)((nc + 1024LL * KLPM_CHARGE_THREADS - 1) / (1024LL * KLPM_CHARGE_THREADS));
            const int32_t per_block = KLPM_CHARGE_THREADS * ipt;
            const int32_t cblocks = (int32_t)((nc + per_block - 1) / per_block);              // at most 1,024
            charge_cost_kernel<<<cblocks, KLPM_CHARGE_THREADS, 0, s>>>(f, tree->fast_gh, tree->fast_bsum, ipt);
            charge_scan_kernel<<<1, 1024, 0, s>>>(f, tree->fast_bsum, cblocks);
            charge_apply_kernel<<<cblocks, KLPM_CHARGE_THREADS, 0, s>>>(f, tree->fast_gh, tree->fast_bsum, ipt);
        }
        CK(cudaGetLastError());
        tree->run_path = 2;
        if (lru) {
            // the nodes that are alive after the loop get their tokens, and the child table is written afresh
            const TreeDev& d = tree->dev;
            lru_unpack_kernel<<<(unsigned)tree->num_sms * 8, 256, 0, s>>>(d, tree->lru_node, tree->lru_info);
            lru_tokens_kernel<<<(unsigned)tree->num_sms * 8, 256, 0, s>>>(d, d_fixed ? d_fixed : d_order, d_q_tokens, d_q_offsets, f.vbase, tree->lru_info);
            lru_table_kernel<<<(unsigned)((d.max_nodes + 255) / 256), 256, 0, s>>>(d, f.vbase, tree->lru_info);
            CK(cudaGetLastError());
            return RT_OK;
        }
        // The processed prompts enter the tree together (the logical clock advances by n).  The loop itself needs
        // no room in the tree; if the tree cannot hold the queue the insertion says so through the status word.
        if (d_fixed) {               // only the prompts of the order, and the clock advances by as many as were processed
            replay_list_kernel<<<(unsigned)((n_fixed + 255) / 256), 256, 0, s>>>(d_fixed, n_fixed, tree->replay_info, tree->bulk_pend_a);
            return bulk_insert(tree, d_q_tokens, d_q_offsets, n_fixed, s, state, tag, true, &tree->replay_info->n_valid);
        }
        return bulk_insert(tree, d_q_tokens, d_q_offsets, n, s, state, tag);
    }
    if (d_fixed) return RT_ERR_INVALID;       // (klpm_replay takes its sequential kernel instead of this loop)
    RunBcast bc0;
    memset(&bc0, 0, sizeof(bc0));
    bc0.now = params->start_tick;
    CK(cudaMemcpyAsync(tree->run_bc, &bc0, sizeof(bc0), cudaMemcpyHostToDevice, s));
    CK(cudaMemsetAsync(tree->run_sy, 0, sizeof(RunSync), s));
    RunArgs a;
    memset(&a, 0, sizeof(a));
    a.tok = d_q_tokens; a.off = d_q_offsets; a.arrival = d_arrival; a.n = n;
    a.policy = params->policy; a.k = params->k; a.c_num = params->c_num; a.c_den = params->c_den; a.start_tick = params->start_tick;
    a.order = d_order; a.uncached = d_uncached; a.ttft = d_ttft; a.completion = d_completion;
    a.soff = tree->run_soff; a.slen = tree->run_slen; a.ntok = tree->run_ntok;
    a.prank = d_tie_priority ? tree->run_prank : nullptr; a.pinv = d_tie_priority ? tree->run_pinv : nullptr;
    a.score_mode = score_mode;
    a.ord = tree->run_ord; a.sorted_t = tree->run_key; a.m = tree->run_m; a.hint = tree->run_hint; a.pos = tree->run_pos;
    a.partial = tree->run_partial; a.bc = tree->run_bc; a.sy = tree->run_sy;
    a.wait_limit_ns = g_knobs.wait_limit_ns;
    const int threads = KLPM_RUN_THREADS;
    int per_sm = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, run_kernel, threads, 0));
    if (per_sm < 1) return RT_ERR_CUDA;
    // one sequencer CTA plus scanners; small queues are handled by the sequencer alone
    long long blocks = 1;
    if (n > threads * 8) blocks = 1 + ((long long)n + threads * KLPM_RUN_SPT - 1) / (threads * KLPM_RUN_SPT);
    if (blocks > tree->num_sms) blocks = tree->num_sms;
    void* kargs[] = {(void*)&tree->dev, (void*)&a};
    CK(cudaLaunchCooperativeKernel((void*)run_kernel, dim3((unsigned)blocks), dim3(threads), kargs, 0, s));
    tree->run_path = 1;
    return RT_OK;
}

rt_status klpm_run_last_only_batch(const int32_t* d_tokens, const int64_t* d_offsets, const int64_t* d_arrival,
                                   const int64_t* d_tie_priority, const int32_t* d_queue_offsets, int32_t n_queues,
                                   const klpm_params* params, int32_t* d_order, int32_t* d_uncached, int64_t* d_ttft,
                                   int64_t* d_completion, int32_t* d_n_skipped, void* stream) {
    if (!params_ok(params) || n_queues < 0 ||
        (n_queues > 0 && (!d_tokens || !d_offsets || !d_arrival || !d_queue_offsets || !d_order || !d_uncached || !d_ttft)))
        return RT_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)stream;
    if (d_n_skipped) CK(cudaMemsetAsync(d_n_skipped, 0, sizeof(int32_t), s));
    if (n_queues == 0) return RT_OK;
    LastOnlyArgs a;
    a.tok = d_tokens; a.off = d_offsets; a.arrival = d_arrival; a.prio = d_tie_priority; a.qoff = d_queue_offsets;
    a.n_queues = n_queues; a.policy = params->policy; a.k = params->k;
    a.c_num = params->c_num; a.c_den = params->c_den; a.start_tick = params->start_tick;
    a.order = d_order; a.uncached = d_uncached; a.ttft = d_ttft; a.completion = d_completion; a.n_skipped = d_n_skipped;
    const unsigned blocks = (unsigned)(((long long)n_queues + KLPM_LAST_ONLY_WARPS - 1) / KLPM_LAST_ONLY_WARPS);
    last_only_batch_kernel<<<blocks, 32 * KLPM_LAST_ONLY_WARPS, 0, s>>>(a);
    CK(cudaGetLastError());
    return RT_OK;
}

rt_status klpm_run_ex(rt_tree* tree, const int32_t* d_q_tokens, const int64_t* d_q_offsets, const int64_t* d_arrival,
                      int32_t n, const klpm_params* params, const int64_t* d_tie_priority, int32_t score_mode,
                      const klpm_match_state* d_match_state, int32_t* d_order, int32_t* d_uncached, int64_t* d_ttft,
                      int64_t* d_completion, void* stream) {
    if (n > 0 && !d_order) return RT_ERR_INVALID;
    return run_impl(tree, d_q_tokens, d_q_offsets, d_arrival, n, params, d_tie_priority, score_mode, d_match_state, d_order,
                    d_uncached, d_ttft, d_completion, nullptr, 0, stream);
}

int32_t klpm_run_path(const rt_tree* tree) { return tree ? tree->run_path : 0; }

rt_status rt_debug_counters(rt_tree* tree, int64_t* out16) {
    if (!tree || !out16) return RT_ERR_INVALID;
    memset(out16, 0, 16 * sizeof(int64_t));
    if (!tree->fast_post) return RT_OK;
    CK(cudaStreamSynchronize(tree->last_stream));
    FastPost h;
    CK(cudaMemcpy(&h, tree->fast_post, sizeof(h), cudaMemcpyDeviceToHost));
    for (int i = 0; i < 16; ++i) out16[i] = h.counters[i];
    return RT_OK;
}

rt_status klpm_debug_set(const char* name, int64_t value) {
    if (!name) return RT_ERR_INVALID;
    const DebugKnobs defaults = {0, 0, 0, KLPM_WAIT_LIMIT_NS, 0x7fffffffLL};
    if (!strcmp(name, "run_one_by_one")) g_knobs.run_one_by_one = value < 0 ? defaults.run_one_by_one : (value != 0);
    else if (!strcmp(name, "fast_max_blocks")) g_knobs.fast_max_blocks = value < 0 ? defaults.fast_max_blocks : value;
    else if (!strcmp(name, "fast_smem_kb")) g_knobs.fast_smem_kb = value < 0 ? defaults.fast_smem_kb : value;
    else if (!strcmp(name, "wait_limit_ns")) g_knobs.wait_limit_ns = value < 0 ? defaults.wait_limit_ns : value;
    else if (!strcmp(name, "list_max_windows")) g_knobs.list_max_windows = value < 0 || value > defaults.list_max_windows ? defaults.list_max_windows : value;
    else return RT_ERR_INVALID;
    return RT_OK;
}

rt_status klpm_run(rt_tree* tree, const int32_t* d_q_tokens, const int64_t* d_q_offsets, const int64_t* d_arrival,
                   int32_t n, const klpm_params* params, int32_t* d_order, int32_t* d_uncached, int64_t* d_ttft,
                   int64_t* d_completion, void* stream) {
    return klpm_run_ex(tree, d_q_tokens, d_q_offsets, d_arrival, n, params, nullptr, 0, nullptr, d_order, d_uncached, d_ttft,
                       d_completion, stream);
}

}  // extern "C"

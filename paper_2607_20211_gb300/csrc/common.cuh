// Internal declarations shared by the kernels of the D-RSF library.
//
// Device state layout (all in HBM, one copy per handle):
//   parent[n], rep[n]           int32   the forest and each vertex's tree root
//   row[n+1]                    16 B    slack-CSR row heads: start, slots in
//                                       use, free slots, capacity
//   col[slots]                  int32   neighbours; -1 = empty or deleted
//   fpos[slots]                 int32   each row's stack of free slots
//   index[H]                    16 B    open-addressing edge index: key ->
//                                       global col positions of the edge in
//                                       the rows of min(u,v) and max(u,v),
//                                       or (POS_OVF, overflow slot)
//   ovf                         16 B    edges with a full row (key, slot taken
//                                       in the other row), and a stack of the
//                                       entries that are free again
//   per-batch work arrays (epoch-stamped, never cleared per batch)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <climits>

#include "../../include/drsf.h"

typedef unsigned long long u64;

#define EMPTY_KEY 0xFFFFFFFFFFFFFFFFull
#define TOMB_KEY 0xFFFFFFFFFFFFFFFEull
#define POS_OVF 0xFFFFFFFFu
#define NIL (-1)

// latched device error bits (ctl->err)
#define ERR_BATCH_ID 1   // out-of-range id in the current batch: batch skipped
#define ERR_TIMEOUT 2    // a bounded grid barrier gave up
#define ERR_CAPACITY 4   // an internal buffer would overflow (never expected)
#define ERR_ROUNDS 8     // an iteration exceeded its round bound (cyclic parent)
#define ERR_MOVED 16     // a recorded batch was replayed after the storage moved: batch skipped
#define ERR_FULL 32      // a recorded insert was replayed without room for it: batch skipped

// grid-barrier wait limit in nanoseconds (globaltimer)
#define BARRIER_TIMEOUT_NS 2000000000ull
#define MAX_ROUNDS 40

// Device control block: latched errors, batch epoch, grid barrier state,
// per-batch counts.  Statistic fields mirror drsf_batch_stats.
struct Ctl {
    int err;
    unsigned skip;          // epoch + 1 of the last rejected batch (ERR_BATCH_ID, ERR_MOVED, ERR_FULL)
    unsigned epoch;         // batch counter; epoch stamps compare against it
    unsigned base;          // the batches before this one (k_begin's blocks all read it; the claim
                            // kernels move it on)
    int op;
    u64 bar[8];             // grid-barrier counters: jump, hook, orient, mark, bfs / scan, Euler marks, detach, cross
                            // (reset at each batch's start and before each static BFS)
    int flag[3];            // per-round "another round needed" flags
    u64 cnt[3];             // per-round list sizes (hook-and-compress)
    u64 dv[3], dp[3];       // top-down delete, per level (ring of 3): vertices appended, and
                            // rows << 32 | entries appended
    u64 dovf;               // top-down delete: tree edges listed from the overflow list
    unsigned depth_hint;    // top-down delete, kept across batches: levels the last search took, or
                            // above the level limit after one gave up (counts down once per skip)
    int det_skip;           // the batch skipped the top-down search (read by the next k_begin)
    u64 nb;                 // normalised batch edges (new / deleted keys)
    u64 ncut;               // cut vertices
    u64 naff;               // affected list
    u64 ndet;               // detached list
    u64 ncand;              // candidates
    u64 ner;                // replacement edges
    u64 npre;               // delete: those of them that the scan chose (k_replace's blocks branch on this
                            // and on ncand: nothing in that launch writes it, where block 0 counts ner on)
    u64 npc;                // distinct pieces touched by E_r
    u64 nact;               // active vertices (path reversal)
    u64 ncore;              // core arcs of the super-forest Euler tour
    u64 ovf_count;          // overflow list length: entries ever taken since the last rebuild
    u64 ovf_free;           // entries of it that are free again
    long long storage;      // generation of the storage and batch buffers (drsf_ctx::gen)
    long long edges;        // live undirected edges of G
    long long htomb;        // index tombstones
    long long ctomb;        // dead CSR entries (deleted ones, and slots lost to overflow edges)
    long long scanned;      // adjacency entries scanned
    long long self_loops;
    long long dropped;
    long long hook_rounds;
    long long rank_rounds;
    long long mark_rounds;
    long long jump_rounds;
    long long jump_visits;
    long long reversed;
    long long batch_len;
    const int *batch;       // the current batch (device), set by k_begin
    int td;                 // delete: the detached vertices were found top-down (else: pointer jumping)
    int need_root;          // delete: a cut tree's root piece is re-rooted (read after a top-down delete)
    int njobs;              // delete: parts of long rows to read
    u64 nagain[2];          // large delete: rows read again, after the first and a second round
    int nlong;              // some path was too long to be reversed by its walk
    long long det_levels;   // top-down levels of the batch (0: not taken)
    long long det_entries;  // adjacency entries the top-down search read
};

// The current batch was rejected: no kernel after k_begin touches anything.
__device__ __forceinline__ bool batch_skipped(const Ctl *ctl) {
    return *(const volatile unsigned *)&ctl->skip == ctl->epoch + 1;
}

// What a batch may assume of the handle's storage.  A batch that the caller
// recorded into a graph of its own carries pointers into the storage as it was
// then, and its room was checked then; k_begin and k_bbegin check again.
struct StorageLimits {
    long long gen;          // ctl->storage as the launches' pointers were taken
    long long index_max;    // index slots in use (live and deleted) after an insert
    u64 ovf_cap;            // overflow entries in use after an insert
};
// (loaded ahead of the check, beside the first loads of the batch: behind them
// an insert and a delete of 100 edges took 130 us instead of 126, R-MAT scale 22)
struct StorageCounts {
    long long gen, used;
    u64 ovf;
};
__device__ __forceinline__ StorageCounts storage_counts(const Ctl *ctl) {
    const volatile Ctl *c = ctl;
    return StorageCounts{c->storage, c->edges + c->htomb, c->ovf_count - c->ovf_free};
}
// One thread of the batch's first kernel: rejects the batch when the launches
// that follow have no business with the storage.
__device__ __forceinline__ void storage_guard(Ctl *ctl, const StorageCounts &c, const StorageLimits &l, int op,
                                              long long len, unsigned epoch) {
    int e = 0;
    if (c.gen != l.gen) e = ERR_MOVED;
    else if (op == DRSF_INSERT && (c.used + len > l.index_max || c.ovf + (u64)len > l.ovf_cap)) e = ERR_FULL;
    if (!e) return;
    atomicOr(&ctl->err, e);
    ctl->skip = epoch + 1;
}

// The edge index.  An entry is one 16-byte record: with keys and positions in
// arrays of their own a deleted edge touched three sectors of a table far
// larger than L2 instead of one, an inserted one too.
struct __align__(16) Entry {
    u64 key;
    uint2 pos;      // x: position of the edge in the row of min(u,v), or POS_OVF
                    // y: position in the row of max(u,v), or overflow slot
};
struct Index {
    Entry *e;
    u64 mask;
};

// The slack CSR.  A row's head is one 16-byte record, so that whoever visits
// a row (append, removal, scan) touches one sector for it.  Its free slots
// form a stack of nfree entries in the row's part of fpos: entry k is the
// free slot's position in the row, or -1 for the position it holds when the
// row is new (cap - 1 - k: the stack of a new row gives its slack in order).
struct __align__(16) Row {
    unsigned start;   // first slot (positions are below 2^32, checked at build)
    int used;         // slots from the start that may hold an entry: what a scan reads
    int nfree;        // free slots
    int cap;
};
struct Csr {
    Row *row;
    int *col;
    int *fpos;
};

__host__ __device__ __forceinline__ u64 ekey(uint32_t u, uint32_t v) {
    return u < v ? ((u64)u << 32) | v : ((u64)v << 32) | u;
}
__host__ __device__ __forceinline__ uint32_t klo(u64 k) { return (uint32_t)(k >> 32); }
__host__ __device__ __forceinline__ uint32_t khi(u64 k) { return (uint32_t)(k & 0xFFFFFFFFu); }

// 64-bit finaliser (MurmurHash3 fmix64) for the edge index.
__device__ __forceinline__ u64 hslot(u64 k, u64 mask) {
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return k & mask;
}

// Edge index probes (open addressing, linear probing).
// Insert-if-absent.  Returns the slot when this call claimed it, -1-slot
// when the key was already present, LLONG_MIN when the table is full.
// The claimed slot is the first deleted or empty one of the key's chain, and
// it is claimed only after the whole chain was seen without the key
// (*reused tells that it was a deleted one).  While keys are being inserted
// slots only go from deleted or empty to a key, so two threads with one key
// meet: a thread whose slot was taken meanwhile looks at the chain again
// from that slot on, and finds the key the other one wrote there or further
// along.  Without the reuse an edge that comes back leaves one more deleted
// slot in its own chain every time: after 1,500 removals of each edge of a
// 100-edge batch the claim alone took 1,115 us (R-MAT scale 22).  Measured
// over a window of returning edges (insert + delete step, R-MAT scale 22):
// 100-edge batches 751 -> 218 us, 10K-edge batches 781 -> 333 us.
__device__ __forceinline__ long long index_claim(Index ix, u64 key, bool *reused) {
    u64 s = hslot(key, ix.mask);
    long long free_slot = -1;   // first deleted slot of the chain
    for (u64 p = 0; p <= 2 * ix.mask; ++p) {
        const u64 cur = __ldcg(&ix.e[s].key);
        if (cur == key) return -1 - (long long)s;
        if (cur == TOMB_KEY && free_slot < 0) free_slot = (long long)s;
        if (cur == EMPTY_KEY) {
            const bool dead = free_slot >= 0;
            const u64 t = dead ? (u64)free_slot : s;
            const u64 old = atomicCAS(&ix.e[t].key, dead ? TOMB_KEY : EMPTY_KEY, key);
            if (old == (dead ? TOMB_KEY : EMPTY_KEY)) {
                *reused = dead;
                return (long long)t;
            }
            if (old == key) return -1 - (long long)t;
            s = t;   // another key took the slot
            free_slot = -1;
        }
        s = (s + 1) & ix.mask;
    }
    return LLONG_MIN;
}

// Pull a whole array into L2, one prefetch per 128-byte line, strided over
// the calling threads (thread tid of nthreads): for arrays that the next
// kernels gather from at random, which would otherwise pay one DRAM latency
// per dependent access.
__device__ __forceinline__ void l2_prefetch(const void *p, long long bytes, long long tid, long long nthreads) {
    const char *c = (const char *)p;
    for (long long off = tid * 128; off < bytes; off += nthreads * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(c + off));
}

// Hook-forest slots of the candidates' endpoints (read by k_replace): the
// kernel that writes a candidate sets up each of its endpoints once per
// batch (whoever stamps it first): its own root in comp, both per-round
// minimum slots empty.
struct HookSlots {
    unsigned *stamp;
    int *comp;
    u64 *best0, *best1;
};
__device__ __forceinline__ void hook_slot_init(const HookSlots &hs, int a, unsigned ep) {
    // one lane per endpoint among the calling lanes (the giant tree's root
    // is an endpoint of most candidates)
    const unsigned grp = __match_any_sync(__activemask(), a);
    if ((int)(threadIdx.x & 31) != __ffs(grp) - 1) return;
    if (__ldcg(&hs.stamp[a]) != ep && atomicExch(&hs.stamp[a], ep) != ep) {
        hs.comp[a] = a;
        hs.best0[a] = EMPTY_KEY;
        hs.best1[a] = EMPTY_KEY;
    }
}

// Lookup; -1 when absent, else the slot and the entry's positions.  Deleted
// entries (TOMB_KEY) are probed past.
__device__ __forceinline__ long long index_find(Index ix, u64 key, uint2 *pos) {
    u64 s = hslot(key, ix.mask);
    for (u64 p = 0; p <= ix.mask; ++p) {
        const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(&ix.e[s]));
        const u64 cur = ((u64)q.y << 32) | q.x;
        if (cur == key) {
            *pos = make_uint2(q.z, q.w);
            return (long long)s;
        }
        if (cur == EMPTY_KEY) return -1;
        s = (s + 1) & ix.mask;
    }
    return -1;
}

// Warp-aggregated append: one atomicAdd per warp; returns the slot of this
// lane (or -1 when pred is false).
__device__ __forceinline__ long long agg_append(u64 *ctr, bool pred) {
    unsigned active = __activemask();
    unsigned m = __ballot_sync(active, pred);
    if (!pred) return -1;
    int lane = threadIdx.x & 31;
    int leader = __ffs(m) - 1;
    u64 base = 0;
    if (lane == leader) base = atomicAdd(ctr, (u64)__popc(m));
    base = __shfl_sync(m, base, leader);
    return (long long)(base + __popc(m & ((1u << lane) - 1u)));
}

__device__ __forceinline__ Row row_head(const Csr &g, int r) {
    const int4 q = __ldcg(reinterpret_cast<const int4 *>(&g.row[r]));
    return Row{(unsigned)q.x, q.y, q.z, q.w};
}

// One free slot of row r (head h) per calling lane, from the top of the
// row's stack; -1 when the row is full.  Slots are only taken while a batch
// is inserted and only given back while one is deleted, so the counter alone
// decides who gets which entry: no retries, and a lane that drew below zero
// puts its draw back.  Lanes of a warp with the same row share one atomic (a
// hub row receives many of a batch's edges).  *grown counts the slots that
// the row's scanned length grew by.  Reusing deleted slots keeps rows at
// their length when edges leave and come back; with append-only rows such a
// window filled the slack and then the overflow list and rebuilt the whole
// storage every 40 steps of 100K-edge batches (R-MAT scale 22).
__device__ __forceinline__ int row_take(const Csr &g, int r, const Row &h, long long *grown) {
    const unsigned grp = __match_any_sync(__activemask(), r);
    const int lane = threadIdx.x & 31, ld = __ffs(grp) - 1, cnt = __popc(grp);
    int base = 0;
    if (lane == ld) {
        base = atomicSub(&g.row[r].nfree, cnt);
        if (base < cnt) atomicAdd(&g.row[r].nfree, base > 0 ? cnt - base : cnt);
    }
    base = __shfl_sync(grp, base, ld);
    const int k = base - 1 - __popc(grp & ((1u << lane) - 1u));
    if (k < 0) return -1;
    const int f = g.fpos[(size_t)h.start + k];
    const int slot = f < 0 ? h.cap - 1 - k : f;
    if (slot >= h.used) {
        const int old = atomicMax(&g.row[r].used, slot + 1);
        if (slot + 1 > old) *grown += slot + 1 - old;
    }
    return slot;
}

// Lanes of the calling ones (act) that give to row r: its first lane draws for
// up to two rows that several lanes share (a hub's, in a batch of its edges),
// the others for themselves.
struct Share {
    int leader, rank, count;
};
__device__ __forceinline__ Share row_share(unsigned act, int r) {
    const int lane = threadIdx.x & 31;
    Share s{lane, 0, 1};
    unsigned m = act;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int l0 = __ffs(m) - 1;
        const unsigned grp = __ballot_sync(act, r == __shfl_sync(act, r, l0));
        if (grp >> lane & 1u) s = Share{l0, __popc(grp & ((1u << lane) - 1u)), __popc(grp)};
        m &= ~grp;
        if (!m) break;
    }
    return s;
}
// Give slot pos (a position in col) of row r back.
__device__ __forceinline__ void row_give(const Csr &g, int r, unsigned start, unsigned pos) {
    const int k = atomicAdd(&g.row[r].nfree, 1);
    g.col[pos] = -1;
    g.fpos[(size_t)start + k] = (int)(pos - start);
}
// The same for both rows of an edge and every calling lane, one atomic per
// shared row and warp: with one per edge the removal of 500K edges of one vertex
// took 227 us instead of 92, of 2M 1,102 instead of 484.
__device__ __forceinline__ void row_give2(const Csr &g, int a, unsigned sa, unsigned pa, int b, unsigned sb, unsigned pb) {
    const unsigned act = __activemask();
    const int lane = threadIdx.x & 31;
    const Share x = row_share(act, a), y = row_share(act, b);
    int ka = 0, kb = 0;
    if (x.leader == lane) ka = atomicAdd(&g.row[a].nfree, x.count);
    if (y.leader == lane) kb = atomicAdd(&g.row[b].nfree, y.count);
    g.col[pa] = g.col[pb] = -1;
    ka = __shfl_sync(act, ka, x.leader) + x.rank;
    kb = __shfl_sync(act, kb, y.leader) + y.rank;
    g.fpos[(size_t)sa + ka] = (int)(pa - sa);
    g.fpos[(size_t)sb + kb] = (int)(pb - sb);
}

// The edges held outside their rows.  An edge of which one row is full took a
// slot of the other: it stays empty, and is given back with the entry.
struct Ovf {
    u64 *e;           // keys; TOMB_KEY where free
    unsigned *pos;    // that slot's position in col, or POS_OVF
    unsigned *free;   // stack of ctl->ovf_free free entries
    u64 cap;
};

// Entry for an edge outside its rows: from the top of the stack, or the list's
// end (a draw that found the stack empty is put back, as with the rows'
// slots).  As with the rows' slots, entries are only taken while a batch is inserted
// and only given back while one is deleted.
__device__ __forceinline__ long long ovf_take(Ctl *ctl, const Ovf &o) {
    const long long have = (long long)atomicAdd(&ctl->ovf_free, ~0ull);   // (minus one)
    if (have > 0) return o.free[have - 1];
    atomicAdd(&ctl->ovf_free, 1ull);
    return (long long)atomicAdd(&ctl->ovf_count, 1ull);
}
// Edge {a, b} leaves entry i: the entry is free again, and the slot that the
// edge held in one of its rows.
__device__ __forceinline__ void ovf_give(Ctl *ctl, const Ovf &o, const Csr &g, unsigned i, int a, int b) {
    o.e[i] = TOMB_KEY;
    const unsigned p = o.pos[i];
    if (p != POS_OVF) {
        const Row ha = row_head(g, a);
        const bool in_a = p - ha.start < (unsigned)ha.cap;
        row_give(g, in_a ? a : b, in_a ? ha.start : g.row[b].start, p);
    }
    o.free[agg_append(&ctl->ovf_free, true)] = i;
}

// Pair table: piece pair (min, max) -> minimum edge key between the two
// pieces.  Probing is bounded; a pair that finds no slot returns false and
// the caller keeps the edge as a plain candidate instead.
#define PAIR_PROBES 64
// Slot of a piece pair key (claimed if absent), or -1 when the probes found
// no slot.
__device__ __forceinline__ long long pair_slot(u64 *pk, u64 mask, u64 pair) {
    u64 s = hslot(pair, mask);
    for (int p = 0; p < PAIR_PROBES; ++p) {
        u64 cur = __ldcg(&pk[s]);
        if (cur == pair) return (long long)s;
        if (cur == EMPTY_KEY) {
            u64 old = atomicCAS(&pk[s], EMPTY_KEY, pair);
            if (old == EMPTY_KEY || old == pair) return (long long)s;
        }
        s = (s + 1) & mask;
    }
    return -1;
}
__device__ __forceinline__ bool pair_min(u64 *pk, u64 *mk, u64 mask, int a, int b, u64 key) {
    const u64 pair = a < b ? ((u64)(unsigned)a << 32) | (unsigned)b : ((u64)(unsigned)b << 32) | (unsigned)a;
    const long long s = pair_slot(pk, mask, pair);
    if (s < 0) return false;
    // (most edges of a pair that has many are no new minimum)
    if (key < __ldcg(&mk[s])) atomicMin(&mk[s], key);
    return true;
}

// Block-wide sum of per-thread counts added to a counter: one atomic per
// block.  Every thread of the block must call it.
__device__ __forceinline__ void block_add(long long *ctr, long long v) {
    __shared__ unsigned long long s_sum;
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_sum, (unsigned long long)v);
    __syncthreads();
    if (threadIdx.x == 0 && s_sum) atomicAdd((unsigned long long *)ctr, s_sum);
    __syncthreads();
}

// Block-aggregated append: one atomicAdd per block.  Every thread of the
// block must call it (the loop around it must be block-uniform); the slots
// of a block are contiguous and ordered by thread index.
__device__ __forceinline__ long long block_append(u64 *ctr, bool pred) {
    __shared__ unsigned s_w[32];
    __shared__ u64 s_base;
    unsigned m = __ballot_sync(0xffffffffu, pred);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) s_w[w] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned tot = 0;
        int nw = (blockDim.x + 31) >> 5;
        for (int k = 0; k < nw; ++k) {
            unsigned c = s_w[k];
            s_w[k] = tot;
            tot += c;
        }
        s_base = tot ? atomicAdd(ctr, (u64)tot) : 0;
    }
    __syncthreads();
    long long r = pred ? (long long)(s_base + s_w[w] + __popc(m & ((1u << lane) - 1u))) : -1;
    __syncthreads();
    return r;
}

// Block-wide exclusive scan (any blockDim multiple of 32, <= 1024);
// *total receives the block sum.  All threads must call it.
__device__ __forceinline__ long long block_excl_scan_ll(long long v, long long *total) {
    __shared__ long long s_ws[32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_ws[w] = x;
    __syncthreads();
    if (w == 0) {
        long long t = lane < nw ? s_ws[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) s_ws[lane] = t;
    }
    __syncthreads();
    long long pre = (w > 0 ? s_ws[w - 1] : 0) + x - v;
    *total = s_ws[nw - 1];
    __syncthreads();
    return pre;
}

// ovf_take for every thread of a block with `on` (all call): the stack and the
// list's end are asked once.
__device__ __forceinline__ long long ovf_take_block(Ctl *ctl, const Ovf &o, bool on) {
    __shared__ long long s_have, s_end;
    long long n;
    const long long k = block_excl_scan_ll(on, &n);
    if (threadIdx.x == 0) {
        const long long have = (long long)atomicAdd(&ctl->ovf_free, (u64)-n);
        const long long got = have < 0 ? 0 : (have < n ? have : n);
        if (got < n) atomicAdd(&ctl->ovf_free, (u64)(n - got));
        s_have = have;
        s_end = got < n ? (long long)atomicAdd(&ctl->ovf_count, (u64)(n - got)) - got : 0;
    }
    __syncthreads();
    const long long i = !on ? -1 : (k < s_have ? (long long)o.free[s_have - 1 - k] : s_end + k);
    __syncthreads();
    return i;
}

// Block-aggregated reservation of `cnt` consecutive slots per thread (one
// atomicAdd per block); returns this thread's first slot.  Every thread of
// the block must call it.
__device__ __forceinline__ long long block_reserve(u64 *ctr, int cnt) {
    __shared__ u64 s_rb;
    long long tot;
    long long pre = block_excl_scan_ll(cnt, &tot);
    if (threadIdx.x == 0) s_rb = tot ? atomicAdd(ctr, (u64)tot) : 0;
    __syncthreads();
    long long r = (long long)s_rb + pre;
    __syncthreads();
    return r;
}

// Block-aggregated reservation for four separate slabs: thread t has
// flags f[0..3] (item k of thread t lies in input slab k); the output keeps
// slab order and, within a slab, thread order, so a compacted list keeps the
// order of its input.  One block scan of the four counts packed in 16-bit
// fields (a block has at most 1024 threads) and one atomicAdd per block.
// Returns the output slot of item k in slot[k] (-1 when its flag is 0).
__device__ __forceinline__ void block_reserve4(u64 *ctr, const bool f[4], long long slot[4]) {
    __shared__ u64 s_rb4;
    long long packed = (long long)f[0] | ((long long)f[1] << 16) | ((long long)f[2] << 32) | ((long long)f[3] << 48);
    long long tot;
    long long pre = block_excl_scan_ll(packed, &tot);
    long long t[4], p[4];
    for (int k = 0; k < 4; ++k) {
        t[k] = (tot >> (16 * k)) & 0xFFFF;
        p[k] = (pre >> (16 * k)) & 0xFFFF;
    }
    long long all = t[0] + t[1] + t[2] + t[3];
    if (threadIdx.x == 0) s_rb4 = all ? atomicAdd(ctr, (u64)all) : 0;
    __syncthreads();
    long long base = (long long)s_rb4, off = 0;
    for (int k = 0; k < 4; ++k) {
        slot[k] = f[k] ? base + off + p[k] : -1;
        off += t[k];
    }
    __syncthreads();
}

// Block-aggregated reservation of list rows together with their entry
// ranges, from one packed counter: rows in the high 32 bits, entries in the
// low 32 bits (the entries of all rows stay below 2^32, so the low half
// never carries into the high half).  Row k of each thread (f[k] set, len[k]
// entries) gets its list position pos[k] and entry offset off[k]; positions
// and offsets follow slab order, then thread order, so the offsets are the
// exclusive prefix sum of the lengths in list order.  One atomicAdd per
// block; every thread of the block must call it.
template <int K>
__device__ __forceinline__ void block_reserve_rows(u64 *ctr, const bool f[K], const int len[K], long long pos[K],
                                                   long long off[K]) {
    __shared__ u64 s_rr;
    long long pre[K], tot[K];
#pragma unroll
    for (int k = 0; k < K; ++k)
        pre[k] = block_excl_scan_ll(f[k] ? (1ll << 32) | (long long)(unsigned)len[k] : 0ll, &tot[k]);
    long long all = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) all += tot[k];
    if (threadIdx.x == 0) s_rr = all ? atomicAdd(ctr, (u64)all) : 0;
    __syncthreads();
    u64 acc = s_rr;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const u64 b = acc + (u64)pre[k];
        pos[k] = f[k] ? (long long)(b >> 32) : -1;
        off[k] = (long long)(b & 0xFFFFFFFFull);
        acc += (u64)tot[k];
    }
    __syncthreads();
}

// 64-bit minimum over a group of lanes (mask from __match_any_sync).
__device__ __forceinline__ u64 group_min_u64(unsigned grp, u64 k) {
    unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    unsigned hmin = __reduce_min_sync(grp, hi);
    unsigned lmin = __reduce_min_sync(grp, hi == hmin ? lo : 0xFFFFFFFFu);
    return ((u64)hmin << 32) | lmin;
}

__device__ __forceinline__ u64 globaltimer_ns() {
    u64 t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ u64 ld_acquire_u64(const u64 *p) {
    u64 v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Grid-wide barrier for cooperative launches (all blocks co-resident).
// Ticket barrier on a monotonic counter owned by one kernel (always launched
// with the same block count, so the counter is a multiple of gridDim.x
// between barriers; or by the first nb blocks only, always the same nb): each
// block takes a ticket t and waits until the counter reaches the end of t's
// group.  The wait is bounded: after
// BARRIER_TIMEOUT_NS it latches ERR_TIMEOUT and returns false, and a block
// that sees another block's timeout returns false too, so the kernel unwinds
// instead of hanging.
__device__ __forceinline__ bool grid_barrier(Ctl *ctl, u64 *bar, u64 nb = gridDim.x) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        u64 t = atomicAdd(bar, 1ull);
        u64 target = (t / nb + 1) * nb;
        int ok = 1;
        if (ld_acquire_u64(bar) < target) {
            u64 t0 = globaltimer_ns();
            unsigned it = 0;
            while (ld_acquire_u64(bar) < target) {
                if ((++it & 255u) == 0) {
                    if (*(volatile int *)&ctl->err & ERR_TIMEOUT) { ok = 0; break; }
                    if (globaltimer_ns() - t0 > BARRIER_TIMEOUT_NS) {
                        atomicOr(&ctl->err, ERR_TIMEOUT);
                        ok = 0;
                        break;
                    }
                }
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Root search with path halving on a hook forest that is not being hooked
// concurrently (halving writes keep every pointer on the path to the same
// root).  The walk is bounded: a cycle (impossible for valid input) latches
// ERR_ROUNDS instead of spinning.
__device__ __forceinline__ int find_root(int *comp, int x, Ctl *ctl) {
    for (int it = 0; it < (1 << 24); ++it) {
        int p = __ldcg(&comp[x]);
        if (p == x) return x;
        int gp = __ldcg(&comp[p]);
        if (gp == p) return p;
        comp[x] = gp;
        x = gp;
    }
    atomicOr(&ctl->err, ERR_ROUNDS);
    return x;
}

// Root of x in the hook forest without writes (for short chains read by
// many threads at once: no stores to shared entries).  Bounded; a cycle
// latches ERR_ROUNDS.
__device__ __forceinline__ int find_root_ro(const int *comp, int x, Ctl *ctl) {
    for (int it = 0; it < (1 << 24); ++it) {
        int p = __ldcg(&comp[x]);
        if (p == x) return x;
        x = p;
    }
    atomicOr(&ctl->err, ERR_ROUNDS);
    return x;
}

// Loads of data that other blocks wrote earlier in the same cooperative
// launch go to L2 (the SM's L1 may hold a stale line).
#define LD(x) __ldcg(&(x))

static inline unsigned grid_for(long long n, int block, unsigned cap) {
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > (long long)cap) g = cap;
    return (unsigned)g;
}

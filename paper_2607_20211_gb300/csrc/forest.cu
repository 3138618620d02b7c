// Forest kernels of the D-RSF batch update (Algorithm 1):
//   - representatives by pointer jumping on the cut forest F^;
//   - replacement edges by hooking and compressing over the trees of F^
//     (Section III-B, Algorithm 2, phase 1), with minimum-key hooking so
//     that the chosen edges are the unique minimum spanning forest of the
//     tree multigraph (Boruvka);
//   - orientation of the replacement edges by an Euler tour of the
//     tree-of-trees (Algorithm 2, phase 2; Euler tour technique, Section I
//     preliminaries) rooted at the tree with the smallest root id;
//   - path reversal of every (x, rep[x]) path at once by pointer doubling
//     over the re-rooted trees, then attachment parent[x] <- y
//     (Algorithm 1; ReversePaths, Section II-C), and the representative
//     refresh.
// Iterative phases run as one cooperative launch each with a bounded grid
// barrier between rounds; no host round trip per round.
#include <climits>

#include "kernels.h"

// cores of up to this many arcs are list-ranked in one block's shared memory:
// for batches of up to 64K edges, and for larger ones, whose grid phases want
// the rest of the SM's memory as L1 (with 216 instead of 128 KB of shared
// memory the hooking and orientation of a 100K-edge batch took 98 + 66 instead
// of 77 + 54 us on R-MAT scale 22, the 256-graph union's 241 + 440 instead of
// 182 + 337)
#define RANK_ARCS 12288
#define RANK_ARCS_LARGE 8192
#define ORIENT_THREADS 1024
// hooking: the live candidates at the start of a round (after round 0) up to
// which block 0 finishes alone, and the candidates that it takes on from the
// start (what k_scan's first round left: usually none or a few; 3,300 took 90
// us by one block against 60 by the grid)
#define HOOK_TAIL 8192
#define HOOK_FEW 1024
// a core of at most this many edges is oriented by one block (measured on
// R-MAT-22: faster than the grid phases for small batches' cores of tens of
// edges, slower for the 100K batches' cores of about 900 edges)
#define ORIENT_SMALL_EDGES 256
// independent items per thread and iteration in the pointer-doubling rounds
#ifndef JU
#define JU 4
#endif
// the same for the final pass of the jump (more state per item)
#define JF 2
// consecutive items per thread in the list-building vertex passes: IPT over
// a list, IPN over all n vertices (more loads in flight per thread: those
// passes are one dependent gather behind a streaming load)
#define IPT 4
#define IPN 16
// k_aff_collect keeps more per item (old root, list position)
#define IPA 8
// the refresh after a large delete, most of whose vertices may change (the
// 4096 x 4096 grid: three quarters): their new representatives are loaded
// together
#define IPD 8
// top-down delete: the longest batch searched by one block per SM
#define SEARCH_FEW 4096
// top-down delete: after a search that gave up at its level limit, the
// deletes that skip it before it is tried again
#define DETACH_BACKOFF 8
// longest path reversed by one walking thread (longer ones: doubling marks)
#define WALK_MAX 64

// a detached piece is left out of the cross-edge scan instead of its tree's
// root piece only if it has this many more vertices (the swap costs a full
// pass over the affected list)
#define HEAVY_SWAP_MIN 4096
// shared-memory piece-count table of the final jump pass
#define WT_BITS 6
#define WT_SLOTS (1 << WT_BITS)
#define WT_PROBES 8

#define GS_LOOP(i, n) \
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)(n); \
         i += (long long)gridDim.x * blockDim.x)

#include "scan.cuh"

__device__ __forceinline__ long long gtid() { return (long long)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ long long gstride() { return (long long)gridDim.x * blockDim.x; }

// The graph that owns position i of an offsets array (the last one that starts
// at or before it).
__device__ __forceinline__ int owner_of(const long long *off, int G, long long i) {
    int lo = 0, hi = G - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Start of a batch: every id is checked (an out-of-range id, or with `groups`
// an edge that leaves its graph's vertices, rejects the whole batch), and one
// thread resets the per-batch counters, sets the epoch and records the batch
// (the kernels after this one read the batch and its length from the control
// block, so their launches do not depend on them).  The rejection carries the
// batch's epoch, so it needs no reset that the checks would race with, and no
// launch of its own.
__global__ void k_begin(Ctl *ctl, BeginArgs a) {
    const unsigned epoch = ctl->base + 1;
    StorageCounts have{};
    if (gtid() == 0) have = storage_counts(ctl);
    GS_LOOP(i, a.len) {
        const int u = a.batch[2 * i], v = a.batch[2 * i + 1];
        bool bad = u < 0 || u >= a.n || v < 0 || v >= a.n;
        if (a.groups) {
            const int g = owner_of(a.boff, a.groups, i);
            const long long lo = a.voff[g], hi = a.voff[g + 1];
            bad |= u < lo || u >= hi || v < lo || v >= hi;
        }
        if (bad) {
            atomicOr(&ctl->err, ERR_BATCH_ID);
            ctl->skip = epoch + 1;
        }
    }
    if (gtid() != 0) return;
    const int op = a.op;
    const long long len = a.len;
    storage_guard(ctl, have, a.lim, op, len, epoch);   // (batch and offsets are the caller's or kept for the recording)
    ctl->batch = a.batch;
    ctl->epoch = epoch;
    ctl->op = op;
    ctl->nb = ctl->ncut = ctl->naff = ctl->ndet = ctl->ncand = ctl->ner = ctl->npc = ctl->nact = 0;
    ctl->scanned = ctl->self_loops = ctl->dropped = 0;
    ctl->hook_rounds = ctl->rank_rounds = ctl->mark_rounds = ctl->jump_rounds = ctl->reversed = 0;
    ctl->jump_visits = 0;
    ctl->nagain[0] = ctl->nagain[1] = 0;
    ctl->td = ctl->need_root = ctl->nlong = ctl->njobs = 0;
    ctl->npre = 0;
    if (ctl->det_skip) {   // the last batch skipped the top-down search
        if (ctl->depth_hint > 0) ctl->depth_hint -= 1;
        ctl->det_skip = 0;
    }
    ctl->det_levels = ctl->det_entries = 0;
    ctl->batch_len = len;
    for (int i = 0; i < 3; ++i) {
        ctl->flag[i] = 0;
        ctl->cnt[i] = 0;
        ctl->dv[i] = ctl->dp[i] = 0;
    }
    ctl->dovf = 0;
    // each barrier counter serves one cooperative launch per batch; its
    // targets are multiples of that launch's grid size, so it restarts at 0
    // (launches of different grid sizes, or a wait that timed out, leave it
    // at any value)
    for (int i = 0; i < 8; ++i) ctl->bar[i] = 0;
}

// Delete: list the vertices of every tree that lost a tree edge (its old
// root was stamped by the cut), with their old root.
// Each thread takes IPN vertices per iteration, k-major (item k of thread t
// is vertex b0 + k * blockDim + t, so every load and store of a warp covers
// 32 consecutive vertices), with all IPN loads and gathers in flight before
// any is used.  A warp's listed vertices take consecutive slots (one block
// reservation of the warps' totals), in vertex order within the warp.
// It runs for the selectable root searches (k_jump) only, and only when the
// top-down search of the detached vertices did not find them.
__global__ void __launch_bounds__(BLK) k_aff_collect(int n, const int *rep, const unsigned *aff_ep, int *A, int *rold,
                                                     unsigned *w, u64 *heavy, Ctl *ctl) {
    static_assert(IPA <= 32, "item masks are 32 bits");
    if (batch_skipped(ctl)) return;
    if (*(volatile int *)&ctl->td) return;
    unsigned ep = ctl->epoch;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long step = (long long)gridDim.x * blockDim.x * IPA;
    for (long long b0 = (long long)blockIdx.x * blockDim.x * IPA; b0 < n; b0 += step) {
        const long long v0 = b0 + threadIdx.x;
        int r[IPA];
#pragma unroll
        for (int k = 0; k < IPA; ++k) {
            const long long v = v0 + (long long)k * blockDim.x;
            r[k] = v < n ? rep[v] : 0;
        }
        unsigned in = 0;
#pragma unroll
        for (int k = 0; k < IPA; ++k) {
            const long long v = v0 + (long long)k * blockDim.x;
            if (v < n && aff_ep[r[k]] == ep) in |= 1u << k;
        }
        // (the warp's ballots are recomputed below rather than kept)
        const int tot = __reduce_add_sync(0xffffffffu, __popc(in));
        long long p = block_reserve(&ctl->naff, lane == 0 ? tot : 0);
        p = __shfl_sync(0xffffffffu, p, 0);
#pragma unroll
        for (int k = 0; k < IPA; ++k) {
            const unsigned bk = __ballot_sync(0xffffffffu, (in >> k) & 1u);
            if ((in >> k) & 1u) {
                const int v = (int)(v0 + (long long)k * blockDim.x);
                A[p + __popc(bk & lt)] = v;
                rold[v] = r[k];
                if (r[k] == v) {        // the old root: piece-weight and heaviest-piece slots
                    w[v] = 0;
                    heavy[v] = 0;
                }
            }
            p += __popc(bk);
        }
    }
}

// Root of v in the forest J by pointer jumping with path halving, in place:
// every J[x] only ever moves to an ancestor of x, so concurrent walks over
// shared paths stay correct and shorten each other's paths (no round
// barrier is needed).  The walk is bounded; a cycle latches ERR_ROUNDS.
__device__ __forceinline__ int find_halving(int *J, int v, Ctl *ctl) {
    int x = v;
    for (int it = 0; it < (1 << 22); ++it) {
        int p = __ldcg(&J[x]);
        int gp = __ldcg(&J[p]);
        if (p == gp) return p;
        J[x] = gp;
        x = gp;
    }
    atomicOr(&ctl->err, ERR_ROUNDS);
    return x;
}

// Adds cnt to the weight of piece p through the block's shared table
// (open addressing, WT_PROBES probes), or to w[p] when no slot is free.
__device__ __forceinline__ void piece_count(int *s_wk, unsigned *s_wc, unsigned *w, int p, unsigned cnt) {
    unsigned h = ((unsigned)p * 0x9E3779B1u) >> (32 - WT_BITS);
    for (int pr = 0; pr < WT_PROBES; ++pr) {
        int key = *(volatile int *)&s_wk[h];
        if (key == -1) key = atomicCAS(&s_wk[h], -1, p);
        if (key == -1 || key == p) {
            atomicAdd(&s_wc[h], cnt);
            return;
        }
        h = (h + 1) & (WT_SLOTS - 1);
    }
    atomicAdd(&w[p], cnt);
}

// tile[T] = row for the tiles of 32 entries whose first entry lies in the
// row of entries [st, st + d), d > 0 (rows are never empty), for the rows of
// the lanes with `on` (called by the whole warp).  A lane writes the tiles of
// a short row itself; a long row (a hub's, up to tens of thousands of tiles)
// is written by the whole warp, so no lane writes more than a few tiles of
// it in sequence.
#define FILL_OWN 4
__device__ __forceinline__ void warp_fill_tiles(int *tile, bool on, long long st, long long d, int row) {
    const int lane = threadIdx.x & 31;
    const long long t0 = (st + 31) >> 5, t1 = on ? ((st + d - 1) >> 5) + 1 : t0;   // tiles [t0, t1)
    const bool big = t1 - t0 > FILL_OWN;
    if (on && !big)
        for (long long T = t0; T < t1; ++T) tile[T] = row;
    unsigned bm = __ballot_sync(0xffffffffu, big);
    while (bm) {
        const int l = __ffs(bm) - 1;
        bm &= bm - 1;
        const long long a = __shfl_sync(0xffffffffu, t0, l), b = __shfl_sync(0xffffffffu, t1, l);
        const int r = __shfl_sync(0xffffffffu, row, l);
        for (long long T = a + lane; T < b; T += 32) tile[T] = r;
    }
}

// Append the non-empty rows (`f`, `len` > 0) of a warp's lanes to the row
// list of the scan, with their entry ranges and the tile map: positions are
// pb (rows << 32 | entries) plus offsets from one atomic per warp on the
// packed counter pc.  All 32 lanes call.
__device__ __forceinline__ void warp_list_rows(u64 *pc, u64 pb, RowList rl, bool f, int w, unsigned st, int len, int p,
                                               int ro) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned fm = __ballot_sync(0xffffffffu, f);
    if (!fm) return;
    // exclusive warp scan of the row lengths
    int x = f ? len : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    const int tot = __shfl_sync(0xffffffffu, x, 31);
    const int ex = x - (f ? len : 0);
    const int fl = __ffs(fm) - 1;
    u64 base = 0;
    if (lane == fl) base = atomicAdd(pc, ((u64)__popc(fm) << 32) | (u64)(unsigned)tot);
    base = __shfl_sync(0xffffffffu, base, fl) + pb;
    const long long q = (long long)(base >> 32) + __popc(fm & lt);
    const long long eo = (long long)(base & 0xFFFFFFFFull) + ex;
    if (f) {
        rl.D[q] = w;
        rl.roff[q] = (unsigned)eo;
        rl.base[q] = st;
        rl.meta[q] = make_int2(p, ro);
    }
    warp_fill_tiles(rl.tile, f, eo, len, (int)q);
}

// Append one warp's detached vertices (lanes with `on`) to the vertex list
// and their non-empty rows (starting at `st`, `len` > 0) to the row list of the scan: positions
// are the level's bases (vb vertices; pb rows << 32 | entries) plus offsets
// taken from the level's own counters (vc, and pc packed like pb), one
// atomic per warp on each.  All 32 lanes call.
__device__ __forceinline__ void warp_detach_append(u64 *vc, u64 *pc, long long vb, u64 pb, RowList rl, int *A,
                                                   bool on, int w, unsigned st, int len, int p, int ro) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (!m) return;
    const int ld = __ffs(m) - 1;
    u64 a0 = 0;
    if (lane == ld) a0 = atomicAdd(vc, (u64)__popc(m));
    a0 = __shfl_sync(0xffffffffu, a0, ld);
    if (on) A[vb + (long long)a0 + __popc(m & ((1u << lane) - 1u))] = w;
    warp_list_rows(pc, pb, rl, on && len > 0, w, st, len, p, ro);
}

// Delete, top-down alternative to the pointer jumping of Algorithm 1 (same
// representatives): the detached vertices are the cut vertices and every
// descendant of one in the cut forest, and a detached vertex's piece is the
// nearest cut vertex above it.  A level-synchronous search goes down from
// the cut vertices over tree children (neighbours w of v with parent[w] ==
// v, found in v's row or, for edges held outside the rows, in the overflow
// list) and touches only the detached vertices' rows, where pointer jumping
// touches every vertex of every cut tree.  Each level's rows are appended to
// the row list of the cross-edge scan as they are found (rows and entry
// ranges from one packed counter, 32-entry tiles), so level k reads exactly
// the rows appended in level k-1 with the tile-window scan of scan_rows, and
// the scan afterwards reuses the list (the piece left out of every tree is
// its root piece).  Every level appends through counters of its own (a ring
// of three: level k appends to slot k+1, reads the final count of slot k
// after the barrier and clears slot k+2), so all blocks see the same level
// sizes although some append while others still read.  New representatives
// go to J1 and are committed only when the search ends within its budget
// (vertices, entries, levels); otherwise nothing is published and the
// pointer-jumping path runs.
// Returns 1 when the pieces were found, 0 when they were not, -1 when a grid
// barrier gave up.
__device__ int detach_top_down(Ctl *ctl, const DetachArgs &a, const RowList &rl, unsigned nb) {
    const long long S = (long long)nb * blockDim.x;   // the threads that search
    const int *const cuts = a.cuts, *const par = a.par, *const rold = a.rold;
    int *const rep = a.rep, *const A = a.A, *const J1 = a.J1, *const oc = a.oc, *const op = a.op;
    unsigned *const det_ep = a.det_ep, *const det_claim = a.det_claim;
    const Csr &g = a.g;
    const u64 *const ovf = a.ovf;
    const int max_levels = a.max_levels;
    // Deep trees below the cuts make the search a long chain of levels
    // (one grid barrier each) where pointer doubling needs a logarithmic
    // number of steps: after a search that gave up at the level limit the
    // next DETACH_BACKOFF deletes go straight to pointer jumping, then the
    // search is tried again.  The hint is not written in this launch before
    // every block has read it (the next batch's k_begin counts it down), so
    // all blocks take the same branch.
    if (*(volatile unsigned *)&ctl->depth_hint > (unsigned)max_levels) {
        if (gtid() == 0) ctl->det_skip = 1;
        return 0;
    }
    const unsigned ep = ctl->epoch;
    const long long nc = (long long)ctl->ncut;
    u64 *bar = &ctl->bar[6];
    const int lane = threadIdx.x & 31;
    // level 0: the cut vertices (pieces of their own), slot 0
    for (long long b0 = gtid() & ~31ll; b0 < nc; b0 += S) {
        const long long i = b0 + lane;
        const bool on = i < nc;
        int c = 0, len = 0, ro = 0;
        unsigned st = 0;
        if (on) {
            c = cuts[i];
            ro = rold[c];
            J1[c] = c;
            __threadfence();   // J1 before the stamp that publishes it
            det_ep[c] = ep;
            const Row h = row_head(g, c);
            st = h.start;
            len = h.used;
        }
        warp_detach_append(&ctl->dv[0], &ctl->dp[0], 0, 0, rl, A, on, c, st, len, c, ro);
    }
    // the tree edges held outside the rows (overflow list), as (child,
    // parent): listed once, read by every level (few: edges land there
    // only when a row is full)
    {
        const long long no = (long long)min((u64)ctl->ovf_count, a.ovf_cap);
        for (long long b0 = gtid() & ~31ll; b0 < no; b0 += S) {
            const long long i = b0 + lane;
            int cw = -1, pv = -1;
            if (i < no) {
                const u64 k = ovf[i];
                if (k != TOMB_KEY) {
                    const int a = (int)klo(k), b = (int)khi(k);
                    if (LD(par[a]) == b) cw = a, pv = b;
                    else if (LD(par[b]) == a) cw = b, pv = a;
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, cw >= 0);
            if (!m) continue;
            const int ld = __ffs(m) - 1;
            u64 q0 = 0;
            if (lane == ld) q0 = atomicAdd(&ctl->dovf, (u64)__popc(m));
            q0 = __shfl_sync(0xffffffffu, q0, ld);
            if (cw >= 0) {
                const u64 q = q0 + __popc(m & ((1u << lane) - 1u));
                oc[q] = cw;
                op[q] = pv;
            }
        }
    }
    long long vb = 0;   // vertices listed before the current level's
    u64 pb = 0;         // rows << 32 | entries listed before it
    int lvl = 0;
    bool ok = true;
    for (;; ++lvl) {
        if (!grid_barrier(ctl, bar, nb)) return -1;
        // the level found in the last round (slot lvl % 3) is final
        const int sl = lvl % 3, sn = (lvl + 1) % 3;
        const long long dv = (long long)*(volatile u64 *)&ctl->dv[sl];
        const u64 dp = *(volatile u64 *)&ctl->dp[sl];
        if (gtid() == 0) ctl->dv[(lvl + 2) % 3] = ctl->dp[(lvl + 2) % 3] = 0;   // read last one level ago
        const unsigned e_lo = (unsigned)pb, r_lo = (unsigned)(pb >> 32);
        const long long vn = vb + dv;
        const u64 pn = pb + dp;
        const unsigned e_hi = (unsigned)pn, r_hi = (unsigned)(pn >> 32);
        if (dv == 0) break;   // the last level found nothing
        if (lvl >= max_levels || vn > a.budget_v || (long long)e_hi > a.budget_e) {
            ok = false;
            break;
        }
        (void)r_lo;
        // tiles covering the entries of the rows found in the last level,
        // a contiguous range of tiles per warp
        const unsigned T0 = e_lo >> 5, T1 = (e_hi + 31) >> 5;
        const unsigned NT = T1 - T0;
        const unsigned nw = (unsigned)(S >> 5), wid = (unsigned)(gtid() >> 5);
        const unsigned per = (NT + nw - 1) / nw;
        for (unsigned it = 0; it < per; ++it) {
            const unsigned T = T0 + wid * per + it;
            bool child = false;
            int w = -1, p = 0, ro = 0;
            if (T < T1) {   // warp-uniform
                const unsigned t0 = T << 5;
                // (rows of earlier levels, written by other blocks: read through L2)
                const int r0 = LD(rl.tile[T]);
                const unsigned wr = (unsigned)r0 + lane;
                const bool wok = wr < r_hi;
                const unsigned wo = wok ? LD(rl.roff[wr]) : 0xFFFFFFFFu;
                const int wv = wok ? LD(rl.D[wr]) : 0;
                const unsigned wb = wok ? LD(rl.base[wr]) : 0;
                const int2 wm = wok ? __ldcg(&rl.meta[wr]) : make_int2(0, 0);
                const unsigned pos = wo - t0;
                const unsigned bit = (lane > 0 && pos < 32) ? (1u << pos) : 0u;
                const unsigned starts = __reduce_or_sync(0xffffffffu, bit);
                const int c = __popc(starts & (lane == 31 ? 0xffffffffu : ((2u << lane) - 1u)));
                const unsigned rstart = __shfl_sync(0xffffffffu, wo, c);
                const int v = __shfl_sync(0xffffffffu, wv, c);
                const unsigned rb = __shfl_sync(0xffffffffu, wb, c);
                p = __shfl_sync(0xffffffffu, wm.x, c);
                ro = __shfl_sync(0xffffffffu, wm.y, c);
                const unsigned e = t0 + lane;
                if (e >= e_lo && e < e_hi) {
                    w = __ldcs(&g.col[(size_t)(rb + (e - rstart))]);
                    child = w >= 0 && LD(par[w]) == v;
                }
            }
            int len = 0;
            unsigned st = 0;
            if (child) {
                const Row h = row_head(g, w);
                J1[w] = p;
                __threadfence();
                det_ep[w] = ep;
                st = h.start;
                len = h.used;
            }
            warp_detach_append(&ctl->dv[sn], &ctl->dp[sn], vn, pn, rl, A, child, w, st, len, p, ro);
        }
        // children joined by a tree edge outside the rows: a vertex whose
        // parent is detached (published: its J1 before its stamp)
        const long long nt = (long long)*(volatile u64 *)&ctl->dovf;
        for (long long b0 = gtid() & ~31ll; b0 < nt; b0 += S) {
            const long long i = b0 + lane;
            bool child = false;
            int w = -1, p = 0, ro = 0, len = 0;
            unsigned st = 0;
            if (i < nt) {
                const int cw = LD(oc[i]), pv = LD(op[i]);
                const bool pd = LD(det_ep[pv]) == ep;
                __threadfence();
                if (pd && LD(det_claim[cw]) != ep && atomicExch(&det_claim[cw], ep) != ep) {
                    child = true;
                    w = cw;
                    p = LD(J1[pv]);
                    ro = LD(rep[w]);   // rep still holds the old roots (read again, new, by the scan)
                }
            }
            if (child) {
                const Row h = row_head(g, w);
                J1[w] = p;
                __threadfence();
                det_ep[w] = ep;
                st = h.start;
                len = h.used;
            }
            warp_detach_append(&ctl->dv[sn], &ctl->dp[sn], vn, pn, rl, A, child, w, st, len, p, ro);
        }
        vb = vn;
        pb = pn;
    }
    // over budget: nothing was published (naff, ndet and rep untouched);
    // the pointer-jumping path takes over from the cut
    if (!ok) {
        if (gtid() == 0) {
            ctl->det_levels = -lvl;
            if (lvl >= max_levels) ctl->depth_hint = (unsigned)max_levels + DETACH_BACKOFF;
        }
        return 0;
    }
    // commit the representatives of the detached vertices
    for (long long i = gtid(); i < vb; i += S) {
        const int v = A[i];
        rep[v] = LD(J1[v]);
    }
    if (gtid() == 0) {
        ctl->naff = (u64)vb;
        ctl->ndet = pb >> 32;
        ctl->det_entries = (long long)(pb & 0xFFFFFFFFull);
        rl.roff[pb >> 32] = (unsigned)pb;
        ctl->det_levels = lvl;
        ctl->depth_hint = (unsigned)lvl;
        ctl->td = 1;
    }
    return 1;
}

// heavy[r] = the piece left out of the scan of the cut tree with old root r
// (weight << 32 | piece; the root piece stays it unless a detached piece
// outweighs it by HEAVY_SWAP_MIN vertices), over the cut list: a cut tree's
// pieces are its root piece and one piece per cut vertex.
__device__ __forceinline__ void heaviest_pieces(const int *cuts, long long nc, const int *rold, const unsigned *w,
                                                u64 *heavy) {
    for (long long i = gtid(); i < nc; i += gstride()) {
        int c = cuts[i];
        int r = rold[c];
        u64 kc = ((u64)LD(w[c]) << 32) | (unsigned)c;
        unsigned act = __activemask();
        unsigned grp = __match_any_sync(act, r);
        unsigned hi = (unsigned)(kc >> 32), lo = (unsigned)kc;
        unsigned hmax = __reduce_max_sync(grp, hi);
        unsigned lmax = __reduce_max_sync(grp, hi == hmax ? lo : 0u);
        if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) {
            atomicMax(&heavy[r], ((u64)hmax << 32) | lmax);
            atomicMax(&heavy[r], ((u64)(LD(w[r]) + HEAVY_SWAP_MIN) << 32) | (unsigned)r);
        }
    }
}

// Delete: the pieces of the cut trees (Algorithm 1, representatives by pointer
// jumping) and the detached vertices, in one launch over all vertices:
//   1. each vertex of a cut tree (its old root was stamped by the cut) follows
//      its parents for up to RELABEL_HOPS steps in the forest, which nobody
//      writes here, and leaves the ancestor it reached, or its root
//      complemented, in J;
//   2. after a grid barrier each warp's vertices still open (deep trees) go on
//      by asynchronous pointer jumping in place, RELABEL_STEPS pointers at
//      once: a pointer only ever moves to an ancestor, whatever mix of old and
//      new values a step reads, so every step moves an open vertex up at least
//      one level (one pointer a step, J[v] <- J[J[v]], is as many loads in all
//      but more passes over the lists and stores that others' loads miss on:
//      the 4096 x 4096 grid's 16M vertices 550 us, three 456, five 462, seven
//      475);
//   3. the vertices whose root changed (the detached ones; on R-MAT a few
//      percent) get their new representative and are listed;
//   4. every cut tree gets the piece that the scan for cross edges leaves out:
//      every cross edge joins two pieces of one old tree, so scanning the rows
//      of all pieces but one finds each of them.  That is the root piece,
//      unless a detached piece has HEAVY_SWAP_MIN more vertices (a cut near
//      the root that detaches most of a tree): then the heaviest piece.  The
//      root piece's size is its tree's (counted in 1) less the detached
//      pieces'.
// Listing the affected vertices, doubling from distance 1 and a pass over that
// whole list took 38 + 99 us of a 100K-edge delete batch on R-MAT scale 22
// (2.5M affected vertices, 100K detached); this 65.  Bound by the gathers of
// the hops, from L2, and by its barriers.
#define RELABEL_HOPS 4
#define RELABEL_STEPS 3
#define RI 4   // vertices per lane and iteration

// Piece counts of a block: a small open-addressing table in shared memory (one
// global atomic per piece and block at the end; a large piece spans many
// blocks), or straight to global memory when the table has no slot.
struct PieceTable {
    int k[WT_SLOTS];
    unsigned c[WT_SLOTS];
};
__device__ __forceinline__ void pt_init(PieceTable &t) {
    for (int i = threadIdx.x; i < WT_SLOTS; i += blockDim.x) {
        t.k[i] = -1;
        t.c[i] = 0;
    }
    __syncthreads();
}
__device__ __forceinline__ void pt_flush(PieceTable &t, unsigned *w) {
    __syncthreads();
    for (int i = threadIdx.x; i < WT_SLOTS; i += blockDim.x)
        if (t.k[i] != -1) atomicAdd(&w[t.k[i]], t.c[i]);
}
// the lanes with `on` count 1 for their piece p (all 32 lanes call)
__device__ __forceinline__ void pt_count(PieceTable &t, unsigned *w, int p, bool on) {
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (!on) return;
    const unsigned grp = __match_any_sync(m, p);
    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) piece_count(t.k, t.c, w, p, (unsigned)__popc(grp));
}

__device__ bool relabel(Ctl *ctl, const RelabelArgs &a) {
    const unsigned ep = ctl->epoch;
    const long long nc = (long long)ctl->ncut;
    if (nc == 0) return true;   // no tree was cut
    u64 *bar = &ctl->bar[0];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    __shared__ PieceTable pt;
    pt_init(pt);
    // chunks of consecutive vertices, dealt out to the blocks in turn (graphs
    // or regions with deep trees spread over all of them); a warp's lists
    // have room for its part of every chunk of its block
    constexpr int CH = BLK * RI;
    const long long nch = ((long long)a.n + CH - 1) / CH, per = (nch + gridDim.x - 1) / gridDim.x;
    const long long own = ((long long)blockIdx.x * CH + (threadIdx.x & ~31) * RI) * per;
    int *const X = a.X + own, *const Y = a.Y + own, *const L = a.L + own;
    int nopen = 0, nd = 0;
    long long naff = 0, vis = 0;
    int tr = -1;           // the tree that this warp counts, and its count so far
    unsigned tc = 0;
    for (long long c = blockIdx.x; c < nch; c += gridDim.x) {
        const int v0 = (int)(c * CH) + (int)(threadIdx.x & ~31) * RI + lane;
        int r[RI], x[RI];
        unsigned on = 0, done = 0;   // vertices of cut trees; those at their root
#pragma unroll
        for (int k = 0; k < RI; ++k) {
            const bool ok = (long long)v0 + k * 32 < a.n;
            r[k] = ok ? a.rep[v0 + k * 32] : -1;
            x[k] = ok ? a.par[v0 + k * 32] : 0;
        }
#pragma unroll
        for (int k = 0; k < RI; ++k) {
            if (r[k] >= 0 && a.aff_ep[r[k]] == ep) on |= 1u << k;
            if (x[k] == v0 + k * 32) done |= 1u << k;
        }
        if (!__any_sync(0xffffffffu, on)) continue;
#pragma unroll
        for (int h = 0; h < RELABEL_HOPS; ++h) {
            int nx[RI];
#pragma unroll
            for (int k = 0; k < RI; ++k) nx[k] = (on & ~done) >> k & 1u ? a.par[x[k]] : -1;
#pragma unroll
            for (int k = 0; k < RI; ++k) {
                if (nx[k] < 0) continue;
                if (nx[k] == x[k]) done |= 1u << k;
                x[k] = nx[k];
            }
        }
#pragma unroll
        for (int k = 0; k < RI; ++k) {
            const bool in = on >> k & 1u, at = done >> k & 1u;
            if (in) a.J[v0 + k * 32] = at ? ~x[k] : x[k];
            const unsigned mi = __ballot_sync(0xffffffffu, in);
            if (!mi) continue;
            const unsigned mo = __ballot_sync(0xffffffffu, in && !at), md = __ballot_sync(0xffffffffu, in && at && x[k] != r[k]);
            if (in && !at) X[nopen + __popc(mo & lt)] = v0 + k * 32;
            if (in && at && x[k] != r[k]) L[nd + __popc(md & lt)] = v0 + k * 32;
            nopen += __popc(mo);
            nd += __popc(md);
            // tree sizes: one tree for the whole warp is the common case
            const int r0 = __shfl_sync(0xffffffffu, r[k], __ffs(mi) - 1);
            if (__all_sync(0xffffffffu, !in || r[k] == r0)) {
                if (r0 != tr) {
                    if (lane == 0 && tc) piece_count(pt.k, pt.c, a.w, tr, tc);
                    tr = r0;
                    tc = 0;
                }
                tc += __popc(mi);
            } else {
                pt_count(pt, a.w, r[k], in);
            }
        }
        naff += __popc(on);
    }
    if (lane == 0 && tc) piece_count(pt.k, pt.c, a.w, tr, tc);
    block_add((long long *)&ctl->naff, naff);
    if (!grid_barrier(ctl, bar)) return false;
    // (each warp reads lists that it wrote itself)
    int *in = X, *out = Y;
    int it = 0;
    __syncwarp();
    for (; nopen > 0; ++it) {
        if (it >= MAX_ROUNDS * 64) {
            if (lane == 0) atomicOr(&ctl->err, ERR_ROUNDS);
            break;
        }
        vis += nopen;
        int left = 0;
        for (int b0 = 0; b0 < nopen; b0 += 32 * RI) {
            int v[RI], w[RI];
#pragma unroll
            for (int k = 0; k < RI; ++k) v[k] = b0 + k * 32 + lane < nopen ? in[b0 + k * 32 + lane] : -1;
#pragma unroll
            for (int k = 0; k < RI; ++k) w[k] = v[k] >= 0 ? LD(a.J[v[k]]) : -1;
#pragma unroll
            for (int h = 0; h < RELABEL_STEPS; ++h) {
#pragma unroll
                for (int k = 0; k < RI; ++k) w[k] = w[k] >= 0 ? LD(a.J[w[k]]) : w[k];
            }
#pragma unroll
            for (int k = 0; k < RI; ++k) {
                const bool ok = v[k] >= 0, op = ok && w[k] >= 0;
                if (ok) a.J[v[k]] = w[k];
                const bool det = ok && !op && ~w[k] != a.rep[v[k]];
                const unsigned mo = __ballot_sync(0xffffffffu, op), md = __ballot_sync(0xffffffffu, det);
                if (op) out[left + __popc(mo & lt)] = v[k];
                if (det) L[nd + __popc(md & lt)] = v[k];
                left += __popc(mo);
                nd += __popc(md);
            }
        }
        __syncwarp();
        nopen = left;
        int *t = in; in = out; out = t;
    }
    if (lane == 0 && vis) {
        atomicAdd((u64 *)&ctl->jump_visits, (u64)vis);
        atomicMax((unsigned long long *)&ctl->jump_rounds, (unsigned long long)it);
    }
    // detached vertices: the list of all of them (one reservation per block),
    // representatives and piece weights (those of the cut vertices were zeroed
    // at the cut)
    {
        const long long q = block_reserve(&ctl->ndet, lane == 0 ? nd : 0);
        int *const D = a.D + __shfl_sync(0xffffffffu, q, 0);
        for (int i0 = 0; i0 < nd; i0 += 32 * JF) {
            int v[JF], p[JF];
#pragma unroll
            for (int k = 0; k < JF; ++k) v[k] = i0 + k * 32 + lane < nd ? L[i0 + k * 32 + lane] : -1;
#pragma unroll
            for (int k = 0; k < JF; ++k) p[k] = v[k] >= 0 ? ~LD(a.J[v[k]]) : 0;
#pragma unroll
            for (int k = 0; k < JF; ++k) {
                if (v[k] >= 0) {
                    D[i0 + k * 32 + lane] = v[k];
                    a.rep[v[k]] = p[k];
                }
                pt_count(pt, a.w, p[k], v[k] >= 0);
            }
        }
    }
    pt_flush(pt, a.w);
    if (!grid_barrier(ctl, bar)) return false;
    // per cut tree: the detached pieces' vertices and the heaviest of them
    for (long long i = gtid(); i < nc; i += gstride()) {
        const int c = a.cuts[i], r = a.rold[c];
        const unsigned wc = LD(a.w[c]);
        const unsigned grp = __match_any_sync(__activemask(), r);
        const unsigned sum = __reduce_add_sync(grp, wc);
        if (lane == __ffs(grp) - 1) atomicAdd(&a.wsum[r], sum);
        if (wc >= HEAVY_SWAP_MIN) atomicMax(&a.heavy[r], ((u64)wc << 32) | (unsigned)c);
    }
    if (!grid_barrier(ctl, bar)) return false;
    bool swap = false;
    for (long long i = gtid(); i < nc; i += gstride()) {
        const int r = a.rold[a.cuts[i]];
        const u64 hv = LD(a.heavy[r]);
        const bool sw = (hv >> 32) >= (u64)(LD(a.w[r]) - LD(a.wsum[r])) + HEAVY_SWAP_MIN;
        const int l = sw ? (int)(unsigned)hv : r;
        a.left[a.cuts[i]] = l;
        if (LD(a.left[r]) != l) a.left[r] = l;   // (one store per tree, not one per cut)
        swap |= sw;
    }
    if (__syncthreads_or(swap) && threadIdx.x == 0) atomicOr(&ctl->flag[0], 1);
    return true;
}

// Large deletes: pieces and scan as launches of their own (the first fits five
// blocks on an SM, the second four).
__global__ void __launch_bounds__(BLK, 5) k_relabel(Ctl *ctl, RelabelArgs a) {
    if (batch_skipped(ctl)) return;
    relabel(ctl, a);
}
template <bool SG>
__global__ void __launch_bounds__(BLK, 4) k_scan(Ctl *ctl, RowList rl, LightArgs a) {
    if (batch_skipped(ctl)) return;
    if (!a.listed) scan_light<SG>(ctl, a);
    else if (!ctl->td) scan_listed<SG>(ctl, rl, a);   // (else k_cross has scanned them)
}
// Small deletes: the top-down search and the scan of the rows it listed, or,
// where it gives up, what large deletes do, in one launch (as four, the ones
// that found nothing to do took 8 us of every batch).  With a selectable root
// search (a.listed) that search and its scan are launches of their own, which
// find nothing to do when the top-down one found the pieces.
template <bool SG>
__global__ void __launch_bounds__(BLK, 4)
    k_cross(Ctl *ctl, DetachArgs d, RelabelArgs r, RowList rl, LightArgs a) {
    if (batch_skipped(ctl)) return;
    // a batch of up to SEARCH_FEW edges is searched by one block per SM (a
    // level of its search is a barrier and little work), the others wait
    const unsigned nb = ctl->batch_len <= SEARCH_FEW && gridDim.x > d.nsm ? d.nsm : gridDim.x;
    int found = 0;
    if (blockIdx.x < nb) {
        found = detach_top_down(ctl, d, rl, nb);
        if (found < 0) return;
    }
    if (nb < gridDim.x) {
        if (!grid_barrier(ctl, &ctl->bar[7])) return;
        found = *(volatile int *)&ctl->td;
    }
    if (!found && (a.listed || !relabel(ctl, r))) return;
    if ((!found || nb == gridDim.x) && !grid_barrier(ctl, &ctl->bar[7])) return;
    if (found) scan_listed<SG>(ctl, rl, a);
    else scan_light<SG>(ctl, a);
}

// Representatives (Algorithm 1, parallel pointer jumping) of the listed
// vertices: rep[v] = root of v in F^ (J starts as a copy of parent).
// Delete mode (1) then chooses the rows to scan for cross edges: every cross
// edge joins two pieces of one old tree, so scanning all pieces but one per
// tree finds each of them.  The piece left out is the root piece, unless a
// detached piece has HEAVY_SWAP_MIN more vertices (a cut near the root that
// detaches most of a tree): then the heaviest piece.  The listed rows get an
// exclusive prefix sum of their lengths in roff (roff[ndet] = total; rows
// and entry ranges are reserved together from one packed counter), their
// CSR start, their (piece, piece left out) and the row of every 32-entry
// tile for the load-balanced scan.
// (The selectable synchronous and halving searches, and the representatives at
// creation; 6 blocks of BLK threads per SM: the rounds are latency-bound.)
template <int sync_rounds>
__global__ void __launch_bounds__(BLK, 6)
    k_jump(const int *A, int use_list, long long cnt_static, Ctl *ctl, const int *par, int *J, int *J1, int *rep,
           RowList rl, int mode, const int *rold, unsigned *w, u64 *heavy, Csr g, int *X, int *Y, const int *cuts) {
    int *const D = rl.D;
    unsigned *const roff = rl.roff;
    if (batch_skipped(ctl)) return;
    if (mode == 1 && *(volatile int *)&ctl->td) return;   // the top-down search found the pieces
    long long cnt = use_list ? (long long)ctl->naff : cnt_static;
    if constexpr (sync_rounds != 0) {
        // synchronous doubling J <- J o J (ping-pong).  A pointer that has
        // reached a root is stored complemented (negative): a converged
        // vertex skips the gather, and the loop ends in the first round in
        // which every listed vertex is converged (no verification round).
        // Round r reads the list of vertices still open (the full list in
        // round 0) and appends the ones still open after it to the other
        // work list (X, Y alternate); a vertex that converges writes its
        // complemented root into both buffers, so later reads of it from
        // either buffer see the root.  Round 0 reads the forest itself
        // (par); its converged vertices still write both buffers.
        int *Jc = J, *Jn = J1;
        int r = 0;
        if (gtid() == 0) {
            ctl->cnt[0] = (u64)cnt;
            ctl->cnt[1] = 0;
        }
        if (!grid_barrier(ctl, &ctl->bar[0])) return;
        for (;; ++r) {
            if (r >= MAX_ROUNDS) {
                if (gtid() == 0) atomicOr(&ctl->err, ERR_ROUNDS);
                return;
            }
            const long long c = (long long)*(volatile u64 *)&ctl->cnt[r % 3];
            if (c == 0) break;
            if (gtid() == 0) {
                ctl->cnt[(r + 2) % 3] = 0;
                ctl->jump_visits += c;
            }
            const int *in = r == 0 ? (use_list ? A : nullptr) : ((r & 1) ? X : Y);
            int *out = (r & 1) ? Y : X;
            // JU independent vertices per thread and iteration: their loads
            // are issued together (more loads in flight per thread)
            const long long S = gstride();
            for (long long base = (long long)blockIdx.x * blockDim.x; base < c; base += S * JU) {
                int v[JU], w0[JU], w2[JU];
                bool ok[JU], open[JU];
#pragma unroll
                for (int k = 0; k < JU; ++k) {
                    long long i = base + k * S + threadIdx.x;
                    ok[k] = i < c;
                    v[k] = ok[k] ? (in ? in[i] : (int)i) : 0;
                }
                const int *Jr = r == 0 ? par : Jc;
#pragma unroll
                for (int k = 0; k < JU; ++k) w0[k] = ok[k] ? LD(Jr[v[k]]) : -1;
#pragma unroll
                for (int k = 0; k < JU; ++k) w2[k] = (ok[k] && w0[k] >= 0) ? LD(Jr[w0[k]]) : 0;
#pragma unroll
                for (int k = 0; k < JU; ++k) {
                    open[k] = false;
                    if (!ok[k]) continue;
                    int nv;
                    if (w0[k] < 0) nv = w0[k];
                    else if (w2[k] < 0) nv = w2[k];
                    else if (w2[k] == w0[k]) nv = ~w0[k];
                    else {
                        nv = w2[k];
                        open[k] = true;
                    }
                    Jn[v[k]] = nv;
                    if (!open[k]) Jc[v[k]] = nv;
                }
                long long q[JU];
                block_reserve4(&ctl->cnt[(r + 1) % 3], open, q);
#pragma unroll
                for (int k = 0; k < JU; ++k)
                    if (open[k]) out[q[k]] = v[k];
            }
            if (!grid_barrier(ctl, &ctl->bar[0])) return;
            int *t = Jc; Jc = Jn; Jn = t;
        }
        if (gtid() == 0) ctl->jump_rounds = r;
        if (mode == 0) {
            for (long long i = gtid(); i < cnt; i += gstride()) {
                int v = use_list ? A[i] : (int)i;
                rep[v] = ~LD(Jc[v]);
            }
            return;
        }
        // final pass: representatives, piece weights (vertex counts; the
        // weight slots of piece roots were zeroed at the cut) and a
        // provisional list of rows to scan: every vertex outside its tree's
        // root piece (only those read their row length).  JU vertices per
        // thread and iteration.  Piece counts go to a small open-addressing
        // table in shared memory (one global atomic per piece and block at
        // the end; a large piece spans many blocks), or straight to global
        // memory when the table has no slot.
        __shared__ int s_wk[WT_SLOTS];
        __shared__ unsigned s_wc[WT_SLOTS];
        for (int t = threadIdx.x; t < WT_SLOTS; t += blockDim.x) {
            s_wk[t] = -1;
            s_wc[t] = 0;
        }
        __syncthreads();
        const long long S = gstride();
        for (long long base = (long long)blockIdx.x * blockDim.x; base < cnt; base += S * JF) {
            int v[JF], p[JF], ro[JF], len[JF];
            unsigned st[JF];
            bool ok[JF], scan[JF];
#pragma unroll
            for (int k = 0; k < JF; ++k) {
                long long i = base + k * S + threadIdx.x;
                ok[k] = i < cnt;
                v[k] = ok[k] ? A[i] : 0;
            }
#pragma unroll
            for (int k = 0; k < JF; ++k) {
                p[k] = ok[k] ? ~LD(Jc[v[k]]) : 0;
                ro[k] = ok[k] ? rold[v[k]] : 0;
            }
#pragma unroll
            for (int k = 0; k < JF; ++k) {
                scan[k] = false;
                len[k] = 0;
                st[k] = 0;
                if (!ok[k]) continue;
                // rep[v] == rold[v] already for the root piece's vertices
                if (p[k] != ro[k]) {
                    rep[v[k]] = p[k];
                    const Row h = row_head(g, v[k]);
                    st[k] = h.start;
                    len[k] = h.used;
                    scan[k] = len[k] > 0;
                }
            }
#pragma unroll
            for (int k = 0; k < JF; ++k) {
                unsigned vm = __ballot_sync(0xffffffffu, ok[k]);
                if (ok[k]) {
                    unsigned grp = __match_any_sync(vm, p[k]);
                    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) {
                        piece_count(s_wk, s_wc, w, p[k], (unsigned)__popc(grp));
                    }
                }
            }
            long long q[JF], eo[JF];
            block_reserve_rows<JF>(&ctl->ndet, scan, len, q, eo);
#pragma unroll
            for (int k = 0; k < JF; ++k) {
                if (scan[k]) {
                    D[q[k]] = v[k];
                    roff[q[k]] = (unsigned)eo[k];
                    rl.base[q[k]] = st[k];
                    rl.meta[q[k]] = make_int2(p[k], ro[k]);
                }
                warp_fill_tiles(rl.tile, scan[k], eo[k], len[k], (int)q[k]);
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < WT_SLOTS; t += blockDim.x)
            if (s_wk[t] != -1) atomicAdd(&w[s_wk[t]], s_wc[t]);
    } else {
        // J[v] may later be overwritten by another walk's halving step with
        // a non-root ancestor; rep[v] takes this thread's own result.
        for (long long i = gtid(); i < cnt; i += gstride()) {
            int v = use_list ? A[i] : (int)i;
            J[v] = par[v];
        }
        if (!grid_barrier(ctl, &ctl->bar[0])) return;
        for (long long i = gtid(); i < cnt; i += gstride()) {
            int v = use_list ? A[i] : (int)i;
            int root = find_halving(J, v, ctl);
            J[v] = root;
            rep[v] = root;
        }
        if (gtid() == 0) ctl->jump_rounds = 1;
        if (mode == 0) return;
        if (!grid_barrier(ctl, &ctl->bar[0])) return;
        for (long long i = gtid(); i < cnt; i += gstride()) {
            int v = A[i];
            atomicAdd(&w[LD(rep[v])], 1u);
        }
    }
    if (!grid_barrier(ctl, &ctl->bar[0])) return;
    // heaviest piece per cut tree: its pieces are the root piece and one
    // piece per cut vertex, so the cut list covers them all
    const long long nc = (long long)ctl->ncut;
    if (gtid() == 0) ctl->flag[0] = 0;   // set by the swap check below
    heaviest_pieces(cuts, nc, rold, w, heavy);
    if (!grid_barrier(ctl, &ctl->bar[0])) return;
    // the provisional list left out each tree's root piece; where another
    // piece is heavier, rebuild the list with the exact rule (rare)
    {
        bool swap = false;
        for (long long i = gtid(); i < nc; i += gstride()) {
            int r = rold[cuts[i]];
            swap |= (int)(unsigned)LD(heavy[r]) != r;
        }
        // (the halving root search builds no provisional list: always exact)
        if (__syncthreads_or(swap || !sync_rounds) && threadIdx.x == 0) atomicOr(&ctl->flag[0], 1);
    }
    if (!grid_barrier(ctl, &ctl->bar[0])) return;
    if (*(volatile int *)&ctl->flag[0]) {
        if (gtid() == 0) ctl->ndet = 0;
        if (!grid_barrier(ctl, &ctl->bar[0])) return;
        for (long long base = (long long)blockIdx.x * blockDim.x; base < cnt; base += gstride()) {
            long long i = base + threadIdx.x;
            bool scan[1] = {false};
            int v = 0, hp = 0, pv = 0, len[1] = {0};
            unsigned st = 0;
            if (i < cnt) {
                v = A[i];
                hp = (int)(unsigned)LD(heavy[rold[v]]);
                const Row h = row_head(g, v);
                st = h.start;
                len[0] = h.used;
                pv = LD(rep[v]);
                scan[0] = pv != hp && len[0] > 0;
            }
            long long q[1], eo[1];
            block_reserve_rows<1>(&ctl->ndet, scan, len, q, eo);
            if (scan[0]) {
                D[q[0]] = v;
                roff[q[0]] = (unsigned)eo[0];
                rl.base[q[0]] = st;
                rl.meta[q[0]] = make_int2(pv, hp);
            }
            warp_fill_tiles(rl.tile, scan[0], eo[0], len[0], (int)q[0]);
        }
        if (!grid_barrier(ctl, &ctl->bar[0])) return;
    }
    // the packed row counter becomes the row count; roff[nd] = all entries
    if (gtid() == 0) {
        const u64 pk = *(volatile u64 *)&ctl->ndet;
        ctl->ndet = pk >> 32;
        roff[pk >> 32] = (unsigned)pk;
    }
}

// Move the pair table into the candidate list (one candidate per piece
// pair, its minimum key) and free the slots for the next batch.
__device__ __forceinline__ void compact_pairs(Ctl *ctl, PairTable pt, u64 *ck, int *ca, int *cb, u64 cand_cap) {
    // four slots per thread and iteration, one counter reservation per
    // block (the table has far more slots than warps have lanes, and most
    // warps hold an occupied slot: a per-warp append would queue on the
    // counter)
    const long long T = (long long)pt.mask + 1;
    const long long S = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < T; base += 4 * S) {
        u64 pair[4], k[4];
        bool on[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            long long i = base + q * S + threadIdx.x;
            pair[q] = i < T ? pt.pk[i] : EMPTY_KEY;
            on[q] = pair[q] != EMPTY_KEY;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            k[q] = 0;
            if (on[q]) {
                long long i = base + q * S + threadIdx.x;
                k[q] = pt.mk[i];
                pt.pk[i] = EMPTY_KEY;
                pt.mk[i] = EMPTY_KEY;
            }
        }
        long long p[4];
        block_reserve4(&ctl->ncand, on, p);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (!on[q]) continue;
            if ((u64)p[q] < cand_cap) {
                ck[p[q]] = k[q];
                ca[p[q]] = (int)(pair[q] >> 32);
                cb[p[q]] = (int)(pair[q] & 0xFFFFFFFFu);
            } else {
                atomicOr(&ctl->err, ERR_CAPACITY);
            }
        }
    }
}
// Per-block table of hot indices for 64-bit minimum updates: lanes of a
// warp with the same index combine first; an index held by two or more
// lanes of a warp (one piece, such as the giant one, can be an endpoint of
// most candidates) is combined in shared memory and sent to global memory
// once per block by hm_flush; a lone index goes straight to global memory.
#define HM_SLOTS 16
#define HM_PROBES 4
struct HotMin {
    int k[HM_SLOTS];
    u64 v[HM_SLOTS];
    int rst[HM_SLOTS];
};
__device__ __forceinline__ void hm_init(HotMin &t) {
    for (int i = threadIdx.x; i < HM_SLOTS; i += blockDim.x) {
        t.k[i] = -1;
        t.v[i] = EMPTY_KEY;
        t.rst[i] = 0;
    }
    __syncthreads();
}
// slot of idx in the table (inserted when ins and absent), or -1
__device__ __forceinline__ int hm_slot(HotMin &t, int idx, bool ins) {
    unsigned h = ((unsigned)idx * 0x9E3779B1u) >> 28;
    for (int p = 0; p < HM_PROBES; ++p) {
        int key = *(volatile int *)&t.k[h];
        if (key == -1 && ins) key = atomicCAS(&t.k[h], -1, idx);
        if (key == idx || (key == -1 && ins)) return (int)h;
        if (key == -1) return -1;
        h = (h + 1) & (HM_SLOTS - 1);
    }
    return -1;
}
// The lanes of the first two indices seen in the warp combine their keys (one
// piece, such as the giant one, can be an end of most candidates); the other
// lanes go to global memory one by one, unless their key is no new minimum.
// (A reduction over each group of equal lanes runs the groups one after
// another: up to 32 times two reductions where most indices differ.)
__device__ __forceinline__ void hm_min(HotMin &t, u64 *arr, int idx, u64 k, bool pred) {
    unsigned m = __ballot_sync(__activemask(), pred);
    if (!pred) return;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int round = 0; round < 2; ++round) {
        const int l0 = __ffs(m) - 1, i0 = __shfl_sync(m, idx, l0);
        const unsigned g = __ballot_sync(m, idx == i0);
        if (__popc(g) > 1) {
            if (idx == i0) {
                const u64 kmin = group_min_u64(g, k);
                if (lane == l0) {
                    const int sl = hm_slot(t, idx, true);
                    if (sl >= 0) atomicMin(&t.v[sl], kmin);
                    else atomicMin(&arr[idx], kmin);
                }
                return;
            }
            m &= ~g;
            if (!m) return;
        } else if (round == 0) {
            if (lane == l0) break;
            m &= ~g;
            if (!m) return;
        }
    }
    if (k < __ldcg(&arr[idx])) atomicMin(&arr[idx], k);
}
// arr[idx] = EMPTY_KEY, once per block for the table's indices, and for the
// others by whoever still finds a key there.  (With a match of all lanes'
// indices and a store for each one an insert of 1M edges between 1,000 trees
// hooked for 1,195 us instead of 995.)
__device__ __forceinline__ void hm_reset(HotMin &t, u64 *arr, int idx, bool pred) {
    unsigned m = __ballot_sync(__activemask(), pred);
    if (!pred) return;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int round = 0; round < 2; ++round) {
        const int l0 = __ffs(m) - 1, i0 = __shfl_sync(m, idx, l0);
        const unsigned g = __ballot_sync(m, idx == i0);
        if (__popc(g) > 1) {
            if (idx == i0) {
                if (lane == l0) {
                    const int sl = hm_slot(t, idx, true);
                    if (sl >= 0) t.rst[sl] = 1;
                    else if (arr[idx] != EMPTY_KEY) arr[idx] = EMPTY_KEY;
                }
                return;
            }
            m &= ~g;
            if (!m) return;
        } else if (round == 0) {
            if (lane == l0) break;
            m &= ~g;
            if (!m) return;
        }
    }
    if (arr[idx] != EMPTY_KEY) arr[idx] = EMPTY_KEY;
}
// sends the table's minima to arr (min) and its resets to rst_arr, then
// clears it; every thread of the block calls it
__device__ __forceinline__ void hm_flush(HotMin &t, u64 *arr, u64 *rst_arr) {
    __syncthreads();
    for (int i = threadIdx.x; i < HM_SLOTS; i += blockDim.x) {
        if (t.k[i] != -1) {
            if (t.v[i] != EMPTY_KEY) atomicMin(&arr[t.k[i]], t.v[i]);
            if (t.rst[i]) rst_arr[t.k[i]] = EMPTY_KEY;
        }
        t.k[i] = -1;
        t.v[i] = EMPTY_KEY;
        t.rst[i] = 0;
    }
    __syncthreads();
}

// Roots of both ends of a candidate, walked side by side.  Nobody hooks
// meanwhile, and a barrier lies behind those who did: the entries may come from
// L1 (the roots of few components are read by all candidates).  One after the
// other and from L2 they took 130 of the 995 us above.
__device__ __forceinline__ void find_roots(const int *comp, int &a, int &b, Ctl *ctl) {
    for (int it = 0; it < (1 << 24); ++it) {
        const int pa = comp[a], pb = comp[b];
        if (pa == a && pb == b) return;
        a = pa;
        b = pb;
    }
    atomicOr(&ctl->err, ERR_ROUNDS);
}

// Replacement edges by hook-and-compress over the trees of F^ (pieces).
// Each round: every component takes the minimum key among its incident
// candidates (64-bit atomicMin); a component whose minimum edge leads to
// another component hooks onto it (a mutual choice hooks the larger id under
// the smaller); each hooking edge joins E_r.  Candidates inside one
// component are dropped, the rest are compacted for the next round.  With
// distinct keys this is Boruvka's algorithm: E_r is the unique minimum
// spanning forest of the piece multigraph, |E_r| = k - l.
// Rounds r, r+1, ... of the hook-and-compress, by the whole grid (ONE
// false: grid barriers between phases) or by block 0 alone (ONE true: block
// barriers).  On the grid, a round that starts with at most HOOK_TAIL live
// candidates (after round 0 on R-MAT batches: about 2.5% of them) is handed
// to block 0: every block reads the same count after the barrier, so all
// take that branch together.  Returns -1 when a grid barrier gave up, the
// round to hand to block 0 (grid only), or 0 when done.
template <bool ONE>
__device__ __forceinline__ int hook_rounds(Ctl *ctl, HotMin &hm, int r, long long c0, u64 *ck0, int *ca0, int *cb0,
                                           u64 *ck1, int *ca1, int *cb1, int *comp, u64 *best0, u64 *best1, u64 *er,
                                           long long er_cap) {
    const long long T = ONE ? (long long)threadIdx.x : gtid();
    const long long S = ONE ? (long long)blockDim.x : gstride();
    const long long B0 = ONE ? 0 : (long long)blockIdx.x * blockDim.x;
    for (;; ++r) {
        if (r >= MAX_ROUNDS) {
            if (T == 0) atomicOr(&ctl->err, ERR_ROUNDS);
            return 0;
        }
        u64 *ck = (r & 1) ? ck1 : ck0, *ckn = (r & 1) ? ck0 : ck1;
        int *ca = (r & 1) ? ca1 : ca0, *can = (r & 1) ? ca0 : ca1;
        int *cb = (r & 1) ? cb1 : cb0, *cbn = (r & 1) ? cb0 : cb1;
        u64 *best = (r & 1) ? best1 : best0, *bestn = (r & 1) ? best0 : best1;
        const long long c = r == 0 ? c0 : (long long)*(volatile u64 *)&ctl->cnt[r % 3];
        if (!ONE && r > 0 && c <= HOOK_TAIL) return r;
        if (T == 0) {
            ctl->cnt[(r + 2) % 3] = 0;
            ctl->flag[(r + 1) % 3] = 0;
        }
        // phase A: roots of both ends, per-component minimum key
        for (long long i = T; i < c; i += S) {
            int a = LD(ca[i]), b = LD(cb[i]);
            const u64 k = LD(ck[i]);
            if (r > 0) {   // every endpoint is its own root in round 0
                find_roots(comp, a, b, ctl);
                ca[i] = a;
                cb[i] = b;
            }
            hm_min(hm, best, a, k, a != b);
            hm_min(hm, best, b, k, a != b);
        }
        hm_flush(hm, best, bestn);
        if (!ONE && !grid_barrier(ctl, &ctl->bar[1])) return -1;
        // phase B: hook along minimum edges, keep the rest (block-uniform
        // loop: list appends are reserved once per block)
        bool hooked = false;
        for (long long b0 = B0; b0 < c; b0 += S) {
            const long long i = b0 + threadIdx.x;
            int a = 0, b = 0;
            bool alive = false, hook = false, keep = false;
            u64 k = 0;
            if (i < c) {
                a = LD(ca[i]);
                b = LD(cb[i]);
                alive = a != b;
                k = LD(ck[i]);
            }
            if (alive) {
                const bool ba = best[a] == k, bb = best[b] == k;   // (final since the barrier: from L1)
                if (ba && bb) comp[a > b ? a : b] = a > b ? b : a;
                else if (ba) comp[a] = b;
                else if (bb) comp[b] = a;
                hook = ba || bb;
                keep = !hook;
            }
            if (r > 0) {   // (both arrays start empty)
                hm_reset(hm, bestn, a, alive);
                hm_reset(hm, bestn, b, alive);
            }
            hooked |= hook;
            long long pe = block_append(&ctl->ner, hook);
            if (hook) {
                if (pe < er_cap) er[pe] = k;
                else atomicOr(&ctl->err, ERR_CAPACITY);
            }
            long long pk = block_append(&ctl->cnt[(r + 1) % 3], keep);
            if (keep) {
                ckn[pk] = k;
                can[pk] = a;
                cbn[pk] = b;
            }
        }
        hm_flush(hm, best, bestn);
        const int any = __syncthreads_or(hooked);
        if (ONE) {
            if (!any) break;
        } else {
            if (any && threadIdx.x == 0) atomicOr(&ctl->flag[r % 3], 1);
            if (!grid_barrier(ctl, &ctl->bar[1])) return -1;
            if (!*(volatile int *)&ctl->flag[r % 3]) break;
        }
    }
    if (T == 0) ctl->hook_rounds = r;
    return 0;
}

// Set up each candidate endpoint once (the first lane to stamp it).
__device__ __forceinline__ void hook_init(const HookArgs &h, long long c0, unsigned ep) {
    for (long long i = gtid(); i < c0; i += gstride()) {
        hook_slot_init(h.hs, LD(h.ca[0][i]), ep);
        hook_slot_init(h.hs, LD(h.cb[0][i]), ep);
    }
}

// All rounds: on the grid while many candidates are live, the rest (or all of
// a short list) by block 0.  Returns -1 when a grid barrier gave up.
__device__ __forceinline__ int hook_all(Ctl *ctl, HotMin &hm, const HookArgs &h, long long c0) {
    int r = 0;
    const bool few = c0 <= HOOK_FEW;
    if (!few)
        r = hook_rounds<false>(ctl, hm, 0, c0, h.ck[0], h.ca[0], h.cb[0], h.ck[1], h.ca[1], h.cb[1], h.hs.comp,
                               h.hs.best0, h.hs.best1, h.er, h.er_cap);
    if ((few || r > 0) && blockIdx.x == 0)
        hook_rounds<true>(ctl, hm, r, c0, h.ck[0], h.ca[0], h.cb[0], h.ck[1], h.ca[1], h.cb[1], h.hs.comp, h.hs.best0,
                          h.hs.best1, h.er, h.er_cap);
    return r;
}

// Path reversal by walking (ReversePaths, Algorithm 1): the path x = v0, v1 =
// parent[v0], ..., vL (the piece root) is read first and then reversed
// (parent[v_j] <- v_{j-1}, parent[v0] <- y).  Each child piece has exactly
// one oriented edge and pieces are disjoint, so the walks never touch the
// same vertex, and a walk needs nothing but its own edge: whoever orients an
// edge can walk it at once.  A path of more than WALK_MAX edges stays as it
// is: its piece is stamped in long_ep and reversed by the pointer-doubling
// marks.  Returns the vertices reversed.
// Reversing while walking, each load behind a store into sectors that other
// walks read and write, took five times as long: 283 -> 51 us per delete
// batch on the 4096 x 4096 grid (100K edges), 118 -> 27 us on the 256-graph
// union (1.6M edges).
__device__ __forceinline__ int walk_path(Ctl *ctl, int *parent, int x, int y, unsigned *long_ep, int piece,
                                         unsigned ep) {
    int path[WALK_MAX];   // path[j] = parent[v_j]
    int len = 0, cur = x;
    for (; len < WALK_MAX; ++len) {
        const int nxt = LD(parent[cur]);
        if (nxt == cur) break;
        path[len] = nxt;
        cur = nxt;
    }
    if (len == WALK_MAX) {
        long_ep[piece] = ep;
        ctl->nlong = 1;
        return 0;
    }
    int prev = y;
    cur = x;
    for (int j = 0; j < len; ++j) {
        const int nxt = path[j];
        parent[cur] = prev;
        prev = cur;
        cur = nxt;
    }
    parent[cur] = prev;
    return len;
}

// Orientation of replacement edge i: down = its lower-id endpoint's piece
// p0 is the parent of the other piece p1.  The child piece P of edge {x, y}
// (x in P) gets the oriented edge x -> y, its attach point x and the
// super-tree's root as its new representative (each non-root piece is the
// child of exactly one edge: one write per piece; the super-root keeps its
// representative).  A child that is the root piece of a cut tree (its root
// was stamped by the cut) is noted: after a top-down delete the affected list
// holds the detached vertices only, and the refresh then has to pass over
// all vertices.  Returns the vertices that its walk reversed.
__device__ __forceinline__ int orient_one(Ctl *ctl, const OrientArgs &a, long long i, bool down, unsigned ep) {
    const u64 k = a.er[i];
    const int x0 = (int)klo(k), x1 = (int)khi(k);
    const int p0 = LD(a.ep[2 * i]), p1 = LD(a.ep[2 * i + 1]);
    const int child = down ? p1 : p0;
    const int x = down ? x1 : x0, y = down ? x0 : x1;
    a.chx[i] = x;
    a.chy[i] = y;
    a.att_x[child] = x;
    a.att_ep[child] = ep;
    a.newrep[child] = LD(a.minp[LD(a.eroot[i])]);
    a.rep_ep[child] = ep;
    if (a.aff_ep[child] == ep) ctl->need_root = 1;
    return a.walk ? walk_path(ctl, a.parent, x, y, a.long_ep, child, ep) : 0;
}

// Wyllie list ranking of ncore list cells in shared memory by one block:
// val (svc) = cells from here to the end of the list, next pointers in snc
// (NIL at the end); svn / snn are the ping-pong buffers.  Returns the rounds
// taken (ERR_ROUNDS latched if the bound is hit) and leaves the ranks in
// *out (one of svc / svn).
__device__ int rank_block(Ctl *ctl, int *svc, int *svn, int *snc, int *snn, int ncore, int **out) {
    int r = 0;
    for (;; ++r) {
        int ch = 0;
        for (int i = threadIdx.x; i < ncore; i += blockDim.x) {
            const int sx = snc[i];
            if (sx != NIL) {
                svn[i] = svc[i] + svc[sx];
                snn[i] = snc[sx];
                ch = 1;
            } else {
                svn[i] = svc[i];
                snn[i] = NIL;
            }
        }
        const int any = __syncthreads_or(ch);
        int *t = svc; svc = svn; svn = t;
        t = snc; snc = snn; snn = t;
        if (!any) break;
        if (r >= MAX_ROUNDS) {
            if (threadIdx.x == 0) atomicOr(&ctl->err, ERR_ROUNDS);
            break;
        }
    }
    *out = svc;
    return r + 1;
}

// The core of the super-forest (the edges that are not leaf edges, listed
// in cel) oriented by one block: adjacency ranges claimed by the first arc
// of each core piece, arcs placed, Euler successors (as in the grid phases
// of orient_grid) written straight into shared memory, ranked there, and each
// core edge oriented by its arc that comes first.  Block barriers only.
__device__ void orient_small_core(Ctl *ctl, const OrientArgs &a, const int *cel, long long nce, unsigned ep) {
    __shared__ int s_nc;
    if (threadIdx.x == 0) s_nc = 0;
    __syncthreads();
    for (long long t = threadIdx.x; t < 2 * nce; t += blockDim.x) {
        const long long j = 2 * (long long)LD(cel[t >> 1]) + (t & 1);
        const int id = LD(a.eid[j]);
        if (atomicCAS(&a.poff[id], -1, -2) == -1) a.poff[id] = atomicAdd(&s_nc, LD(a.cdeg[id]));
    }
    __syncthreads();
    const int ncore = s_nc;
    for (long long t = threadIdx.x; t < 2 * nce; t += blockDim.x) {
        const long long j = 2 * (long long)LD(cel[t >> 1]) + (t & 1);
        const int id = LD(a.eid[j]);
        const int slot = a.poff[id] + atomicAdd(&a.pcur[id], 1);
        a.adj[slot] = (int)j;
        a.apos[j] = slot;
    }
    __syncthreads();
    extern __shared__ int s_rank[];
    int *svc = s_rank, *svn = svc + a.rank_arcs, *snc = svn + a.rank_arcs, *snn = snc + a.rank_arcs;
    for (long long t = threadIdx.x; t < 2 * nce; t += blockDim.x) {
        const long long j = 2 * (long long)LD(cel[t >> 1]) + (t & 1);
        const long long tw = j ^ 1;
        const int hid = LD(a.eid[tw]);   // the arc's head = the twin's source
        const int start = a.poff[hid], end = start + LD(a.cdeg[hid]);
        const int nx = a.apos[tw] + 1;
        int succ;
        if (nx == end) {
            const bool is_root = LD(a.minp[LD(a.eroot[j >> 1])]) == LD(a.ep[tw]);
            succ = is_root ? NIL : start;
        } else {
            succ = nx;
        }
        const int si = a.apos[j];
        snc[si] = succ;
        svc[si] = 1;
    }
    __syncthreads();
    int *rank = nullptr;
    const int rounds = rank_block(ctl, svc, svn, snc, snn, ncore, &rank);
    int rev = 0;
    for (long long t = threadIdx.x; t < nce; t += blockDim.x) {
        const long long i = LD(cel[t]);
        rev += orient_one(ctl, a, i, rank[a.apos[2 * i]] > rank[a.apos[2 * i + 1]], ep);
    }
    block_add(&ctl->reversed, rev);
    if (threadIdx.x == 0) {
        ctl->ncore = (u64)ncore;
        ctl->rank_rounds = rounds;
    }
}

// Orientation of E_r (Algorithm 2, phase 2).  The replacement edges form a
// forest over the pieces (the super-forest); each super-tree is rooted at
// its piece with the smallest root id.  A non-root piece with a single
// replacement edge is a leaf: its parent is its only neighbour, no tour
// needed.  The rest (the core, a tree per super-tree that still holds the
// root) is rooted by the Euler tour technique: circular adjacency lists give
// the successor of arc a->b as the arc after b->a in b's list; the circuit is
// opened at the root, the arcs are ranked by Wyllie's pointer jumping, and
// each edge is oriented by its arc that comes first.  The child piece P of
// edge {x, y} (x in P) gets the oriented replacement edge x -> y; every piece
// of the super-tree gets the root as its new representative.
__device__ void orient_grid(Ctl *ctl, const OrientArgs &a) {
    const long long ner = (long long)*(volatile u64 *)&ctl->ner;
    const unsigned ep = ctl->epoch;
    u64 *bar = &ctl->bar[2];
    // Arc j of edge j/2 runs from the piece of its (j odd ? larger : smaller)
    // endpoint to the other piece.  Phase 1 caches each arc's source piece
    // (ep), later phases its dense id (eid) and each edge's super-tree root
    // (eroot), so no phase re-walks rep / pidx / the hook forest.
    // phase 1: dense ids for the pieces touched by E_r
    if (gtid() == 0) ctl->ncore = ctl->cnt[0] = ctl->cnt[1] = 0;
    // the path walks follow parent pointers one dependent load at a time:
    // pull the forest into L2 now, while the phases below wait at their
    // barriers (one 128-byte line per thread or so)
    if (ner > 0) l2_prefetch(a.parent, 4 * a.n, gtid(), gstride());
    // (block-uniform loop: the dense ids are reserved once per block)
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < 2 * ner; b0 += gstride()) {
        const long long j = b0 + threadIdx.x;
        bool first = false;
        int p = 0;
        if (j < 2 * ner) {
            u64 k = a.er[j >> 1];
            p = a.rep[(j & 1) ? khi(k) : klo(k)];
            a.ep[j] = p;
            // one lane per piece among the warp's lanes claims it (a piece
            // such as the giant one is an endpoint of most of the edges)
            unsigned grp = __match_any_sync(__activemask(), p);
            bool lead = (int)(threadIdx.x & 31) == __ffs(grp) - 1;
            first = lead && __ldcg(&a.pstamp[p]) != ep && atomicExch(&a.pstamp[p], ep) != ep;
        }
        long long id = block_append(&ctl->npc, first);
        if (first) {
            a.pidx[p] = (int)id;
            a.plist[id] = p;
            a.pdeg[id] = 0;
            a.cdeg[id] = 0;
            a.pcur[id] = 0;
            a.poff[id] = -1;   // (claimed by the core path for small cores)
            // the root piece of the hook forest holds its super-tree's slot
            if (find_root(a.comp, p, ctl) == p) a.minp[p] = INT_MAX;
        }
    }
    if (!grid_barrier(ctl, bar)) return;
    // phase 2: smallest piece id per super-tree, degrees (lanes with the
    // same target combine first: one super-tree or piece can collect most
    // of the batch's edges)
    for (long long j = gtid(); j < 2 * ner; j += gstride()) {
        int p = LD(a.ep[j]);
        int id = LD(a.pidx[p]);
        int root = find_root(a.comp, p, ctl);
        a.eid[j] = id;
        if (!(j & 1)) a.eroot[j >> 1] = root;
        unsigned act = __activemask();
        unsigned g1 = __match_any_sync(act, root);
        int pm = (int)__reduce_min_sync(g1, (unsigned)p);
        if ((int)(threadIdx.x & 31) == __ffs(g1) - 1) atomicMin(&a.minp[root], pm);
        unsigned g2 = __match_any_sync(act, id);
        if ((int)(threadIdx.x & 31) == __ffs(g2) - 1) atomicAdd(&a.pdeg[id], __popc(g2));
    }
    if (!grid_barrier(ctl, bar)) return;
    // phase 2b: leaf edges (a non-root piece with one edge); core degrees
    for (long long i = gtid(); i < ner; i += gstride()) {
        int p0 = LD(a.ep[2 * i]), p1 = LD(a.ep[2 * i + 1]);
        int id0 = LD(a.eid[2 * i]), id1 = LD(a.eid[2 * i + 1]);
        int sr = LD(a.minp[LD(a.eroot[i])]);
        bool leaf0 = LD(a.pdeg[id0]) == 1 && sr != p0;
        bool leaf1 = LD(a.pdeg[id1]) == 1 && sr != p1;
        unsigned char lf = leaf0 ? 1 : (leaf1 ? 2 : 0);
        a.lf[i] = lf;
        unsigned act = __activemask();
        unsigned core = __ballot_sync(act, !lf);
        if (!lf) {
            unsigned g0 = __match_any_sync(core, id0);
            if ((int)(threadIdx.x & 31) == __ffs(g0) - 1) atomicAdd(&a.cdeg[id0], __popc(g0));
            unsigned g1 = __match_any_sync(core, id1);
            if ((int)(threadIdx.x & 31) == __ffs(g1) - 1) atomicAdd(&a.cdeg[id1], __popc(g1));
        }
        // the core edges, listed for the one-block path of small cores
        if (!lf) {
            const int ld = __ffs(core) - 1;
            u64 b = 0;
            if ((int)(threadIdx.x & 31) == ld) b = atomicAdd(&ctl->cnt[0], (u64)__popc(core));
            b = __shfl_sync(core, b, ld);
            a.cel[b + __popc(core & ((1u << (threadIdx.x & 31)) - 1u))] = (int)i;
        }
    }
    if (!grid_barrier(ctl, bar)) return;
    {
        // A small core (small batches: tens of edges) is done by block 0
        // alone with block barriers (adjacency, Euler successors, ranking in
        // shared memory, orientation), while every block orients the leaf
        // edges.  A larger one first gets a second round of leaf raking
        // (phase 2c: on R-MAT it leaves about a tenth of the core), and
        // takes the grid phases below only if it is still large.
        long long nce = (long long)*(volatile u64 *)&ctl->cnt[0];
        const int *cel = a.cel;
        if (nce > ORIENT_SMALL_EDGES) {
            // phase 2c: a core piece with a single core edge that is not its
            // super-tree's root is a leaf of the remaining core; its edge is
            // oriented towards the other piece (lf) and both core degrees
            // drop.  Core degrees only fall, so a stale read can miss a leaf
            // but never make one up (the edge being looked at is still
            // alive, so a degree read as 1 is exactly 1), and both ends of
            // one edge cannot be such leaves (every core component holds its
            // root).  The edges left are listed again (second half of cel).
            int *cel2 = a.cel + ner;
            for (long long b0 = gtid() & ~31ll; b0 < nce; b0 += gstride()) {
                const long long t = b0 + (threadIdx.x & 31);
                bool keep = false;
                long long i = 0;
                if (t < nce) {
                    i = LD(a.cel[t]);
                    const int id0 = LD(a.eid[2 * i]), id1 = LD(a.eid[2 * i + 1]);
                    const int p0 = LD(a.ep[2 * i]), p1 = LD(a.ep[2 * i + 1]);
                    const int sr = LD(a.minp[LD(a.eroot[i])]);
                    const bool l0 = LD(a.cdeg[id0]) == 1 && p0 != sr;
                    const bool l1 = !l0 && LD(a.cdeg[id1]) == 1 && p1 != sr;
                    if (l0 || l1) {
                        a.lf[i] = l0 ? 1 : 2;
                        atomicSub(&a.cdeg[id0], 1);
                        atomicSub(&a.cdeg[id1], 1);
                    } else {
                        keep = true;
                    }
                }
                const unsigned km = __ballot_sync(0xffffffffu, keep);
                if (km) {
                    const int lane = threadIdx.x & 31, ld = __ffs(km) - 1;
                    u64 q0 = 0;
                    if (lane == ld) q0 = atomicAdd(&ctl->cnt[1], (u64)__popc(km));
                    q0 = __shfl_sync(0xffffffffu, q0, ld);
                    if (keep) cel2[q0 + __popc(km & ((1u << lane) - 1u))] = (int)i;
                }
            }
            if (!grid_barrier(ctl, bar)) return;
            nce = (long long)*(volatile u64 *)&ctl->cnt[1];
            cel = cel2;
        }
        if (nce <= ORIENT_SMALL_EDGES) {
            // (block 0 leaves the leaf edges to the others: its core and
            // their walks run side by side)
            if (blockIdx.x == 0) orient_small_core(ctl, a, cel, nce, ep);
            const bool alone = gridDim.x == 1;
            if (blockIdx.x == 0 && !alone) return;
            const long long t0 = alone ? gtid() : gtid() - blockDim.x, st = alone ? gstride() : gstride() - blockDim.x;
            int rev = 0;
            for (long long i = t0; i < ner; i += st) {
                const unsigned char lf = LD(a.lf[i]);
                if (lf) rev += orient_one(ctl, a, i, lf == 2, ep);
            }
            block_add(&ctl->reversed, rev);
            return;
        }
    }
    // phase 3: adjacency ranges of the core pieces, reserved per block from
    // one cursor (ctl->ncore ends as the number of core arcs; the order of
    // the ranges is immaterial)
    const long long np = (long long)*(volatile u64 *)&ctl->npc;
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < np; b0 += gstride()) {
        const long long i = b0 + threadIdx.x;
        const long long d = i < np ? LD(a.cdeg[i]) : 0;
        const long long off = block_reserve(&ctl->ncore, d);
        if (i < np) a.poff[i] = (int)off;
    }
    if (!grid_barrier(ctl, bar)) return;
    // phase 4: place core arcs in their source piece's adjacency
    for (long long j = gtid(); j < 2 * ner; j += gstride()) {
        bool core = !LD(a.lf[j >> 1]);
        unsigned cm = __ballot_sync(__activemask(), core);
        if (!core) continue;
        int id = LD(a.eid[j]);
        unsigned grp = __match_any_sync(cm, id);
        int lane = threadIdx.x & 31, leader = __ffs(grp) - 1;
        int base = 0;
        if (lane == leader) base = atomicAdd(&a.pcur[id], __popc(grp));
        base = __shfl_sync(grp, base, leader);
        int slot = LD(a.poff[id]) + base + __popc(grp & ((1u << lane) - 1u));
        a.adj[slot] = (int)j;
        a.apos[j] = slot;
    }
    if (!grid_barrier(ctl, bar)) return;
    // phase 5: Euler successors of core arcs, in slot space (the position of
    // an arc in the core adjacency array): the successor of arc a->b is the
    // slot after b->a's slot in b's list, wrapping to the list start; the
    // circuit is opened at each super-tree root
    for (long long j = gtid(); j < 2 * ner; j += gstride()) {
        if (LD(a.lf[j >> 1])) continue;
        long long tw = j ^ 1;
        int hid = LD(a.eid[tw]);                  // the arc's head = the twin's source
        int start = LD(a.poff[hid]), end = start + LD(a.cdeg[hid]);
        int nx = LD(a.apos[tw]) + 1;
        int succ;
        if (nx == end) {
            bool is_root = LD(a.minp[LD(a.eroot[j >> 1])]) == LD(a.ep[tw]);
            succ = is_root ? NIL : start;
        } else {
            succ = nx;
        }
        int si = LD(a.apos[j]);
        a.nx0[si] = succ;
        a.val0[si] = 1;
    }
    if (!grid_barrier(ctl, bar)) return;
    // phase 6: list ranking (Wyllie): val = arcs from here to the tour end.
    // A core of at most rank_arcs arcs is ranked by block 0 alone in
    // shared memory (block barriers instead of grid barriers per round).
    const long long ncore = (long long)*(volatile u64 *)&ctl->ncore;
    int *vc = a.val0, *vn = a.val1, *nc = a.nx0, *nn = a.nx1;
    int r = 0;
    if (ncore <= a.rank_arcs) {
        if (blockIdx.x == 0) {
            extern __shared__ int s_rank[];
            int *svc = s_rank, *svn = svc + a.rank_arcs, *snc = svn + a.rank_arcs, *snn = snc + a.rank_arcs;
            for (long long i = threadIdx.x; i < ncore; i += blockDim.x) {
                svc[i] = LD(a.val0[i]);
                snc[i] = LD(a.nx0[i]);
            }
            __syncthreads();
            int *rank = nullptr;
            const int rounds = rank_block(ctl, svc, svn, snc, snn, (int)ncore, &rank);
            for (long long i = threadIdx.x; i < ncore; i += blockDim.x) a.val0[i] = rank[i];
            if (threadIdx.x == 0) ctl->rank_rounds = rounds;
        }
        if (!grid_barrier(ctl, bar)) return;
        vc = a.val0;
    } else {
        for (;; ++r) {
            if (r >= MAX_ROUNDS) {
                if (gtid() == 0) atomicOr(&ctl->err, ERR_ROUNDS);
                return;
            }
            if (gtid() == 0) ctl->flag[(r + 1) % 3] = 0;
            bool ch = false;
            for (long long i = gtid(); i < ncore; i += gstride()) {
                int sx = LD(nc[i]);
                if (sx != NIL) {
                    vn[i] = LD(vc[i]) + LD(vc[sx]);
                    nn[i] = LD(nc[sx]);
                    ch = true;
                } else {
                    vn[i] = LD(vc[i]);
                    nn[i] = NIL;
                }
            }
            if (__syncthreads_or(ch) && threadIdx.x == 0) atomicOr(&ctl->flag[r % 3], 1);
            if (!grid_barrier(ctl, bar)) return;
            int again = *(volatile int *)&ctl->flag[r % 3];
            int *t = vc; vc = vn; vn = t;
            t = nc; nc = nn; nn = t;
            if (!again) break;
        }
        if (gtid() == 0) ctl->rank_rounds = r + 1;
    }
    // phase 7: orient, attach points, new roots
    int rev = 0;
    for (long long i = gtid(); i < ner; i += gstride()) {
        const unsigned char lf = LD(a.lf[i]);
        const bool down = lf ? lf == 2 : LD(vc[LD(a.apos[2 * i])]) > LD(vc[LD(a.apos[2 * i + 1])]);
        rev += orient_one(ctl, a, i, down, ep);
    }
    block_add(&ctl->reversed, rev);
}
// Replacement edges and their orientation for a batch with at most C
// candidates, by one block in shared memory: the pieces get dense ids through
// a hash table, the hook-and-compress rounds and the orientation run on
// those.  On the grid the same batch is a chain of some twenty phases with a
// grid barrier, two or three dependent global loads and up to a launch between
// them, whatever its size.  The results (attach points, new roots, walks) are
// scattered stores and pointer chains: up to SMALL_OUT edges the same block
// writes them, more go to the whole grid after one barrier (35 of 90 us for
// 3,300 edges on one SM).
// The `pre` replacement edges that k_scan chose join the candidates again (the
// minimum spanning forest is the same), all with their own pieces as ends.
// Pieces: at most two per candidate.  A piece's minimum key is taken in two
// halves, which shared memory has native atomics for; what is needed one after
// the other shares memory.
#define SMALL_OUT 256
template <int C>
struct SmallTail {
    static constexpr int cand = C, pieces = 2 * C, slots = 3 * C;   // hash slots: two thirds full at most
    u64 key[C];
    union {
        unsigned short hl[slots];   // a hash slot's dense id
        struct {
            unsigned bhi[pieces], blo[pieces];   // a piece's minimum key
        };
        struct {
            int minp[pieces];
            unsigned char vis[pieces];
            unsigned short apos[pieces];   // an arc's place among its source's
        };
    };
    union {
        int hk[slots];              // hash table: piece, -1 free
        struct {
            unsigned short start[pieces];   // a piece's arcs
            unsigned arc[pieces];           // tour: arcs to the end << 16 | next place
        };
    };
    int pid[pieces];
    unsigned short comp[pieces];
    unsigned short a[C], b[C], er[C];
    int ner;
    static_assert(slots % ORIENT_THREADS == 0 && pieces % ORIENT_THREADS == 0, "items per thread");
    static_assert(pieces < 0xFFFF, "places and ranks of the tour are 16 bits");
};

// slot of piece p in the hash table (entered when absent)
template <class T>
__device__ __forceinline__ int tail_slot(T &t, int p) {
    unsigned h = ((unsigned)p * 0x9E3779B1u) % T::slots;
    for (;;) {
        int k = *(volatile int *)&t.hk[h];
        if (k == -1) k = atomicCAS(&t.hk[h], -1, p);
        if (k == -1 || k == p) return (int)h;
        h = h + 1 == T::slots ? 0 : h + 1;
    }
}
// root of dense piece x; the path is halved as it is walked (one round's hooks
// can make a chain of all pieces: a path whose keys rise), by several threads
// at once: an entry only ever moves to an ancestor
template <class T>
__device__ __forceinline__ int tail_root(T &t, int x) {
    volatile unsigned short *const c = t.comp;
    for (int it = 0; it < T::pieces; ++it) {
        const int p = c[x];
        if (p == x) break;
        const int g = c[p];
        if (g == p) return p;
        c[x] = (unsigned short)g;
        x = g;
    }
    return x;
}

// Ranks the arcs of the super-forest's Euler tour (as orient_grid does its
// core's): a piece's arcs side by side, the arc after b->a in b's list follows
// a->b, the circuit opened at each super-root, Wyllie's ranking with the arcs
// of a round in registers.  For super-forests deeper than TAIL_LEVELS, which
// the orientation by levels would take one barrier per level for: an insert
// that joins 4,000 vertices to a path took 3,852 us by levels and unhalved
// chains, 124 so (a path of 250: 135 and 61, of 60: 59 and 57; a random tree of
// 4,000, at most 32 deep: 92 and 89).
// arc[apos[2 e]] >> 16 and arc[apos[2 e + 1]] >> 16 are then the ranks of edge
// e's arcs from its first end and from its second.  Returns the rounds.
#define TAIL_LEVELS 32
#define TAIL_NIL 0xFFFFu
template <class T>
__device__ __noinline__ int tail_rank(int ner, int np) {
    extern __shared__ __align__(16) int s_rank[];
    T &t = *reinterpret_cast<T *>(s_rank);
    const int arcs = 2 * ner;
    auto source = [&](int j) { return (int)(j & 1 ? t.b[t.er[j >> 1]] : t.a[t.er[j >> 1]]); };
    for (int l = threadIdx.x; l < np; l += ORIENT_THREADS) t.arc[l] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < arcs; j += ORIENT_THREADS) t.apos[j] = (unsigned short)atomicAdd(&t.arc[source(j)], 1u);
    __syncthreads();
    {
        const int per = (np + ORIENT_THREADS - 1) / ORIENT_THREADS, l0 = threadIdx.x * per, l1 = min(np, l0 + per);
        int deg = 0;
        for (int l = l0; l < l1; ++l) deg += (int)t.arc[l];
        long long tot;
        int at = (int)block_excl_scan_ll(deg, &tot);
        for (int l = l0; l < l1; ++l) {
            t.start[l] = (unsigned short)at;
            at += (int)t.arc[l];
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < arcs; j += ORIENT_THREADS) t.apos[j] = (unsigned short)(t.apos[j] + t.start[source(j)]);
    __syncthreads();
    for (int j = threadIdx.x; j < arcs; j += ORIENT_THREADS) {
        const int head = source(j ^ 1), end = head + 1 < np ? t.start[head + 1] : arcs;
        unsigned next = t.apos[j ^ 1] + 1u;
        if ((int)next == end) next = t.minp[tail_root(t, head)] == t.pid[head] ? TAIL_NIL : t.start[head];
        t.arc[t.apos[j]] = 1u << 16 | next;
    }
    __syncthreads();
    int r = 0;
    for (;;) {
        unsigned w[T::pieces / ORIENT_THREADS];
        bool more = false;
#pragma unroll
        for (int q = 0; q < T::pieces / ORIENT_THREADS; ++q) {
            const int i = q * ORIENT_THREADS + threadIdx.x;
            w[q] = i < arcs ? t.arc[i] : TAIL_NIL;
            if ((w[q] & 0xFFFFu) != TAIL_NIL) {
                const unsigned o = t.arc[w[q] & 0xFFFFu];
                w[q] = (w[q] & 0xFFFF0000u) + (o & 0xFFFF0000u) | (o & 0xFFFFu);
                more = true;
            }
        }
        if (!__syncthreads_or(more) || ++r > MAX_ROUNDS) return r;
#pragma unroll
        for (int q = 0; q < T::pieces / ORIENT_THREADS; ++q) {
            const int i = q * ORIENT_THREADS + threadIdx.x;
            if (i < arcs) t.arc[i] = w[q];
        }
        __syncthreads();
    }
}

// Results of one oriented edge: child piece p of edge k takes its attach point
// and new root (as in orient_one) and its path is reversed.  Returns the
// vertices reversed.
__device__ __forceinline__ int tail_out(Ctl *ctl, const OrientArgs &oa, long long e, u64 k, int p, int root,
                                        unsigned ep) {
    const int x0 = (int)klo(k), x1 = (int)khi(k);
    const bool low = oa.rep[x0] == p;
    const int x = low ? x0 : x1, y = low ? x1 : x0;
    oa.chx[e] = x;
    oa.chy[e] = y;
    oa.att_x[p] = x;
    oa.att_ep[p] = ep;
    oa.newrep[p] = root;
    oa.rep_ep[p] = ep;
    if (oa.aff_ep[p] == ep) ctl->need_root = 1;
    return oa.walk ? walk_path(ctl, oa.parent, x, y, oa.long_ep, p, ep) : 0;
}

template <class T>
__device__ void replace_small(Ctl *ctl, const HookArgs &h, const OrientArgs &oa, int c0, int pre, unsigned ep) {
    extern __shared__ __align__(16) int s_rank[];
    T &t = *reinterpret_cast<T *>(s_rank);
    constexpr int IT = T::cand / ORIENT_THREADS;   // candidates per thread
    const int lane = threadIdx.x & 31;
    const int all = c0 + pre;
    for (int i = threadIdx.x; i < T::slots; i += ORIENT_THREADS) t.hk[i] = -1;
    if (threadIdx.x == 0) t.ner = 0;
    __syncthreads();
    u64 key[IT];
    int ra[IT], rb[IT];
    bool alive[IT];
#pragma unroll
    for (int q = 0; q < IT; ++q) {
        const int i = q * ORIENT_THREADS + threadIdx.x;
        alive[q] = i < all;
        key[q] = 0;
        ra[q] = rb[q] = 0;
        if (!alive[q]) continue;
        key[q] = i < pre ? LD(h.er[i]) : LD(h.ck[0][i - pre]);
        if (pre) {
            ra[q] = oa.rep[klo(key[q])];
            rb[q] = oa.rep[khi(key[q])];
        } else {
            ra[q] = LD(h.ca[0][i]);
            rb[q] = LD(h.cb[0][i]);
        }
    }
#pragma unroll
    for (int q = 0; q < IT; ++q) {
        if (alive[q]) {
            ra[q] = tail_slot(t, ra[q]);
            rb[q] = tail_slot(t, rb[q]);
        }
    }
    __syncthreads();
    // dense ids in slot order
    int np;
    {
        constexpr int HT = T::slots / ORIENT_THREADS;
        const int s0 = threadIdx.x * HT;
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < HT; ++q) cnt += t.hk[s0 + q] != -1;
        long long tot;
        int l = (int)block_excl_scan_ll(cnt, &tot);
        np = (int)tot;
#pragma unroll
        for (int q = 0; q < HT; ++q) {
            if (t.hk[s0 + q] == -1) continue;
            t.hl[s0 + q] = (unsigned short)l;
            t.pid[l] = t.hk[s0 + q];
            t.comp[l] = (unsigned short)l;
            ++l;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < IT; ++q) {
        const int i = q * ORIENT_THREADS + threadIdx.x;
        if (alive[q]) {
            ra[q] = t.hl[ra[q]];
            rb[q] = t.hl[rb[q]];
            t.key[i] = key[q];
            t.a[i] = (unsigned short)ra[q];
            t.b[i] = (unsigned short)rb[q];
        }
    }
    __syncthreads();
    for (int l = threadIdx.x; l < np; l += ORIENT_THREADS) t.bhi[l] = t.blo[l] = 0xFFFFFFFFu;
    __syncthreads();
    // hook and compress (as in hook_rounds)
    int r = 0;
    for (; r < MAX_ROUNDS; ++r) {
        bool any = false;
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            if (!alive[q]) continue;
            ra[q] = tail_root(t, ra[q]);
            rb[q] = tail_root(t, rb[q]);
            alive[q] = ra[q] != rb[q];
            if (!alive[q]) continue;
            any = true;
            const unsigned hi = (unsigned)(key[q] >> 32);
            if (hi < *(volatile unsigned *)&t.bhi[ra[q]]) atomicMin(&t.bhi[ra[q]], hi);
            if (hi < *(volatile unsigned *)&t.bhi[rb[q]]) atomicMin(&t.bhi[rb[q]], hi);
        }
        if (!__syncthreads_or(any)) break;
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            if (!alive[q]) continue;
            const unsigned hi = (unsigned)(key[q] >> 32), lo = (unsigned)key[q];
            if (t.bhi[ra[q]] == hi) atomicMin(&t.blo[ra[q]], lo);
            if (t.bhi[rb[q]] == hi) atomicMin(&t.blo[rb[q]], lo);
        }
        __syncthreads();
        unsigned used = 0;
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            bool hook = false;
            if (alive[q]) {
                used |= 1u << q;
                const int a = ra[q], b = rb[q];
                const unsigned hi = (unsigned)(key[q] >> 32), lo = (unsigned)key[q];
                const bool ba = t.bhi[a] == hi && t.blo[a] == lo, bb = t.bhi[b] == hi && t.blo[b] == lo;
                if (ba && bb) t.comp[a > b ? a : b] = (unsigned short)(a > b ? b : a);
                else if (ba) t.comp[a] = (unsigned short)b;
                else if (bb) t.comp[b] = (unsigned short)a;
                hook = ba || bb;
                alive[q] = !hook;
            }
            const unsigned m = __ballot_sync(0xffffffffu, hook);
            if (!m) continue;
            int base = 0;
            if (lane == 0) base = atomicAdd(&t.ner, __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (hook) t.er[base + __popc(m & ((1u << lane) - 1u))] = (unsigned short)(q * ORIENT_THREADS + threadIdx.x);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < IT; ++q)
            if (used >> q & 1u) t.bhi[ra[q]] = t.bhi[rb[q]] = t.blo[ra[q]] = t.blo[rb[q]] = 0xFFFFFFFFu;
        __syncthreads();
    }
    __syncthreads();
    if (r >= MAX_ROUNDS && threadIdx.x == 0) atomicOr(&ctl->err, ERR_ROUNDS);
    // super-roots: the smallest piece of every super-tree
    const int ner = t.ner;
    for (int l = threadIdx.x; l < np; l += ORIENT_THREADS) {
        t.minp[l] = INT_MAX;
        t.vis[l] = 0;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < np; l += ORIENT_THREADS) {
        const int root = tail_root(t, l), p = t.pid[l];
        if (p < *(volatile int *)&t.minp[root]) atomicMin(&t.minp[root], p);
    }
    __syncthreads();
    for (int l = threadIdx.x; l < np; l += ORIENT_THREADS)
        if (t.minp[tail_root(t, l)] == t.pid[l]) t.vis[l] = 1;
    __syncthreads();
    // orientation: an edge with one visited end makes the other end its
    // child (every piece is reached over one edge only)
    int child[IT];
    bool open[IT];
#pragma unroll
    for (int q = 0; q < IT; ++q) {
        open[q] = q * ORIENT_THREADS + (int)threadIdx.x < ner;
        child[q] = -1;
    }
    bool deep = ner > 0;
    for (int lvl = 0; deep && lvl < TAIL_LEVELS; ++lvl) {
        bool more = false;
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            if (!open[q]) continue;
            const int i = t.er[q * ORIENT_THREADS + threadIdx.x];
            const int a = t.a[i], b = t.b[i];
            const bool va = *(volatile unsigned char *)&t.vis[a], vb = *(volatile unsigned char *)&t.vis[b];
            if (va == vb) {
                more = true;
                continue;
            }
            open[q] = false;
            child[q] = va ? b : a;
            t.vis[child[q]] = 1;
        }
        deep = __syncthreads_or(more);
    }
    if (deep) {
        const int rounds = tail_rank<T>(ner, np);
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            if (!open[q]) continue;
            const int e = q * ORIENT_THREADS + threadIdx.x, i = t.er[e];
            child[q] = t.arc[t.apos[2 * e]] >> 16 > t.arc[t.apos[2 * e + 1]] >> 16 ? t.b[i] : t.a[i];
        }
        if (threadIdx.x == 0) {
            if (rounds > MAX_ROUNDS) atomicOr(&ctl->err, ERR_ROUNDS);
            ctl->rank_rounds = rounds;
        }
    }
    int rev = 0;
#pragma unroll
    for (int q = 0; q < IT; ++q) {
        if (child[q] < 0) continue;
        const int e = q * ORIENT_THREADS + threadIdx.x;
        const u64 k = t.key[t.er[e]];
        const int p = t.pid[child[q]], root = t.minp[tail_root(t, child[q])];
        if (all <= SMALL_OUT) {
            rev += tail_out(ctl, oa, e, k, p, root, ep);
        } else {
            oa.er_out[e] = k;
            oa.ep[e] = p;
            oa.eid[e] = root;
        }
    }
    block_add(&ctl->reversed, rev);
    if (threadIdx.x == 0) {
        ctl->ner = (u64)ner;
        ctl->hook_rounds = r;
        ctl->ncore = deep ? 2 * (u64)ner : 0;
    }
}

// Replacement edges of a batch in one cooperative launch: the pair table is
// moved into the candidate list (h.pairs), the candidates are hooked, the
// replacement edges oriented and their paths walked.  Up to C candidates go to
// one block (replace_small); the other blocks then only pull
// the forest into L2 for its walks (and the representatives for the refresh
// that follows an insert) and take part in the results.  As launches of their
// own the pair compaction, hooking, orientation and walks of a 100-edge batch
// took 68 us on R-MAT scale 22.
template <int C>
__global__ void __launch_bounds__(ORIENT_THREADS, 1) k_replace(Ctl *ctl, HookArgs h, OrientArgs a) {
    if (batch_skipped(ctl)) return;
    __shared__ HotMin hm;
    const unsigned ep = ctl->epoch;
    if (gtid() == 0) {
        ctl->cnt[1] = ctl->cnt[2] = 0;
        ctl->flag[0] = ctl->flag[1] = ctl->flag[2] = 0;
    }
    if (h.pairs) {
        compact_pairs(ctl, h.pt, h.ck[0], h.ca[0], h.cb[0], h.cand_cap);
        if (!grid_barrier(ctl, &ctl->bar[1])) return;
    }
    const long long c0 = (long long)*(volatile u64 *)&ctl->ncand;
    const long long pre = (long long)ctl->npre;
    if (c0 + pre <= C) {
        if (c0 + pre == 0) return;
        if (blockIdx.x == 0) {
            replace_small<SmallTail<C>>(ctl, h, a, (int)c0, (int)pre, ep);
        } else {
            const long long t = gtid() - blockDim.x, nt = gstride() - blockDim.x;
            l2_prefetch(a.parent, 4 * a.n, t, nt);
            if (ctl->op == DRSF_INSERT) l2_prefetch(a.rep, 4 * a.n, t, nt);
        }
        if (c0 + pre <= SMALL_OUT) return;
        if (!grid_barrier(ctl, &ctl->bar[1])) return;
        const long long ner = (long long)*(volatile u64 *)&ctl->ner;
        int rev = 0;
        // (one warp of every block after another: few edges reach many SMs)
        for (long long w = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; w * 32 < ner;
             w += (long long)gridDim.x * (blockDim.x >> 5)) {
            const long long e = w * 32 + (threadIdx.x & 31);
            if (e < ner) rev += tail_out(ctl, a, e, LD(a.er_out[e]), LD(a.ep[e]), LD(a.eid[e]), ep);
        }
        block_add(&ctl->reversed, rev);
        return;
    }
    hm_init(hm);
    if (h.init) {
        hook_init(h, c0, ep);
        if (!grid_barrier(ctl, &ctl->bar[1])) return;
    }
    if (hook_all(ctl, hm, h, c0) < 0) return;
    if (!grid_barrier(ctl, &ctl->bar[1])) return;
    orient_grid(ctl, a);
}

// The walks as a launch of their own, for batches above LARGE_BATCH edges: one
// thread per replacement edge at full occupancy, where the orientation (one
// block per SM) would take them in several rounds.  For a 100K-edge batch the
// launch costs 10 us more than it saves (R-MAT scale 22).
__global__ void k_walk(Ctl *ctl, OrientArgs a) {
    if (batch_skipped(ctl)) return;
    const unsigned ep = ctl->epoch;
    const long long ner = (long long)ctl->ner;
    int rev = 0;
    GS_LOOP(i, ner) {
        const int x = a.chx[i];
        rev += walk_path(ctl, a.parent, x, a.chy[i], a.long_ep, a.rep[x], ep);
    }
    block_add(&ctl->reversed, rev);
}

// Path-reversal set-up fused with the representative refresh: every vertex
// of a merged piece takes the super-tree's root as its new rep; with `marks`
// a vertex of a piece that is reversed through the marks (selected in
// sel_ep, re-rooted at an attach point x != its root) is active (its old
// parent is saved, J0 seeded, x marked).
// IP items per thread and iteration (IPT over a list or few vertices, IPN
// over many), k-major as in k_aff_collect, one slot reservation per block.
// Only the pieces stay in registers; the few items whose piece changed are
// handled from bit masks (the common item costs one stamp gather).  With DENSE
// many change, and their new representatives are loaded side by side.
template <int IP, bool DENSE>
__device__ __forceinline__ void refresh_pass(Ctl *ctl, const FinishArgs &a, const int *L, long long cnt, unsigned ep,
                                             bool marks) {
    static_assert(IP <= 32, "item masks are 32 bits");
    const long long step = (long long)gridDim.x * blockDim.x * IP;
    for (long long b0 = (long long)blockIdx.x * blockDim.x * IP; b0 < cnt; b0 += step) {
        const long long i0 = b0 + threadIdx.x;
        int p[IP];
        if (L) {
#pragma unroll
            for (int k = 0; k < IP; ++k) {
                const long long i = i0 + (long long)k * blockDim.x;
                p[k] = i < cnt ? L[i] : 0;
            }
#pragma unroll
            for (int k = 0; k < IP; ++k) p[k] = i0 + (long long)k * blockDim.x < cnt ? a.rep[p[k]] : 0;
        } else {
#pragma unroll
            for (int k = 0; k < IP; ++k) {
                const long long i = i0 + (long long)k * blockDim.x;
                p[k] = i < cnt ? a.rep[i] : 0;
            }
        }
        // the pieces selected for the marks are re-rooted child pieces, all
        // of which get a new representative: one gather in the common case
        unsigned chg = 0;
#pragma unroll
        for (int k = 0; k < IP; ++k)
            if (i0 + (long long)k * blockDim.x < cnt && a.rep_ep[p[k]] == ep) chg |= 1u << k;
        unsigned on = 0;
        long long q = 0;
        int nr[DENSE ? IP : 1];
        if (DENSE) {
#pragma unroll
            for (int k = 0; k < IP; ++k) nr[k] = chg >> k & 1u ? a.newrep[p[k]] : 0;
        }
        if (marks) {   // (the same value in every thread)
            if (DENSE) {
#pragma unroll
                for (int k = 0; k < IP; ++k)
                    if ((chg >> k & 1u) && LD(a.sel_ep[p[k]]) == ep) on |= 1u << k;
                for (unsigned m = on; m; m &= m - 1) {
                    const int k = __ffs(m) - 1;
                    if (a.att_x[p[k]] == p[k]) on &= ~(1u << k);
                }
            } else {
                for (unsigned m = chg; m; m &= m - 1) {
                    const int k = __ffs(m) - 1;
                    const int pk = p[k];
                    if (LD(a.sel_ep[pk]) == ep && a.att_x[pk] != pk) on |= 1u << k;
                }
            }
            q = block_reserve(&ctl->nact, __popc(on));
        }
        if (DENSE) {
#pragma unroll
            for (int k = 0; k < IP; ++k) {
                const long long i = i0 + (long long)k * blockDim.x;
                if (chg >> k & 1u) a.rep[L ? L[i] : (int)i] = nr[k];
            }
        }
        for (unsigned m = DENSE ? on : chg; m; m &= m - 1) {
            const int k = __ffs(m) - 1;
            const int pk = p[k];
            const long long i = i0 + (long long)k * blockDim.x;
            const int v = L ? L[i] : (int)i;
            if ((on >> k) & 1u) {
                const int pv = LD(a.parent[v]);
                a.act[q] = v;
                a.pold[q] = pv;
                a.J0[v] = pv;
                a.mark[v] = v == a.att_x[pk];
                a.aidx[v] = (int)q;   // dense index (Euler-tour marks)
                a.aroot[q] = pk;      // the piece root
                ++q;
            }
            if (!DENSE) a.rep[v] = a.newrep[pk];
        }
    }
}

// Mark every ancestor of each attach point x inside its piece by pointer
// doubling over the active vertices: round j, a marked v marks J_j[v] (its
// 2^j-th ancestor, clamped at the root) and J_{j+1} = J_j o J_j.  After
// round j the marks cover distances [0, 2^{j+1}); the loop stops once every
// J_{j+1} is a root, which bounds the path length.  Marks only ever land on
// ancestors of x, so reads racing with writes within a round are harmless.
// Returns false when a grid barrier gave up or the rounds ran out.
__device__ bool mark_paths(Ctl *ctl, const FinishArgs &a, long long na) {
    int *Jc = a.J0, *Jn = a.J1;
    int r = 0;
    for (;; ++r) {
        if (r >= MAX_ROUNDS) {
            if (gtid() == 0) atomicOr(&ctl->err, ERR_ROUNDS);
            return false;
        }
        if (gtid() == 0) ctl->flag[(r + 1) % 3] = 0;
        bool more = false;
        const long long S = gstride();
        for (long long base = gtid(); base < na; base += S * JU) {
            int v[JU], w[JU], w2[JU];
            bool ok[JU];
            unsigned char mk[JU];
#pragma unroll
            for (int k = 0; k < JU; ++k) {
                long long i = base + k * S;
                ok[k] = i < na;
                v[k] = ok[k] ? LD(a.act[i]) : 0;
            }
#pragma unroll
            for (int k = 0; k < JU; ++k) {
                w[k] = ok[k] ? LD(Jc[v[k]]) : 0;
                mk[k] = ok[k] ? LD(a.mark[v[k]]) : 0;
            }
#pragma unroll
            for (int k = 0; k < JU; ++k) w2[k] = ok[k] ? LD(Jc[w[k]]) : 0;
#pragma unroll
            for (int k = 0; k < JU; ++k) {
                if (!ok[k]) continue;
                if (mk[k]) a.mark[w[k]] = 1;
                Jn[v[k]] = w2[k];
                more |= LD(a.parent[w2[k]]) != w2[k];
            }
        }
        if (__syncthreads_or(more) && threadIdx.x == 0) atomicOr(&ctl->flag[r % 3], 1);
        if (!grid_barrier(ctl, &ctl->bar[3])) return false;
        int again = *(volatile int *)&ctl->flag[r % 3];
        int *t = Jc; Jc = Jn; Jn = t;
        if (!again) break;
    }
    if (gtid() == 0) ctl->mark_rounds = r + 1;
    return true;
}

// ReversePaths + attach (Algorithm 1): for each marked non-root vertex u,
// parent'[old parent of u] = u (old parents come from the saved snapshot, so
// no thread reads a pointer another thread rewrites); then parent[x] = y for
// every oriented replacement edge x -> y.
__device__ __forceinline__ void reverse_marked(Ctl *ctl, const FinishArgs &a, long long na) {
    const long long ner = (long long)ctl->ner;
    long long c = 0;
    GS_LOOP(i, na) {
        const int v = LD(a.act[i]);
        const int p = LD(a.pold[i]);
        if (LD(a.mark[v]) && p != v) {
            a.parent[p] = v;
            ++c;
        }
    }
    block_add(&ctl->reversed, c);
    GS_LOOP(i, ner) a.parent[a.chx[i]] = a.chy[i];
}

// End of a batch: the representative refresh, and, when some walk was too
// long (ctl->nlong), the doubling marks and the reversal of those pieces, in
// one cooperative launch: without long walks (the common case) it is one
// pass and no grid barrier, where two launches that found nothing to do cost
// 10 us of every batch.  A top-down delete passes over the list of its
// detached vertices, unless it re-rooted a tree's root piece (need_root);
// the other batches pass over all vertices.  With a.euler the marks are the
// Euler tour's (a launch of its own) and k_reverse follows it.
__global__ void __launch_bounds__(BLK, 5) k_finish(Ctl *ctl, FinishArgs a) {
    if (batch_skipped(ctl)) return;
    const unsigned ep = ctl->epoch;
    if (ctl->ner == 0) return;   // no piece was merged
    const bool marks = a.euler || *(volatile int *)&ctl->nlong;
    if (ctl->op == DRSF_DELETE && ctl->td && !*(volatile int *)&ctl->need_root)
        refresh_pass<IPT, true>(ctl, a, a.A, (long long)ctl->naff, ep, marks);
    else if (a.n <= gstride() * IPT)
        refresh_pass<IPT, false>(ctl, a, nullptr, a.n, ep, marks);
    else if (ctl->op == DRSF_DELETE)
        refresh_pass<IPD, true>(ctl, a, nullptr, a.n, ep, marks);
    else
        refresh_pass<IPN, false>(ctl, a, nullptr, a.n, ep, marks);
    if (a.euler || !marks) return;
    if (!grid_barrier(ctl, &ctl->bar[3])) return;
    const long long na = (long long)*(volatile u64 *)&ctl->nact;
    if (na == 0) return;
    if (!mark_paths(ctl, a, na)) return;
    reverse_marked(ctl, a, na);
}
__global__ void k_reverse(Ctl *ctl, FinishArgs a) {
    if (batch_skipped(ctl)) return;
    reverse_marked(ctl, a, (long long)ctl->nact);
}

// Component labels: smallest vertex id per tree (drsf_labels).
__global__ void k_label_init(int n, int *tmp) {
    GS_LOOP(v, n) tmp[v] = INT_MAX;
}
__global__ void k_label_min(int n, const int *rep, int *tmp) {
    GS_LOOP(v, n) {
        int r = rep[v];
        unsigned same = __match_any_sync(__activemask(), r);
        // lanes hold increasing v: the lowest lane of each group has the minimum
        if ((threadIdx.x & 31) == __ffs(same) - 1) atomicMin(&tmp[r], (int)v);
    }
}
__global__ void k_label_out(int n, const int *rep, const int *tmp, int *out) {
    GS_LOOP(v, n) out[v] = tmp[rep[v]];
}

// Failure-detection self-test: block 1 never arrives at the barrier, so
// block 0's bounded wait runs out, latches ERR_TIMEOUT and returns.
__global__ void k_barrier_selftest(Ctl *ctl) {
    if (blockIdx.x != 0) return;
    grid_barrier(ctl, &ctl->bar[0]);
}

// ------------------------------------------------------------- wrappers

static unsigned gsz(long long n) { return grid_for(n, BLK, 152u * 16u); }

static unsigned coop_blocks(const void *fn, int nsm, int cap_per_sm) {
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, BLK, 0) != cudaSuccess || per < 1) per = 1;
    if (per > cap_per_sm) per = cap_per_sm;
    return (unsigned)(per * nsm);
}
// The vertex passes (k_aff_collect, k_finish) loop over their range with
// the blocks that are resident at once: no partial last wave.
unsigned grid_vertex_pass(int nsm) { return coop_blocks((const void *)k_aff_collect, nsm, 8); }
unsigned coop_blocks_relabel(int nsm) { return coop_blocks((const void *)k_relabel, nsm, 8); }
unsigned coop_blocks_finish(int nsm) { return coop_blocks((const void *)k_finish, nsm, 8); }
unsigned coop_blocks_jump(int nsm) {
    const unsigned a = coop_blocks((const void *)k_jump<0>, nsm, 8), b = coop_blocks((const void *)k_jump<1>, nsm, 8);
    return a < b ? a : b;
}
template <int C>
static constexpr int replace_smem(int arcs) {
    return (int)sizeof(SmallTail<C>) > 16 * arcs ? (int)sizeof(SmallTail<C>) : 16 * arcs;
}
unsigned coop_blocks_replace(int nsm) {
    cudaFuncSetAttribute((const void *)k_replace<SMALL_CAND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         replace_smem<SMALL_CAND>(RANK_ARCS));
    cudaFuncSetAttribute((const void *)k_replace<SMALL_CAND_LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         replace_smem<SMALL_CAND_LARGE>(RANK_ARCS_LARGE));
    return (unsigned)nsm;   // one block per SM (threads and registers)
}

cudaError_t launch_begin(Ctl *ctl, BeginArgs a, long long grid_len, cudaStream_t s) {
    k_begin<<<gsz(grid_len), BLK, 0, s>>>(ctl, a);
    return cudaGetLastError();
}
cudaError_t set_begin(cudaGraphExec_t exec, cudaGraphNode_t node, Ctl *ctl, BeginArgs a, long long grid_len) {
    void *args[] = {(void *)&ctl, (void *)&a};
    cudaKernelNodeParams p = {};
    p.func = (void *)k_begin;
    p.gridDim = dim3(gsz(grid_len));
    p.blockDim = dim3(BLK);
    p.kernelParams = args;
    return cudaGraphExecKernelNodeSetParams(exec, node, &p);
}
cudaError_t launch_aff_collect(const Dev &d, int n, const int *rep, const unsigned *aff_ep, int *A, int *rold,
                               unsigned *w, u64 *heavy, Ctl *ctl, cudaStream_t s) {
    k_aff_collect<<<d.grid_pass, BLK, 0, s>>>(n, rep, aff_ep, A, rold, w, heavy, ctl);
    return cudaGetLastError();
}
cudaError_t launch_cross(const Dev &d, Ctl *ctl, DetachArgs da, RelabelArgs ra, RowList rl, LightArgs la, bool sg,
                         cudaStream_t s) {
    void *args[] = {(void *)&ctl, (void *)&da, (void *)&ra, (void *)&rl, (void *)&la};
    return cudaLaunchCooperativeKernel(sg ? (const void *)k_cross<true> : (const void *)k_cross<false>,
                                       d.few ? (unsigned)d.nsm : d.coop_cross, BLK, args, 0, s);
}
unsigned coop_blocks_cross(int nsm) {
    const unsigned a = coop_blocks((const void *)k_cross<true>, nsm, 4), b = coop_blocks((const void *)k_cross<false>, nsm, 4);
    return a < b ? a : b;
}
cudaError_t launch_scan(const Dev &d, Ctl *ctl, RowList rl, LightArgs a, bool sg, cudaStream_t s) {
    void *args[] = {(void *)&ctl, (void *)&rl, (void *)&a};
    return cudaLaunchCooperativeKernel(sg ? (const void *)k_scan<true> : (const void *)k_scan<false>, d.grid_scan, BLK,
                                       args, 0, s);
}
// The blocks that are resident at once (grid barriers; the row list's tiles
// are dealt out in equal shares).
unsigned scan_grid(int nsm) {
    int per = 8;
    for (const void *fn : {(const void *)k_scan<true>, (const void *)k_scan<false>}) {
        int o = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, BLK, 0) != cudaSuccess || o < 1) o = 1;
        if (o < per) per = o;
    }
    return (unsigned)(per * nsm);
}
cudaError_t launch_relabel(const Dev &d, Ctl *ctl, RelabelArgs a, cudaStream_t s) {
    void *args[] = {(void *)&ctl, (void *)&a};
    return cudaLaunchCooperativeKernel((const void *)k_relabel, d.coop_relabel, BLK, args, 0, s);
}
cudaError_t launch_jump(const Dev &d, const int *A, int use_list, long long cnt_static, Ctl *ctl, const int *par,
                        int *J, int *J1, int *rep, RowList rl, int mode, const int *rold, unsigned *w, u64 *heavy,
                        Csr g, int sync_rounds, int *X, int *Y, const int *cuts, cudaStream_t s) {
    void *args[] = {(void *)&A,    (void *)&use_list, (void *)&cnt_static, (void *)&ctl, (void *)&par,
                    (void *)&J,    (void *)&J1,       (void *)&rep,        (void *)&rl,  (void *)&mode,
                    (void *)&rold, (void *)&w,        (void *)&heavy,      (void *)&g,   (void *)&X,
                    (void *)&Y,    (void *)&cuts};
    const void *fn = sync_rounds ? (const void *)k_jump<1> : (const void *)k_jump<0>;
    return cudaLaunchCooperativeKernel(fn, d.coop_jump, BLK, args, 0, s);
}
cudaError_t launch_replace(const Dev &d, Ctl *ctl, HookArgs h, OrientArgs a, bool large, cudaStream_t s) {
    static_assert(replace_smem<SMALL_CAND>(RANK_ARCS) <= 225 * 1024, "one block's shared memory");
    a.rank_arcs = large ? RANK_ARCS_LARGE : RANK_ARCS;
    void *args[] = {(void *)&ctl, (void *)&h, (void *)&a};
    return large ? cudaLaunchCooperativeKernel((const void *)k_replace<SMALL_CAND_LARGE>, d.coop_replace,
                                               ORIENT_THREADS, args, replace_smem<SMALL_CAND_LARGE>(RANK_ARCS_LARGE), s)
                 : cudaLaunchCooperativeKernel((const void *)k_replace<SMALL_CAND>, d.coop_replace, ORIENT_THREADS, args,
                                               replace_smem<SMALL_CAND>(RANK_ARCS), s);
}
cudaError_t launch_walk(const Dev &d, Ctl *ctl, OrientArgs a, cudaStream_t s) {
    k_walk<<<d.grid, BLK, 0, s>>>(ctl, a);
    return cudaGetLastError();
}
cudaError_t launch_finish(const Dev &d, Ctl *ctl, FinishArgs a, cudaStream_t s) {
    void *args[] = {(void *)&ctl, (void *)&a};
    return cudaLaunchCooperativeKernel((const void *)k_finish, d.few ? (unsigned)d.nsm : d.coop_finish, BLK, args, 0, s);
}
cudaError_t launch_reverse(const Dev &d, Ctl *ctl, FinishArgs a, cudaStream_t s) {
    k_reverse<<<d.grid, BLK, 0, s>>>(ctl, a);
    return cudaGetLastError();
}
cudaError_t launch_labels(int n, const int *rep, int *tmp, int *out, cudaStream_t s) {
    k_label_init<<<gsz(n), BLK, 0, s>>>(n, tmp);
    k_label_min<<<gsz(n), BLK, 0, s>>>(n, rep, tmp);
    k_label_out<<<gsz(n), BLK, 0, s>>>(n, rep, tmp, out);
    return cudaGetLastError();
}
cudaError_t launch_barrier_selftest(Ctl *ctl, cudaStream_t s) {
    void *args[] = {(void *)&ctl};
    return cudaLaunchCooperativeKernel((const void *)k_barrier_selftest, 2, 32, args, 0, s);
}

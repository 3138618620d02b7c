// Cross-edge scans of a delete batch: over a list of rows (after a top-down
// search), and over the rows of all detached vertices with the first hooking
// round taken from them (after a root search over all vertices).
#pragma once

#include "kernels.h"

// Delete, cross-edge scan (key edges M = E(G) - E(F) - B, Algorithm 1,
// restricted).  The rows of the listed vertices (every vertex outside the
// piece left out of its cut tree) are flattened by the prefix sum roff and
// cut into tiles of 32 entries, whatever rows they fall in (load balanced:
// a hub row is spread over many warps, short rows share a tile); each warp
// takes a contiguous range of tiles.  For a tile the warp loads the list
// entries of the 32 rows starting at the tile's first row (one coalesced
// load per field) and lane e takes its row's fields from the lane that
// loaded them, so an entry costs one column load and one rep gather.  A
// live neighbour x of u in another piece gives the cross edge {u, x}; every
// cross edge has a listed endpoint and, when both are listed, the smaller
// id emits it.  Parallel edges between two pieces are reduced to the one
// with the minimum key, which is the only one that can be in the minimum
// spanning forest: lanes holding the same piece pair take the minimum
// first, then one lane updates the pair table.  A pair that finds no table
// slot is emitted as a plain candidate.  This reduction is the supergraph
// variant's super-edge dedupe (SG, Section III-A); with SG false (HS,
// Section III-B) every cross edge is emitted as a candidate of the hooking.
// Entry positions are below 2^32, so the tile arithmetic is 32-bit.
template <bool SG>
__device__ __forceinline__ void scan_rows(const RowList &rl, Ctl *ctl, const Csr &g, const int *rep,
                                          const PairTable &pt, u64 *ck, int *ca, int *cb, u64 cand_cap) {
    const unsigned nd = (unsigned)ctl->ndet;
    if (nd == 0) return;
    const unsigned E = rl.roff[nd];
    const unsigned NT = (E + 31) >> 5;
    const int lane = threadIdx.x & 31;
    const unsigned warp = (unsigned)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const unsigned nw = (unsigned)((gridDim.x * blockDim.x) >> 5);
    if (warp == 0 && lane == 0) atomicAdd((u64 *)&ctl->scanned, (u64)E);
    const unsigned per = (NT + nw - 1) / nw;
    const unsigned t_lo = warp * per, t_hi = t_lo + per < NT ? t_lo + per : NT;
    // the pair this lane updated last, its table slot and the minimum key
    // seen for it since: a hub row repeats one piece pair over many tiles,
    // so its minimum is kept in a register and written to the table once
    // when the pair changes (no probe, and no stream of atomics on one
    // slot from every tile of the row)
    u64 cpair = EMPTY_KEY, cslot = 0, cmin = EMPTY_KEY;
    for (unsigned T = t_lo; T < t_hi; ++T) {
        const unsigned t0 = T << 5;
        // window: rows r0 .. r0+31 from the tile's first row
        const unsigned wr = (unsigned)rl.tile[T] + lane;
        const bool wok = wr < nd;
        const unsigned wv = wok ? rl.roff[wr] : 0xFFFFFFFFu;
        const int wu = wok ? rl.D[wr] : 0;
        const unsigned wb = wok ? rl.base[wr] : 0;
        const int2 wm = wok ? rl.meta[wr] : make_int2(0, 0);
        // the rows after the first that start inside this tile set a bit at
        // their start position (a row that starts before the tile wraps to
        // a large offset); the row of position p is the first row plus the
        // number of such starts at positions <= p
        const unsigned pos = wv - t0;
        const unsigned bit = (lane > 0 && pos < 32) ? (1u << pos) : 0u;
        const unsigned starts = __reduce_or_sync(0xffffffffu, bit);
        const int c = __popc(starts & (lane == 31 ? 0xffffffffu : ((2u << lane) - 1u)));
        // all lanes take part in the shuffles
        const unsigned rstart = __shfl_sync(0xffffffffu, wv, c);
        const int u = __shfl_sync(0xffffffffu, wu, c);
        const unsigned rb = __shfl_sync(0xffffffffu, wb, c);
        const int ru = __shfl_sync(0xffffffffu, wm.x, c);
        const int hp = __shfl_sync(0xffffffffu, wm.y, c);
        const unsigned e = t0 + lane;
        const int x = e < E ? __ldcs(&g.col[(size_t)(rb + (e - rstart))]) : -1;
        const int rx = x >= 0 ? rep[x] : 0;
        const bool emit = x >= 0 && rx != ru && (rx == hp || u < x);
        const unsigned m = __ballot_sync(0xffffffffu, emit);
        if (!m) continue;
        bool raw = false;
        u64 key = 0;
        if (!SG) {
            raw = emit;
            key = ekey((uint32_t)u, (uint32_t)x);
        } else if (emit) {
            // one piece pair for the whole warp is the common case (a hub
            // row against one other piece): no match needed then
            const int ld = __ffs(m) - 1;
            const int lru = __shfl_sync(m, ru, ld), lrx = __shfl_sync(m, rx, ld);
            const unsigned grp = __all_sync(m, ru == lru && rx == lrx)
                                     ? m
                                     : __match_any_sync(m, ((u64)(unsigned)ru << 32) | (unsigned)rx);
            key = group_min_u64(grp, ekey((uint32_t)u, (uint32_t)x));
            if (lane == __ffs(grp) - 1) {
                const u64 pair = ru < rx ? ((u64)(unsigned)ru << 32) | (unsigned)rx
                                         : ((u64)(unsigned)rx << 32) | (unsigned)ru;
                if (pair == cpair) {
                    cmin = key < cmin ? key : cmin;
                } else {
                    const long long sl = pair_slot(pt.pk, pt.mask, pair);
                    if (sl >= 0) {
                        if (cpair != EMPTY_KEY) atomicMin(&pt.mk[cslot], cmin);
                        cpair = pair;
                        cslot = (u64)sl;
                        cmin = key;
                    } else {
                        raw = true;
                    }
                }
            }
        }
        const long long p = agg_append(&ctl->ncand, raw);
        if (raw) {
            if ((u64)p < cand_cap) {
                ck[p] = key;
                ca[p] = ru;
                cb[p] = rx;
            } else {
                atomicOr(&ctl->err, ERR_CAPACITY);
            }
        }
    }
    if (SG && cpair != EMPTY_KEY) atomicMin(&pt.mk[cslot], cmin);
}

// Delete, cross-edge scan of the overflow list (edges outside their rows),
// through the same pair table (SG) or straight to the candidates (HS).
template <bool SG>
__device__ __forceinline__ void scan_ovf(const u64 *ovf, Ctl *ctl, const int *rep, const PairTable &pt, u64 *ck,
                                         int *ca, int *cb, u64 cand_cap) {
    long long no = (long long)ctl->ovf_count;
    GS_LOOP(i, no) {
        u64 k = ovf[i];
        bool raw = false;
        int ra = -1, rb = -1;
        if (k != TOMB_KEY) {
            ra = rep[klo(k)];
            rb = rep[khi(k)];
            if (ra != rb) raw = !SG || !pair_min(pt.pk, pt.mk, pt.mask, ra, rb, k);
        }
        long long p = agg_append(&ctl->ncand, raw);
        if (raw) {
            if ((u64)p < cand_cap) {
                ck[p] = k;
                ca[p] = ra;
                cb[p] = rb;
            } else {
                atomicOr(&ctl->err, ERR_CAPACITY);
            }
        }
    }
}

// Delete after a root search over all vertices (large batches): hook-and-
// compress whose first round is taken from the rows themselves.
//   1. Every listed row (vertices outside the piece left out of their tree)
//      gives its piece the smallest key of its cross edges: a minimum in
//      registers, one check or atomic per row.  No candidate is written.
//   2. Every scanned piece hooks along its minimum edge (a mutual choice hooks
//      the larger root under the smaller): replacement edges.  By the cut
//      property each is one whatever the other pieces do, so the piece left
//      out, whose rows are not read, need not choose.
//   3. The hook forest of the pieces is flattened and the rows of every
//      component without the piece left out are read once more (on R-MAT most
//      pieces hang under that one by now; where most do not, after a second
//      round from the rows): the cross edges that still join two
//      components are the candidates of the rounds that follow (k_replace),
//      reduced per pair of components through the pair table (SG) or one by
//      one (HS).
// A batch that detaches much of a graph has more pairs of pieces than the pair
// table (or a hash table of any size that fits L2) can take.  Few of them are
// left after the first round: a window of 1M-edge batches over R-MAT scale 20
// (W below; its deletes cut 480K tree edges, 4.1M pairs) took 1,410 us to scan
// and 1,120 to hook with every cross edge as a candidate, and takes 435 and 322
// with all that is said here.
//
// A lane reads a row of up to LONG_ROW entries by itself, LU entries in flight
// (flattening the rows of a warp by a prefix sum and reading 32 entries per
// step took twice the instructions even on R-MAT rows, and the grid's scan
// 520 us instead of 290); longer rows become jobs of JOB_LEN entries, dealt
// out to all warps.
#define LONG_ROW 32
#define JOB_LEN 128
#define LU 8
#define FLAT_WALK 16
// what a pass over the rows does: step 1's minima per piece, a further round's
// minima per component, or the candidates left
enum { FIND = 0, AGAIN = 1, EMIT = 2 };
__device__ __forceinline__ void piece_min(u64 *best, int p, u64 k) {
    if (k < __ldcg(&best[p])) atomicMin(&best[p], k);
}
// A row as its lane or warp holds it while earlier rows are read.
struct LightRow {
    int v, p;          // vertex (-1: none) and piece
    unsigned st;       // first slot
    int used;
    int lp, cp;        // step 1: the piece left out; step 3: its component and the row's
    u64 best;          // step 1: the piece's minimum when the row was loaded
};
__device__ __forceinline__ void light_head(const LightArgs &a, LightRow &r, int v) {
    r.v = v;
    r.p = v >= 0 ? __ldcg(&a.rep[v]) : 0;
    const int2 h = v >= 0 ? __ldcg(reinterpret_cast<const int2 *>(&a.g.row[v])) : make_int2(0, 0);
    r.st = (unsigned)h.x;
    r.used = h.y;
}
// Step 1 skips the piece left out, step 3 its whole component: another
// component's cross edges are all in its own rows.
template <int MODE>
__device__ __forceinline__ void light_piece(const LightArgs &a, LightRow &r) {
    r.lp = r.cp = 0;
    r.best = EMPTY_KEY;
    if (r.v < 0) return;
    r.lp = a.left[r.p];
    r.cp = r.p;
    if (MODE != FIND) {
        r.cp = __ldcg(&a.comp[r.p]);
        r.lp = __ldcg(&a.comp[r.lp]);
    }
    if (MODE != EMIT) r.best = __ldcg(&a.best[r.cp]);
    if (r.cp == r.lp) r.used = 0;
}
// A cross edge of step 3, seen from component cv: appended to the candidates
// unless the pair table takes it (all lanes call; `raw`: the lane has one).
template <bool SG>
__device__ __forceinline__ void light_emit(Ctl *ctl, const LightArgs &a, bool raw, u64 key, int cv, int cx) {
    if (SG && raw) raw = !pair_min(a.pt.pk, a.pt.mk, a.pt.mask, cv, cx, key);
    if (!__any_sync(0xffffffffu, raw)) return;
    const long long q = agg_append(&ctl->ncand, raw);
    if (!raw) return;
    if ((u64)q < a.cand_cap) {
        a.ck[q] = key;
        a.ca[q] = cv;
        a.cb[q] = cx;
    } else {
        atomicOr(&ctl->err, ERR_CAPACITY);
    }
}
// Entries at, at + step, ... (LU of them, below `used`) of row r: the minimum of
// their cross edges, or (EMIT) they are emitted.
template <int MODE, bool SG>
__device__ __forceinline__ u64 light_entries(Ctl *ctl, const LightArgs &a, const LightRow &r, int at, int step) {
    int x[LU], rx[LU];
    u64 k = EMPTY_KEY;
#pragma unroll
    for (int u = 0; u < LU; ++u) x[u] = at + u * step < r.used ? a.g.col[(size_t)r.st + at + u * step] : -1;
#pragma unroll
    for (int u = 0; u < LU; ++u) rx[u] = x[u] >= 0 ? a.rep[x[u]] : r.p;
    if (MODE == FIND) {
#pragma unroll
        for (int u = 0; u < LU; ++u) {
            const u64 key = ekey((uint32_t)r.v, (uint32_t)x[u]);
            if (rx[u] != r.p && key < k) k = key;
        }
    } else if (MODE == AGAIN) {
#pragma unroll
        for (int u = 0; u < LU; ++u) rx[u] = rx[u] != r.p ? __ldcg(&a.comp[rx[u]]) : r.cp;
#pragma unroll
        for (int u = 0; u < LU; ++u) {
            const u64 key = ekey((uint32_t)r.v, (uint32_t)x[u]);
            if (rx[u] != r.cp && key < k) k = key;
        }
    } else {
#pragma unroll
        for (int u = 0; u < LU; ++u) {
            if (!__any_sync(0xffffffffu, rx[u] != r.p)) continue;
            const int cx = rx[u] != r.p ? __ldcg(&a.comp[rx[u]]) : r.cp;
            const bool raw = cx != r.cp && (cx == r.lp || r.v < x[u]);
            light_emit<SG>(ctl, a, raw, ekey((uint32_t)r.v, (uint32_t)x[u]), r.cp, cx);
        }
    }
    return k;
}

// One pass over the listed rows and the overflow edges (step 1 or 3).  Step 1
// keeps which rows have a cross edge, one bit each, and step 3 reads only
// those again (in the 4096 x 4096 grid's pieces a third; with `again`, the
// list of those that are in no component of a piece left out).  Vertex, piece
// and row head, and what the piece says are loaded up to three rows ahead.
template <int MODE, bool SG>
__device__ __forceinline__ bool light_pass(Ctl *ctl, const LightArgs &a, long long nd, u64 *bar, bool again) {
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    long long read = 0;
    const long long nb = (nd + 31) >> 5;
    auto vertex = [&](long long b) {
        if (b >= nb || b * 32 + lane >= nd) return -1;
        if (MODE == FIND) return __ldcg(&a.D[b * 32 + lane]);
        if (again) return __ldcg(&a.root[b * 32 + lane]);
        return __ldcg(&a.rows[b]) >> lane & 1u ? __ldcg(&a.D[b * 32 + lane]) : -1;
    };
    LightRow r0, r1;
    light_head(a, r0, vertex(warp));
    light_piece<MODE>(a, r0);
    light_head(a, r1, vertex(warp + nw));
    int v2 = vertex(warp + 2 * nw);
    for (long long b = warp; b < nb; b += nw) {
        const int v3 = vertex(b + 3 * nw);
        LightRow r2;
        light_head(a, r2, v2);
        light_piece<MODE>(a, r1);
        const bool big = r0.used > LONG_ROW;
        if (MODE == FIND) {
            read += r0.used;
            unsigned bm = __ballot_sync(0xffffffffu, big);
            if (bm) {
                const int jobs = big ? (r0.used + JOB_LEN - 1) / JOB_LEN : 0;
                int inc = jobs;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += y;
                }
                int base = 0;
                if (lane == 31) base = atomicAdd(&ctl->njobs, inc);
                base = __shfl_sync(0xffffffffu, base, 31) + inc - jobs;
                if (jobs == 1) *reinterpret_cast<int2 *>(&a.job[2 * (size_t)base]) = make_int2(r0.v, 0);
                bm = __ballot_sync(0xffffffffu, jobs > 1);
                while (bm) {   // the whole warp writes a longer row's jobs
                    const int l = __ffs(bm) - 1;
                    bm &= bm - 1;
                    const int j0 = __shfl_sync(0xffffffffu, base, l), nj = __shfl_sync(0xffffffffu, jobs, l);
                    const int jv = __shfl_sync(0xffffffffu, r0.v, l);
                    for (int t = lane; t < nj; t += 32)
                        *reinterpret_cast<int2 *>(&a.job[2 * (size_t)(j0 + t)]) = make_int2(jv, t);
                }
            }
        }
        if (big) r0.used = 0;
        const int most = __reduce_max_sync(0xffffffffu, r0.used);
        u64 k = EMPTY_KEY;
        for (int at = 0; at < most; at += LU) {
            const u64 e = light_entries<MODE, SG>(ctl, a, r0, at, 1);
            k = e < k ? e : k;
        }
        if (MODE != EMIT) {
            const bool hit = k != EMPTY_KEY;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (MODE == FIND && lane == 0) a.rows[b] = m;
            if (m) {
                // rows of one piece combine first (a large piece's rows fill warps)
                const int p0 = __shfl_sync(0xffffffffu, r0.cp, __ffs(m) - 1);
                if (__all_sync(0xffffffffu, !hit || r0.cp == p0)) {
                    k = group_min_u64(0xffffffffu, k);
                    if (lane == __ffs(m) - 1 && k < r0.best) atomicMin(&a.best[p0], k);
                } else if (hit && k < r0.best) {
                    atomicMin(&a.best[r0.cp], k);
                }
            }
        }
        r0 = r1;
        r1 = r2;
        v2 = v3;
    }
    if (MODE == FIND && !grid_barrier(ctl, bar)) return false;   // the jobs are all listed
    const long long nj = *(volatile int *)&ctl->njobs;
    auto job = [&](long long t) {
        return t < nj ? __ldcg(reinterpret_cast<const int2 *>(&a.job[2 * t])) : make_int2(-1, 0);
    };
    int2 j0 = job(warp), j1 = job(warp + nw);
    light_head(a, r0, j0.x);
    for (long long t = warp; t < nj; t += nw) {
        const int2 j2 = job(t + 2 * nw);
        light_piece<MODE>(a, r0);
        light_head(a, r1, j1.x);
        const int at = j0.y * JOB_LEN;
        r0.used = min(r0.used, at + JOB_LEN);
        u64 k = EMPTY_KEY;
        for (int i = at; i < r0.used; i += 32 * LU) {
            const u64 e = light_entries<MODE, SG>(ctl, a, r0, i + lane, 32);
            k = e < k ? e : k;
        }
        if (MODE != EMIT) {
            k = group_min_u64(0xffffffffu, k);
            if (lane == 0 && k < r0.best) atomicMin(&a.best[r0.cp], k);
        }
        r0 = r1;
        j0 = j1;
        j1 = j2;
    }
    if (MODE == FIND) block_add(&ctl->scanned, read);
    // edges held outside the rows
    const long long no = (long long)ctl->ovf_count;
    const long long S = (long long)gridDim.x * blockDim.x;
    for (long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; i0 < no; i0 += S) {
        const u64 k = i0 + lane < no ? a.ovf[i0 + lane] : TOMB_KEY;
        int ra = 0, rb = 0;
        if (k != TOMB_KEY) {
            ra = __ldcg(&a.rep[klo(k)]);
            rb = __ldcg(&a.rep[khi(k)]);
        }
        if (MODE == FIND) {
            if (ra == rb) continue;
            // (the piece left out does not choose: its minimum stays empty)
            const int l = a.left[ra];
            if (ra != l) piece_min(a.best, ra, k);
            if (rb != l) piece_min(a.best, rb, k);
        } else {
            const int ca = ra != rb ? __ldcg(&a.comp[ra]) : 0, cb = ra != rb ? __ldcg(&a.comp[rb]) : 0;
            if (MODE == EMIT) {
                light_emit<SG>(ctl, a, ca != cb, k, ca, cb);
            } else if (ca != cb) {
                const int l = __ldcg(&a.comp[a.left[ra]]);
                if (ca != l) piece_min(a.best, ca, k);
                if (cb != l) piece_min(a.best, cb, k);
            }
        }
    }
    return true;
}

// Step 2 for piece q: hooks it along its minimum edge; true (and the key) when
// that is a replacement edge of its own.
__device__ __forceinline__ bool light_hook(const LightArgs &a, int q, u64 *key) {
    const u64 k = __ldcg(&a.best[q]);
    if (k == EMPTY_KEY) return false;
    const int pa = __ldcg(&a.rep[klo(k)]), pb = __ldcg(&a.rep[khi(k)]);
    const int o = pa == q ? pb : pa;
    if (__ldcg(&a.best[o]) == k && q < o) return false;   // o hooks under q
    a.comp[q] = o;
    *key = k;
    return true;
}

// Lists the rows that step 3 reads: those with a cross edge whose component
// does not hold the piece left out.  From AGAIN_MIN rows on: few rows of many
// are left (one in ten of those with a cross edge in the 4096 x 4096 grid), and
// a warp that met one of them among its 32 read it alone.  Scan, us, without and
// with the list: the grid 404 and 348, the 256-graph union 635 and 521, W 554
// and 524.  A shorter list keeps too few blocks busy: R-MAT scale 22 with 98K
// rows 71 and 88, 179K 103 and 119, 378K 172 and 180; scale 20 with 434K 189 and
// 196; but 64 graphs with 464K rows 141 and 130: the line lies about here.
#define AGAIN_MIN (1 << 19)
// From so many listed rows on, a quarter of all or more, a second round is taken
// from them, not only the first: most of the graph is in components without the
// piece left out, and their pairs would fill the pair table (R-MAT scale 20
// after ten batches of 1M deletes, half of them tree edges, which W is not:
// 2.5M candidates; scan and hooking 1,400 + 1,320 us, 1,002 + 359 with the
// round).  With fewer rows the
// reading costs more than the candidates it saves: at 2^17 the 256-graph
// union's scan and hooking took 584 + 310 us instead of 521 + 337, the grid's
// (one row in twenty left) 503 + 185 instead of 347 + 223.
#define ROUND_MIN (1 << 19)
__device__ __forceinline__ void list_again(Ctl *ctl, const LightArgs &a, long long nd, u64 *count) {
    const long long step = (long long)blockDim.x * LU;
    for (long long b0 = blockIdx.x * step; b0 < nd; b0 += gridDim.x * step) {
        int v[LU], p[LU], l[LU], cp[LU];
        unsigned in = 0;
#pragma unroll
        for (int u = 0; u < LU; ++u) {
            const long long i = b0 + u * blockDim.x + threadIdx.x;
            v[u] = i < nd && (__ldcg(&a.rows[i >> 5]) >> (i & 31) & 1u) ? __ldcg(&a.D[i]) : -1;
        }
#pragma unroll
        for (int u = 0; u < LU; ++u) p[u] = v[u] >= 0 ? __ldcg(&a.rep[v[u]]) : -1;
#pragma unroll
        for (int u = 0; u < LU; ++u) {
            l[u] = p[u] >= 0 ? a.left[p[u]] : -1;
            cp[u] = p[u] >= 0 ? __ldcg(&a.comp[p[u]]) : -1;
        }
#pragma unroll
        for (int u = 0; u < LU; ++u)
            if (p[u] >= 0 && __ldcg(&a.comp[l[u]]) != cp[u]) in |= 1u << u;
        long long q = block_reserve(count, __popc(in));
#pragma unroll
        for (int u = 0; u < LU; ++u)
            if (in >> u & 1u) a.root[q++] = v[u];
    }
}

// The same in a further round, for component q: comp keeps the hooked ones
// complemented until a barrier (the others go on asking which component a
// piece is in: a complemented piece is the root of its own).
__device__ __forceinline__ int light_component(const LightArgs &a, int p) {
    const int c = __ldcg(&a.comp[p]);
    return c < 0 ? p : c;
}
__device__ __forceinline__ bool light_hook_again(const LightArgs &a, int q, u64 *key) {
    const u64 k = __ldcg(&a.best[q]);
    if (k == EMPTY_KEY || __ldcg(&a.comp[q]) != q) return false;
    const int pa = light_component(a, __ldcg(&a.rep[klo(k)])), pb = light_component(a, __ldcg(&a.rep[khi(k)]));
    const int o = pa == q ? pb : pa;
    if (__ldcg(&a.best[o]) == k && q < o) return false;
    a.comp[q] = ~o;
    *key = k;
    return true;
}

// Hooks every scanned piece (or, AGAIN, every component of them) along its
// minimum edge: the cut vertices' pieces and, where a detached piece is left
// out in its place, the root piece, by the thread that meets the one left out
// (a cut vertex like the others; when every cut asked its old root's stamp, all
// warps went to one sector).  Block-uniform loop: the edges are appended per
// block.
template <int MODE>
__device__ __forceinline__ void hook_pieces(Ctl *ctl, const LightArgs &a, long long nc) {
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < nc; b0 += (long long)gridDim.x * blockDim.x) {
        const long long i = b0 + threadIdx.x;
        bool h1 = false, h2 = false;
        u64 k1 = 0, k2 = 0;
        if (i < nc) {
            const int c = a.cuts[i], r = a.rold[c], l = a.left[r];
            if (MODE == FIND) {
                if (c != l) h1 = light_hook(a, c, &k1);
                else h2 = light_hook(a, r, &k2);
            } else {
                h1 = light_hook_again(a, c, &k1);
                if (c == l) h2 = light_hook_again(a, r, &k2);
            }
        }
        const long long q1 = block_append(&ctl->ner, h1);
        if (h1) a.er[q1] = k1;
        if (__syncthreads_or(h2)) {
            const long long q2 = block_append(&ctl->ner, h2);
            if (h2) a.er[q2] = k2;
        }
    }
}

// Flattens the hook forest: every piece's root is found by a walk that writes
// nothing (a path of more than FLAT_WALK steps is halved as it is walked) and
// kept aside; after a barrier it is stored.  (Walks that halved every path, and
// stores of roots beside walks that were still reading, made each other's
// loads miss: W, 480K pieces, paths of at most 6 steps: the whole scan 694 us
// so, 545 in this way.)
__device__ __forceinline__ bool flatten_pieces(Ctl *ctl, const LightArgs &a, long long nc, u64 *bar) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc; i += (long long)gridDim.x * blockDim.x) {
        int x = __ldcg(&a.comp[a.cuts[i]]);
        bool at = false;
        for (int h = 0; h < FLAT_WALK && !at; ++h) {
            const int p = __ldcg(&a.comp[x]);
            at = p == x;
            x = p;
        }
        a.root[i] = at ? x : find_root(a.comp, x, ctl);
    }
    if (!grid_barrier(ctl, bar)) return false;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc; i += (long long)gridDim.x * blockDim.x) {
        const int c = a.cuts[i], r = a.rold[c];
        a.comp[c] = a.root[i];
        if (c == a.left[r]) a.comp[r] = find_root_ro(a.comp, r, ctl);
    }
    return grid_barrier(ctl, bar);
}

// The scan of a row list (top-down deletes, selectable root searches).
template <bool SG>
__device__ __forceinline__ void scan_listed(Ctl *ctl, const RowList &rl, const LightArgs &a) {
    scan_rows<SG>(rl, ctl, a.g, a.rep, a.pt, a.ck, a.ca, a.cb, a.cand_cap);
    scan_ovf<SG>(a.ovf, ctl, a.rep, a.pt, a.ck, a.ca, a.cb, a.cand_cap);
}

// Steps 1 to 3 above.
template <bool SG>
__device__ void scan_light(Ctl *ctl, const LightArgs &a) {
    const long long nc = (long long)ctl->ncut;
    if (nc == 0) return;   // no tree was cut
    const unsigned ep = ctl->epoch;
    u64 *bar = &ctl->bar[4];
    if (*(volatile int *)&ctl->flag[0]) {
        // some tree's root piece is scanned, a heavier one left out: list it
        // (LU vertices per thread, one reservation per block and iteration)
        const long long step = (long long)blockDim.x * LU;
        for (long long b0 = blockIdx.x * step; b0 < a.n; b0 += gridDim.x * step) {
            int p[LU];
            unsigned in = 0;
#pragma unroll
            for (int u = 0; u < LU; ++u) {
                const long long v = b0 + u * blockDim.x + threadIdx.x;
                p[u] = v < a.n ? a.rep[v] : -1;
            }
#pragma unroll
            for (int u = 0; u < LU; ++u)
                if (p[u] >= 0 && a.aff_ep[p[u]] == ep && a.left[p[u]] != p[u]) in |= 1u << u;
            long long q = block_reserve(&ctl->ndet, __popc(in));
#pragma unroll
            for (int u = 0; u < LU; ++u)
                if (in >> u & 1u) a.D[q++] = (int)(b0 + u * blockDim.x + threadIdx.x);
        }
        if (!grid_barrier(ctl, bar)) return;
    }
    const long long nd = (long long)*(volatile u64 *)&ctl->ndet;
    if (!light_pass<FIND, SG>(ctl, a, nd, bar, false)) return;
    if (!grid_barrier(ctl, bar)) return;
    hook_pieces<FIND>(ctl, a, nc);
    if (!grid_barrier(ctl, bar)) return;
    if (nd < AGAIN_MIN) {
        if (!flatten_pieces(ctl, a, nc, bar)) return;
        light_pass<EMIT, SG>(ctl, a, nd, bar, false);
    } else {
        if (!flatten_pieces(ctl, a, nc, bar)) return;
        list_again(ctl, a, nd, &ctl->nagain[0]);
        if (!grid_barrier(ctl, bar)) return;
        long long na = (long long)*(volatile u64 *)&ctl->nagain[0];
        if (na >= ROUND_MIN && na >= nd / 4) {
            // another round from the rows: minima per component, which hook
            for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
                 i += (long long)gridDim.x * blockDim.x) {
                const int c = a.cuts[i], r = a.rold[c];
                a.best[c] = EMPTY_KEY;
                if (c == a.left[r]) a.best[r] = EMPTY_KEY;
            }
            if (!grid_barrier(ctl, bar)) return;
            if (!light_pass<AGAIN, SG>(ctl, a, na, bar, true) || !grid_barrier(ctl, bar)) return;
            hook_pieces<AGAIN>(ctl, a, nc);
            if (!grid_barrier(ctl, bar)) return;
            for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
                 i += (long long)gridDim.x * blockDim.x) {
                const int c = a.cuts[i], r = a.rold[c], x = __ldcg(&a.comp[c]);
                if (x < 0) a.comp[c] = ~x;
                if (c == a.left[r] && __ldcg(&a.comp[r]) < 0) a.comp[r] = ~__ldcg(&a.comp[r]);
            }
            if (!grid_barrier(ctl, bar) || !flatten_pieces(ctl, a, nc, bar)) return;
            list_again(ctl, a, nd, &ctl->nagain[1]);
            if (!grid_barrier(ctl, bar)) return;
            na = (long long)*(volatile u64 *)&ctl->nagain[1];
        }
        light_pass<EMIT, SG>(ctl, a, na, bar, true);
    }
    // (every hooking round ended at a barrier: the count is final)
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->npre = *(volatile u64 *)&ctl->ner;
}

// Graph storage kernels: slack CSR + edge index build, batch normalisation,
// insertion and deletion of the batch ("Insert/Delete B of edges to/from G",
// Algorithm 1), and the cross-edge scans that produce the candidate set
// (key edges with rep[u] != rep[v], Section II-A).
#include <climits>

#include "kernels.h"

#define GS_LOOP(i, n) \
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)(n); \
         i += (long long)gridDim.x * blockDim.x)

// Warp-aggregated counter increment.
__device__ __forceinline__ void agg_count(long long *ctr, bool pred, long long sign = 1) {
    unsigned m = __ballot_sync(__activemask(), pred);
    if (m && (threadIdx.x & 31) == __ffs(m) - 1 && pred)
        atomicAdd((u64 *)ctr, (u64)(sign * (long long)__popc(m)));
}

// ------------------------------------------------------------------ build

__global__ void k_check_range(const int *a, long long cnt, int n, int *bad) {
    GS_LOOP(i, cnt) {
        int x = a[i];
        if (x < 0 || x >= n) atomicOr(bad, 1);
    }
}

// Deduplicate the input edge list through the index; winners are appended.
__global__ void k_create_claim(const int *edges, long long m, Index ix, u64 *dkey, u64 *dslot, u64 *cnt,
                               long long *self_loops) {
    GS_LOOP(i, m) {
        int u = edges[2 * i], v = edges[2 * i + 1];
        bool keep = false;
        u64 key = 0;
        long long s = -1;
        if (u != v) {
            key = ekey((uint32_t)u, (uint32_t)v);
            bool reused = false;
            s = index_claim(ix, key, &reused);
            keep = s >= 0;
        }
        agg_count(self_loops, u == v);
        long long p = agg_append(cnt, keep);
        if (keep) {
            dkey[p] = key;
            dslot[p] = (u64)s;
        }
    }
}

// Row degrees; each edge keeps the places that it takes in its two rows.
__global__ void k_degree(const u64 *dkey, long long m, int *deg, int2 *place) {
    GS_LOOP(i, m) {
        const u64 k = dkey[i];
        place[i] = make_int2(atomicAdd(&deg[klo(k)], 1), atomicAdd(&deg[khi(k)], 1));
    }
}

// Row capacity: degree plus max(4, degree / 4) free slots.
__global__ void k_caps(const int *deg, int n, long long *cap) {
    GS_LOOP(u, n) {
        int d = deg[u];
        int slack = d / 4 > 4 ? d / 4 : 4;
        cap[u] = (long long)d + slack;
    }
}

// Exclusive scan of int64: tiles of SCAN_TILE elements.
#define SCAN_ITEMS 16
#define SCAN_TILE (BLK * SCAN_ITEMS)

__device__ long long block_excl_scan_i64(long long v, long long *total) {
    __shared__ long long ws[BLK / 32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        long long t = lane < BLK / 32 ? ws[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < BLK / 32) ws[lane] = t;
    }
    __syncthreads();
    long long pre = (w > 0 ? ws[w - 1] : 0) + x - v;
    *total = ws[BLK / 32 - 1];
    __syncthreads();
    return pre;
}

__global__ void k_scan_tiles(const long long *in, long long n, long long *bsum) {
    long long base = (long long)blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_ITEMS;
    long long s = 0;
    for (int j = 0; j < SCAN_ITEMS; ++j)
        if (base + j < n) s += in[base + j];
    long long tot;
    block_excl_scan_i64(s, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_sums(long long *bsum, long long nb) {
    // one block: exclusive scan of nb block sums in place
    long long per = (nb + BLK - 1) / BLK;
    long long lo = threadIdx.x * per, hi = lo + per < nb ? lo + per : nb;
    long long s = 0;
    for (long long i = lo; i < hi; ++i) s += bsum[i];
    long long tot;
    long long pre = block_excl_scan_i64(s, &tot);
    for (long long i = lo; i < hi; ++i) {
        long long t = bsum[i];
        bsum[i] = pre;
        pre += t;
    }
}

__global__ void k_scan_apply(const long long *in, long long *out, long long n, const long long *bsum) {
    long long base = (long long)blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_ITEMS;
    long long s = 0;
    for (int j = 0; j < SCAN_ITEMS; ++j)
        if (base + j < n) s += in[base + j];
    long long tot;
    long long pre = block_excl_scan_i64(s, &tot) + bsum[blockIdx.x];
    for (int j = 0; j < SCAN_ITEMS; ++j)
        if (base + j < n) {
            out[base + j] = pre;
            pre += in[base + j];
        }
    if (base <= n - 1 && base + SCAN_ITEMS > n - 1) out[n] = pre;   // total after the last element
}

// Row heads of a new CSR: the slots past a row's degree are free (row n
// closes the array).
__global__ void k_rows_init(const long long *off, const int *deg, int n, Row *row) {
    GS_LOOP(u, (long long)n + 1) {
        const int cap = u < n ? (int)(off[u + 1] - off[u]) : 0, d = u < n ? deg[u] : 0;
        row[u] = Row{(unsigned)off[u], d, cap - d, cap};
    }
}

// Place the deduplicated edges at the places taken in k_degree, record
// their positions.
__global__ void k_fill(const u64 *dkey, const u64 *dslot, const int2 *place, long long m, Csr g, Index ix) {
    GS_LOOP(i, m) {
        u64 k = dkey[i];
        uint32_t a = klo(k), b = khi(k);
        const int2 pl = place[i];
        const unsigned qa = g.row[a].start + (unsigned)pl.x, qb = g.row[b].start + (unsigned)pl.y;
        g.col[qa] = (int)b;
        g.col[qb] = (int)a;
        ix.e[dslot[i]].pos = make_uint2(qa, qb);
    }
}

// ------------------------------------------------------------ per batch

// Insert, step 1 (batch normalisation): drop self-loops, repeated pairs and
// edges already in G; claim an index slot for each new edge.
__global__ void k_ins_claim(Index ix, Ctl *ctl, u64 *nkey, u64 *nslot) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->base = ctl->epoch;
    if (batch_skipped(ctl)) return;
    const int *batch = ctl->batch;
    const long long len = ctl->batch_len;
    // block-uniform loop: counters and the list append are aggregated per
    // block (one atomic per block instead of one per warp)
    long long loops = 0, drops = 0, reuse = 0;
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < len; b0 += (long long)gridDim.x * blockDim.x) {
        const long long i = b0 + threadIdx.x;
        bool keep = false;
        u64 key = 0;
        long long s = -1;
        if (i < len) {
            int u = batch[2 * i], v = batch[2 * i + 1];
            if (u != v) {
                key = ekey((uint32_t)u, (uint32_t)v);
                bool reused = false;
                s = index_claim(ix, key, &reused);
                if (s == LLONG_MIN) atomicOr(&ctl->err, ERR_CAPACITY);
                keep = s >= 0;
                reuse += reused;
                drops += !keep;
            } else {
                ++loops;
            }
        }
        long long p = block_append(&ctl->nb, keep);
        if (keep) {
            nkey[p] = key;
            nslot[p] = (u64)s;
        }
    }
    block_add(&ctl->self_loops, loops);
    block_add(&ctl->dropped, drops);
    block_add(&ctl->htomb, -reuse);
}

// Insert, step 2, for the edge of every calling thread with `on` (key k, index
// slot s; the whole block calls): a free slot of both CSR rows (row_take), or,
// when one of them is full, whole to the overflow list (Ovf).  The cross test of the
// insert case (M = B, Algorithm 1) is fused here: rep[u] != rep[v] makes a
// candidate.  With SG (the supergraph variant, Section III-A) a candidate goes
// into the pair table instead, which keeps the minimum key per pair of trees
// (one super-edge per pair; k_replace then lists them); without it (HS,
// Section III-B) every cross edge is a candidate of the hooking.  `slots`: set
// up the candidates' hook-forest slots too, so that the hooking needs no
// initialisation phase of its own (few candidates are hooked in shared
// memory).  *dead: change of the slots that scans read and hold no entry.
template <bool SG>
__device__ __forceinline__ void place_edge(bool on, u64 k, u64 s, const PlaceArgs &p, Ctl *ctl, unsigned ep, bool slots,
                                           long long *dead) {
    bool cross = false, over = false;
    unsigned held = POS_OVF;
    int ra = 0, rb = 0;
    if (on) {
        const uint32_t a = klo(k), b = khi(k);
        const Row ha = row_head(p.g, (int)a), hb = row_head(p.g, (int)b);
        const int pa = row_take(p.g, (int)a, ha, dead), pb = row_take(p.g, (int)b, hb, dead);
        if (pa >= 0 && pb >= 0) {
            const unsigned qa = ha.start + (unsigned)pa, qb = hb.start + (unsigned)pb;
            p.g.col[qa] = (int)b;
            p.g.col[qb] = (int)a;
            p.ix.e[s].pos = make_uint2(qa, qb);
            *dead -= 2;
        } else {
            over = true;
            held = pa >= 0 ? ha.start + (unsigned)pa : (pb >= 0 ? hb.start + (unsigned)pb : POS_OVF);
        }
        ra = p.rep[a];
        rb = p.rep[b];
        cross = ra != rb;
        if (SG && cross) cross = !pair_min(p.pt.pk, p.pt.mk, p.pt.mask, ra, rb, k);   // no slot: plain candidate
    }
    // (asked for per block: a million-edge batch can overflow 100K rows)
    if (__syncthreads_or(over)) {
        const long long o = ovf_take_block(ctl, p.ovf, over);
        if (over) {
            if ((u64)o < p.ovf.cap) {
                p.ovf.e[o] = k;
                p.ovf.pos[o] = held;
                p.ix.e[s].pos = make_uint2(POS_OVF, (uint32_t)o);
            } else {
                atomicOr(&ctl->err, ERR_CAPACITY);
            }
        }
    }
    const long long q = block_append(&ctl->ncand, cross);
    if (cross) {
        if ((u64)q < p.cand_cap) {
            p.ck[q] = k;
            p.ca[q] = ra;
            p.cb[q] = rb;
            if (!SG && slots) {
                hook_slot_init(p.hs, ra, ep);
                hook_slot_init(p.hs, rb, ep);
            }
        } else {
            atomicOr(&ctl->err, ERR_CAPACITY);
        }
    }
}

template <bool SG>
__global__ void k_ins_place(const u64 *nkey, const u64 *nslot, Ctl *ctl, PlaceArgs p) {
    if (batch_skipped(ctl)) return;
    const unsigned ep = ctl->epoch;
    const long long nb = (long long)ctl->nb;
    long long dead = 0;
    // block-uniform loop: the candidate append is aggregated per block
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < nb; b0 += (long long)gridDim.x * blockDim.x) {
        const long long i = b0 + threadIdx.x;
        const bool on = i < nb;
        place_edge<SG>(on, on ? nkey[i] : 0, on ? nslot[i] : 0, p, ctl, ep, nb > p.small, &dead);
    }
    block_add(&ctl->ctomb, dead);
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd((u64 *)&ctl->edges, (u64)nb);
}

// Both insert steps in one launch, for batches up to SMALL_INSERT edges: an
// edge is placed by the thread that claimed it, without the list of kept edges
// and the launch between.  Small batches are bound by launches and by the chain
// of loads: an insert and a delete of 100 edges in 4M vertices took 122 us
// with two launches and 117 with one, 10K edges 223 and 217, 100K edges 401
// and 397.  Larger batches are bound by the sectors they touch: the compacted
// list keeps every lane of the placing busy, and the 256-graph union's batch
// of 1.5M edges took longer in one launch.
template <bool SG>
__global__ void k_ins_small(Ctl *ctl, PlaceArgs p) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->base = ctl->epoch;
    if (batch_skipped(ctl)) return;
    const unsigned ep = ctl->epoch;
    const int *batch = ctl->batch;
    const long long len = ctl->batch_len;
    long long loops = 0, drops = 0, reuse = 0, kept = 0, dead = 0;
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < len; b0 += (long long)gridDim.x * blockDim.x) {
        const long long i = b0 + threadIdx.x;
        bool keep = false;
        u64 key = 0;
        long long s = -1;
        if (i < len) {
            const int u = batch[2 * i], v = batch[2 * i + 1];
            if (u != v) {
                key = ekey((uint32_t)u, (uint32_t)v);
                bool reused = false;
                s = index_claim(p.ix, key, &reused);
                if (s == LLONG_MIN) atomicOr(&ctl->err, ERR_CAPACITY);
                keep = s >= 0;
                reuse += reused;
                drops += !keep;
            } else {
                ++loops;
            }
        }
        kept += keep;
        place_edge<SG>(keep, key, (u64)s, p, ctl, ep, len > p.small, &dead);
    }
    block_add(&ctl->self_loops, loops);
    block_add(&ctl->dropped, drops);
    block_add(&ctl->htomb, -reuse);
    block_add((long long *)&ctl->nb, kept);
    block_add(&ctl->edges, kept);
    block_add(&ctl->ctomb, dead);
}

// Delete, step 1: normalisation (absent edges and repeats dropped), removal
// from the index and the CSR, and the tree-edge cut of Algorithm 1: for a
// deleted edge {u, v} with parent[u] == v, parent[u] <- u (either
// orientation).  The old root of a cut tree is stamped "affected"; the cut
// vertex becomes a piece root.
__global__ void k_del_claim(Index ix, Csr g, Ovf ovf, int *parent, const int *rep, Ctl *ctl, PieceSlots ps,
                            int *cutlist) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->base = ctl->epoch;
    if (batch_skipped(ctl)) return;
    const int *batch = ctl->batch;
    const long long len = ctl->batch_len;
    unsigned ep = ctl->epoch;
    // block-uniform loop: counters and the cut list append are aggregated
    // per block (one atomic per block instead of one per warp)
    long long loops = 0, drops = 0, wins = 0, dead = 0;
    const bool early = len <= 1 << 16;
    for (long long b0 = (long long)blockIdx.x * blockDim.x; b0 < len; b0 += (long long)gridDim.x * blockDim.x) {
        const long long i = b0 + threadIdx.x;
        int c = -1, rc = -1;
        if (i < len) {
            int u = batch[2 * i], v = batch[2 * i + 1];
            bool won = false;
            if (u != v) {
                // loaded up front, beside the index probe: parent[u] changes in
                // this kernel only by the cut of the edge {u, parent[u]}, which
                // only the thread deleting that edge makes
                const int par_u = parent[u], par_v = parent[v];
                // (the old root is needed for cuts only: large batches, bound
                // by the sectors they touch, load it then)
                const int rep_u = early ? rep[u] : 0, rep_v = early ? rep[v] : 0;
                const unsigned st_u = g.row[u].start, st_v = g.row[v].start;
                u64 key = ekey((uint32_t)u, (uint32_t)v);
                uint2 pos;
                long long s = index_find(ix, key, &pos);
                if (s >= 0) won = atomicCAS(&ix.e[s].key, key, TOMB_KEY) == key;
                if (won) {
                    if (pos.x == POS_OVF) {
                        ovf_give(ctl, ovf, g, pos.y, u, v);
                    } else {
                        row_give2(g, u, st_u, u < v ? pos.x : pos.y, v, st_v, u < v ? pos.y : pos.x);
                        dead += 2;
                    }
                    if (par_u == v) {
                        c = u;
                        rc = early ? rep_u : rep[u];
                    } else if (par_v == u) {
                        c = v;
                        rc = early ? rep_v : rep[v];
                    }
                    if (c >= 0) {   // c roots a new piece
                        parent[c] = c;
                        ps.rold[c] = rc;
                        ps.w[c] = 0;
                        ps.comp[c] = c;
                        ps.best[c] = EMPTY_KEY;
                    }
                }
                wins += won;
                drops += !won;
            } else {
                ++loops;
            }
        }
        {
            // stamp the cut trees' old roots; lanes cutting the same tree
            // write once (most cuts can fall in one giant tree)
            int r = rc;
            unsigned m = __ballot_sync(0xffffffffu, c >= 0);
            if (c >= 0) {
                unsigned grp = __match_any_sync(m, r);
                if ((int)(threadIdx.x & 31) == __ffs(grp) - 1 && __ldcg(&ps.aff_ep[r]) != ep) {
                    ps.aff_ep[r] = ep;
                    ps.w[r] = ps.wsum[r] = 0;
                    ps.heavy[r] = 0;
                    ps.comp[r] = r;
                    ps.best[r] = EMPTY_KEY;
                }
            }
        }
        long long p = block_append(&ctl->ncut, c >= 0);
        if (c >= 0) cutlist[p] = c;
    }
    block_add(&ctl->self_loops, loops);
    block_add(&ctl->dropped, drops);
    block_add(&ctl->htomb, wins);
    block_add(&ctl->ctomb, dead);
    block_add(&ctl->edges, -wins);
    block_add((long long *)&ctl->nb, wins);
}

// Edge-list export (rebuild and drsf_export_edges): warp per row, pairs
// (u, x) with u < x, then the live overflow edges.
__global__ void k_extract(int n, Csr g, const u64 *ovf, const Ctl *ctl, int *out, long long cap, u64 *cnt,
                          int *bad) {
    int lane = threadIdx.x & 31;
    long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long u = warp; u < n; u += nw) {
        const long long o = g.row[u].start, used = g.row[u].used;
        for (long long j0 = 0; j0 < used; j0 += 32) {
            long long j = j0 + lane;
            int x = j < used ? g.col[o + j] : -1;
            bool emit = x > (int)u;
            long long p = agg_append(cnt, emit);
            if (emit) {
                if (p < cap) {
                    out[2 * p] = (int)u;
                    out[2 * p + 1] = x;
                } else {
                    atomicOr(bad, 1);
                }
            }
        }
    }
    long long no = (long long)ctl->ovf_count;
    GS_LOOP(i, no) {
        u64 k = ovf[i];
        bool emit = k != TOMB_KEY;
        long long p = agg_append(cnt, emit);
        if (emit) {
            if (p < cap) {
                out[2 * p] = (int)klo(k);
                out[2 * p + 1] = (int)khi(k);
            } else {
                atomicOr(bad, 1);
            }
        }
    }
}

// DRSF_VALIDATE: every parent pointer must be an edge of G.
__global__ void k_check_tree_edges(int n, const int *parent, Index ix, int *bad) {
    GS_LOOP(v, n) {
        int p = parent[v];
        uint2 pos;
        if (p != (int)v && index_find(ix, ekey((uint32_t)v, (uint32_t)p), &pos) < 0) atomicOr(bad, 2);
    }
}

// DRSF_VALIDATE: no edge of G joins two different trees (one root per
// component, given acyclic pointers along edges of G).
__global__ void k_check_cross(const int *pairs, long long m, const int *rep, int *bad) {
    GS_LOOP(i, m) {
        if (rep[pairs[2 * i]] != rep[pairs[2 * i + 1]]) atomicOr(bad, 4);
    }
}

// ------------------------------------------------------------- wrappers

static unsigned gsz(long long n) { return grid_for(n, BLK, 152u * 16u); }

cudaError_t launch_check_range(const int *a, long long cnt, int n, int *bad, cudaStream_t s) {
    k_check_range<<<gsz(cnt), BLK, 0, s>>>(a, cnt, n, bad);
    return cudaGetLastError();
}
cudaError_t launch_create_claim(const int *edges, long long m, Index ix, u64 *dkey, u64 *dslot, u64 *cnt,
                                long long *self_loops, cudaStream_t s) {
    k_create_claim<<<gsz(m), BLK, 0, s>>>(edges, m, ix, dkey, dslot, cnt, self_loops);
    return cudaGetLastError();
}
cudaError_t launch_degree(const u64 *dkey, long long m, int *deg, int2 *place, cudaStream_t s) {
    k_degree<<<gsz(m), BLK, 0, s>>>(dkey, m, deg, place);
    return cudaGetLastError();
}
cudaError_t launch_caps(const int *deg, int n, long long *cap, cudaStream_t s) {
    k_caps<<<gsz(n), BLK, 0, s>>>(deg, n, cap);
    return cudaGetLastError();
}
cudaError_t launch_scan_i64(const long long *in, long long *out, long long n, long long *bsum, cudaStream_t s) {
    long long tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (tiles < 1) tiles = 1;
    k_scan_tiles<<<(unsigned)tiles, BLK, 0, s>>>(in, n, bsum);
    k_scan_sums<<<1, BLK, 0, s>>>(bsum, tiles);
    k_scan_apply<<<(unsigned)tiles, BLK, 0, s>>>(in, out, n, bsum);
    return cudaGetLastError();
}
cudaError_t launch_rows_init(const long long *off, const int *deg, int n, Row *row, cudaStream_t s) {
    k_rows_init<<<gsz((long long)n + 1), BLK, 0, s>>>(off, deg, n, row);
    return cudaGetLastError();
}
cudaError_t launch_fill(const u64 *dkey, const u64 *dslot, const int2 *place, long long m, Csr g, Index ix,
                        cudaStream_t s) {
    k_fill<<<gsz(m), BLK, 0, s>>>(dkey, dslot, place, m, g, ix);
    return cudaGetLastError();
}
// The batch kernels read the batch and its length from the control block;
// `len` only sizes their grid (a captured launch sequence is keyed by it).
cudaError_t launch_ins_claim(long long len, Index ix, Ctl *ctl, u64 *nkey, u64 *nslot, cudaStream_t s) {
    k_ins_claim<<<gsz(len), BLK, 0, s>>>(ix, ctl, nkey, nslot);
    return cudaGetLastError();
}
cudaError_t launch_ins_place(const Dev &d, const u64 *nkey, const u64 *nslot, Ctl *ctl, PlaceArgs p, bool sg,
                             cudaStream_t s) {
    if (sg) k_ins_place<true><<<d.grid, BLK, 0, s>>>(nkey, nslot, ctl, p);
    else k_ins_place<false><<<d.grid, BLK, 0, s>>>(nkey, nslot, ctl, p);
    return cudaGetLastError();
}
cudaError_t launch_ins_small(long long len, Ctl *ctl, PlaceArgs p, bool sg, cudaStream_t s) {
    if (sg) k_ins_small<true><<<gsz(len), BLK, 0, s>>>(ctl, p);
    else k_ins_small<false><<<gsz(len), BLK, 0, s>>>(ctl, p);
    return cudaGetLastError();
}
cudaError_t launch_del_claim(long long len, Index ix, Csr g, Ovf ovf, int *parent, const int *rep, Ctl *ctl,
                             PieceSlots ps, int *cutlist, cudaStream_t s) {
    k_del_claim<<<gsz(len), BLK, 0, s>>>(ix, g, ovf, parent, rep, ctl, ps, cutlist);
    return cudaGetLastError();
}
cudaError_t launch_extract(const Dev &d, int n, Csr g, const u64 *ovf, u64 novf_max, Ctl *ctl, int *out,
                           long long cap, u64 *cnt, cudaStream_t s) {
    (void)novf_max;
    k_extract<<<d.grid, BLK, 0, s>>>(n, g, ovf, ctl, out, cap, cnt, (int *)(cnt + 1));
    return cudaGetLastError();
}
cudaError_t launch_check_tree_edges(int n, const int *parent, Index ix, int *bad, cudaStream_t s) {
    k_check_tree_edges<<<gsz(n), BLK, 0, s>>>(n, parent, ix, bad);
    return cudaGetLastError();
}
cudaError_t launch_check_cross(const int *pairs, long long m, const int *rep, int *bad, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    k_check_cross<<<gsz(m), BLK, 0, s>>>(pairs, m, rep, bad);
    return cudaGetLastError();
}

// Launch wrappers of the D-RSF kernels (host side).  Each wrapper enqueues
// on `s` and returns the launch status.
#pragma once

#include "common.cuh"

// Fixed launch shapes.
#define BLK 256
// batches with at most this many candidates are replaced and oriented by one
// block in shared memory: batches of up to 64K edges, and larger ones (which
// leave more of the SM's memory to L1)
#define SMALL_CAND 4096
#define SMALL_CAND_LARGE 2048

// graphs of at most this many vertices: a grid barrier of one block per SM
// takes 1.3 us, of four 2.5, and the passes are short
#define FEW_VERTICES (1 << 18)

struct Dev {
    int nsm;
    unsigned grid;        // grid-stride kernels: nsm * 8 blocks of BLK
    unsigned coop_jump;   // cooperative kernels: co-resident block counts
    unsigned coop_replace;
    unsigned coop_relabel;
    unsigned coop_finish;
    unsigned coop_bfs;
    unsigned coop_et;
    unsigned coop_cross;
    bool few;             // few vertices: one block per SM where blocks wait for each other
    unsigned grid_scan;   // row scan: the co-resident block count
    unsigned grid_pass;   // affected list: co-resident blocks
};

// graph.cu -------------------------------------------------------------
unsigned scan_grid(int nsm);
cudaError_t launch_check_range(const int *a, long long cnt, int n, int *bad, cudaStream_t s);
cudaError_t launch_create_claim(const int *edges, long long m, Index ix, u64 *dkey, u64 *dslot, u64 *cnt,
                                long long *self_loops, cudaStream_t s);
cudaError_t launch_degree(const u64 *dkey, long long m, int *deg, int2 *place, cudaStream_t s);
cudaError_t launch_caps(const int *deg, int n, long long *cap, cudaStream_t s);
cudaError_t launch_scan_i64(const long long *in, long long *out, long long n, long long *bsum, cudaStream_t s);
cudaError_t launch_rows_init(const long long *off, const int *deg, int n, Row *row, cudaStream_t s);
cudaError_t launch_fill(const u64 *dkey, const u64 *dslot, const int2 *place, long long m, Csr g, Index ix,
                        cudaStream_t s);
// (the batch kernels read the batch from the control block; len sizes the grid)

// Per-piece slots that a cut sets up: for the cut vertex and for its tree's
// old root (k_relabel, k_scan).
struct PieceSlots {
    unsigned *aff_ep;   // old roots of this batch's cut trees
    int *rold, *comp;
    u64 *best, *heavy;
    unsigned *w, *wsum;
};
cudaError_t launch_del_claim(long long len, Index ix, Csr g, Ovf ovf, int *parent, const int *rep, Ctl *ctl,
                             PieceSlots ps, int *cutlist, cudaStream_t s);
// The rows a delete batch scans for cross edges, one entry per listed
// vertex u: u itself, the exclusive prefix sum of the row lengths (roff[nd]
// = total), the row's start in the CSR, and (rep[u], piece left out of the
// scan in u's tree); and for each tile of 32 consecutive entries of the
// flattened rows, the row of its first entry.
struct RowList {
    int *D;
    unsigned *roff;   // entry counts and CSR positions are below 2^32
    unsigned *base;   // (checked at build)
    int2 *meta;
    int *tile;        // tile[T] = the row holding entry 32 T (tiles of 32 entries)
};
struct PairTable {
    u64 *pk;   // piece pair key, EMPTY_KEY when free
    u64 *mk;   // minimum edge key of the pair
    u64 mask;
};
// sg: supergraph variant (pair-table dedupe to one minimum-key edge per
// pair of trees), else every cross edge is a candidate (hooking variant)
cudaError_t launch_ins_claim(long long len, Index ix, Ctl *ctl, u64 *nkey, u64 *nslot, cudaStream_t s);
struct PlaceArgs {
    Csr g;
    Index ix;
    Ovf ovf;
    const int *rep;
    PairTable pt;
    u64 *ck;             // candidates
    int *ca, *cb;
    u64 cand_cap;
    HookSlots hs;
    int small;           // HS: the slots of more than this many candidates are set up (HookSlots)
};
cudaError_t launch_ins_place(const Dev &d, const u64 *nkey, const u64 *nslot, Ctl *ctl, PlaceArgs p, bool sg,
                             cudaStream_t s);
// claim and placement in one launch
#define SMALL_INSERT (1 << 18)
cudaError_t launch_ins_small(long long len, Ctl *ctl, PlaceArgs p, bool sg, cudaStream_t s);
struct LightArgs {
    int n;
    Csr g;
    const int *rep;
    const unsigned *aff_ep;   // old roots of the cut trees
    const int *rold, *left;   // per cut vertex: its tree's old root; per piece: the one left out in its tree
    unsigned *rows;           // per 32 listed rows: those with a cross edge
    int *D;                   // the vertices whose rows are read
    int *job;                 // long rows: vertex, part
    int *comp;                // hook forest of the pieces
    int *root;                // per cut vertex, while the hook forest is flattened: its root; then the rows
                              // read again
    u64 *best;                // per piece: its minimum cross edge
    const int *cuts;
    u64 *er;                  // replacement edges
    const u64 *ovf;
    PairTable pt;
    u64 *ck;                  // candidates left
    int *ca, *cb;
    u64 cand_cap;
    int listed;               // the rows come as a RowList (selectable root searches)
};
cudaError_t launch_scan(const Dev &d, Ctl *ctl, RowList rl, LightArgs a, bool sg, cudaStream_t s);
cudaError_t launch_extract(const Dev &d, int n, Csr g, const u64 *ovf, u64 novf_max, Ctl *ctl, int *out,
                           long long cap, u64 *cnt, cudaStream_t s);
cudaError_t launch_check_tree_edges(int n, const int *parent, Index ix, int *bad, cudaStream_t s);
cudaError_t launch_check_cross(const int *pairs, long long m, const int *rep, int *bad, cudaStream_t s);

// forest.cu ------------------------------------------------------------
struct BeginArgs {
    int op, n;
    long long len;
    const int *batch;
    StorageLimits lim;
    int groups;                    // graphs with a slice of the batch and a vertex range each; 0: none
    const long long *voff, *boff;  // their offsets (groups + 1)
};
// (grid_len sizes the grid)
cudaError_t launch_begin(Ctl *ctl, BeginArgs a, long long grid_len, cudaStream_t s);
// the same launch's node in an instantiated graph, for another batch
cudaError_t set_begin(cudaGraphExec_t exec, cudaGraphNode_t node, Ctl *ctl, BeginArgs a, long long grid_len);
cudaError_t launch_aff_collect(const Dev &d, int n, const int *rep, const unsigned *aff_ep, int *A, int *rold,
                               unsigned *w, u64 *heavy, Ctl *ctl, cudaStream_t s);
// delete: detached vertices top-down from the cut vertices (over budget, the
// root search takes over).
// DETACH_LEVELS: its level limit (measured on R-MAT, where it pays, the
// search takes 2-7 levels; on deep trees each level costs about as much as
// a whole pointer-jumping round)
#define DETACH_LEVELS 16
struct DetachArgs {
    const int *cuts, *par, *rold;
    int *rep;
    Csr g;
    const u64 *ovf;
    u64 ovf_cap;
    int *A, *J1;                    // detached vertices; their new representatives until the search ends
    unsigned *det_ep, *det_claim;
    long long budget_v, budget_e;
    int max_levels;
    unsigned nsm;
    int *oc, *op;                   // tree edges held outside the rows
};
struct RelabelArgs {
    int n;
    int *rep;
    const int *par;
    const unsigned *aff_ep;   // old roots of the cut trees
    int *J;                   // ancestor, or ~root
    int *X, *Y, *L;           // per-warp lists: open vertices (ping-pong), detached vertices
    int *D;                   // all detached vertices
    const int *rold;          // per cut vertex: the old root of its tree
    unsigned *w;              // vertices per detached piece; per old root: of its tree
    unsigned *wsum;           // per old root: vertices of the detached pieces
    u64 *heavy;               // per old root: the heaviest large detached piece
    int *left;                // per piece: the one that the scan leaves out in its tree
    const int *cuts;
};
// entries of each list array: blocks take chunks of BLK * 4 vertices in turn,
// every block has room for as many as the first one
static inline long long relabel_room(long long n, unsigned blocks) {
    const long long ch = BLK * 4, nch = (n + ch - 1) / ch, per = (nch + blocks - 1) / blocks;
    return (nch < (long long)blocks ? nch : (long long)blocks) * per * ch;
}
cudaError_t launch_relabel(const Dev &d, Ctl *ctl, RelabelArgs a, cudaStream_t s);
cudaError_t launch_cross(const Dev &d, Ctl *ctl, DetachArgs da, RelabelArgs ra, RowList rl, LightArgs la, bool sg,
                         cudaStream_t s);
unsigned coop_blocks_cross(int nsm);
unsigned coop_blocks_relabel(int nsm);
cudaError_t launch_jump(const Dev &d, const int *A, int use_list, long long cnt_static, Ctl *ctl, const int *par,
                        int *J, int *J1, int *rep, RowList rl, int mode, const int *rold, unsigned *w, u64 *heavy,
                        Csr g, int sync_rounds, int *X, int *Y, const int *cuts, cudaStream_t s);
struct HookArgs {
    u64 *ck[2];          // candidates: key and the two pieces (ping-pong)
    int *ca[2], *cb[2];
    u64 cand_cap;
    HookSlots hs;
    u64 *er;             // replacement edges
    long long er_cap;
    int init;            // set up the candidates' endpoints first (0: their writer did, HookSlots)
    int pairs;           // move the pair table into the candidate list first
    PairTable pt;
};
struct OrientArgs {
    const u64 *er;
    int rank_arcs;       // core arcs that one block ranks in shared memory
    u64 *er_out;         // (the same array: replace_small's edges for the grid)
    const int *rep;
    int *comp, *minp, *pidx, *plist;
    unsigned *pstamp;
    int *pdeg, *pcur, *poff, *adj, *apos;
    int *val0, *val1, *nx0, *nx1;
    long long *bsum;
    int *chx, *chy;
    unsigned *att_ep, *rep_ep;
    int *att_x, *newrep;
    unsigned char *lf;   // per replacement edge: 0 core, 1 lo-side piece is a leaf, 2 hi-side
    int *cdeg;           // core degree per dense piece
    int *ep, *eid;       // per arc: source piece, its dense id
    int *eroot;          // per edge: hook-forest root of its super-tree
    int *cel;            // core edges (for the one-block path of small cores)
    int *parent;         // the forest: paths are reversed in place
    unsigned *long_ep;   // pieces whose path is too long to walk
    int walk;            // walk each path as its edge is oriented (0: k_walk does, or the Euler tour's marks)
    const unsigned *aff_ep;   // old roots of this batch's cut trees
    long long n;
};
cudaError_t launch_replace(const Dev &d, Ctl *ctl, HookArgs h, OrientArgs a, bool large, cudaStream_t s);
// batches above this many edges walk their paths in a launch of its own
#define LARGE_BATCH (1 << 18)
cudaError_t launch_walk(const Dev &d, Ctl *ctl, OrientArgs a, cudaStream_t s);
struct FinishArgs {
    const int *A;             // delete: the affected list
    long long n;
    int *rep, *parent;
    const unsigned *sel_ep;   // pieces reversed through the marks
    const int *att_x;
    const unsigned *rep_ep;
    const int *newrep;
    int *act, *pold, *J0, *J1, *aidx, *aroot;
    unsigned char *mark;
    const int *chx, *chy;
    int euler;
};
cudaError_t launch_finish(const Dev &d, Ctl *ctl, FinishArgs a, cudaStream_t s);
cudaError_t launch_reverse(const Dev &d, Ctl *ctl, FinishArgs a, cudaStream_t s);
cudaError_t launch_labels(int n, const int *rep, int *tmp, int *out, cudaStream_t s);

unsigned coop_blocks_jump(int nsm);
unsigned grid_vertex_pass(int nsm);
unsigned coop_blocks_finish(int nsm);
unsigned coop_blocks_replace(int nsm);
cudaError_t launch_barrier_selftest(Ctl *ctl, cudaStream_t s);
// static.cu ------------------------------------------------------------
cudaError_t launch_static_forest(const Dev &d, int n, Csr g, const u64 *ovf, Ctl *ctl, int *lab, int *comp,
                                 int *parent, int *f0, int *f1, u64 *levels, long long gen, cudaStream_t s);
unsigned coop_blocks_bfs(int nsm);
// euler.cu -------------------------------------------------------------
struct EtArgs {
    const int *act, *pold, *aidx, *aroot, *att_x;
    int *ccnt, *ccur, *coff, *kids, *kpos;
    int *val0, *val1, *nx0, *nx1;
    long long *bsum;
    unsigned char *mark;
};
cudaError_t launch_et_marks(const Dev &d, Ctl *ctl, EtArgs a, cudaStream_t s);
unsigned coop_blocks_et(int nsm);
// batched.cu -----------------------------------------------------------
// Persistent per-graph kernels over the disjoint union of many graphs.
#define BCLASSES 4
struct BDesc {               // per call
    const int *batch;        // union batch (ids offset per graph)
    long long len;
    const long long *voff;   // G + 1 vertex offsets
    const long long *boff;   // G + 1 batch offsets
    const int *order;        // graphs in queue order, class by class
    int G;
    int op;
    StorageLimits lim;
};
struct BState {              // device pointers of one handle (per call)
    Ctl *ctl;
    int *parent, *rep;
    Csr g;
    Index ix;
    Ovf ovf;
    u64 *nkey, *nslot;       // batch-indexed
    // vertex-indexed scratch (graph g uses its own vertex range)
    int *J, *R, *A, *Dv, *roff, *comp, *minp, *pidx, *plist, *pdeg, *poff, *pcur, *newroot, *flist, *chx, *chy;
    int *adj;                // 2 per vertex
    int *tile;               // row of the first entry of each 32-entry tile of a graph's scanned rows
    unsigned *st_aff, *st_cut, *st_piece, *st_vis, *st_rr;   // epoch stamps
    u64 *best, *er;
    // candidate pool, handed out in chunks
    u64 *pk;
    int *pa, *pb;
    u64 pool_cap;
    u64 *pool_ctr;
    u64 *pt_pk, *pt_mk;      // pair table (shared with the grid path; empty between calls)
    u64 pt_mask;
    unsigned *qctr;          // queue counter per class
    int *gcnt, *gcur;        // overflow edges per graph
    long long *govf_start;
    u64 *govf;               // positions in ovf, grouped by graph
    BDesc *desc;
};
cudaError_t launch_bset(BState *dst_state, const BState &st, BDesc *dst_desc, const BDesc &d, cudaStream_t s);
cudaError_t launch_bprologue(const Dev &dv, const BState *S, cudaStream_t s);
unsigned bpersist_grid(int nsm, int threads, int per_sm, int cluster);
cudaError_t launch_bpersist(const BState *S, int cls, int q_lo, int q_hi, int threads, unsigned grid, int cluster,
                            cudaStream_t s);

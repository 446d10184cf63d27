// Internal interface between the kernel translation units and the engine.
// Every function enqueues work on the given stream and returns at once.
#pragma once
#include "common.cuh"

namespace upr {

// The graph as the kernels see it (device pointers; adjw / vwgt may be null =
// unit weights).  wI[v] = omega(I(v)) < 2^31.
//
// Sparse form of the gain table for large k: row v holds the blocks adjacent
// to v in off[v+1] - off[v] slots (a power of two, at least min(k, 2 deg(v))
// + 1), each (local block or kEmpty, weight), open addressing with linear
// probing from a hashed home slot.  Keys are only ever inserted (a weight may
// drop to 0 and its key stays), so concurrent inserts of one block meet at
// the same first free slot; the table is rebuilt at every round start.  A row
// without a free slot for a new block sets *overflow, and the round is run
// again with the dense table.
constexpr int32_t kEmpty = -1;
constexpr int kSparseRowMax = 512;   // slots of the largest sparse row (k <= 256: 2k rounded up)
struct SparseRows {
    const int64_t *off;   // [n+1] first slot of each row
    int2 *slot;           // (local block or kEmpty, weight); null: the table is dense
    int32_t *overflow;
    __host__ __device__ bool on() const { return slot != nullptr; }
};

// A context holds one graph or a batch of ng independent graphs packed as one
// CSR (graph g owns the nodes [noff[g], noff[g+1]) and no edge joins two
// graphs).  Blocks are numbered globally: graph g owns blocks [g*k, g*k + k),
// part[] holds global block ids, and everything indexed by block has K = ng*k
// entries.  Gain-table rows keep k columns: the column of global block p is
// p mod k (blk_local).  With one graph, global and local ids coincide.
struct GraphDev {
    int64_t n, m;
    int32_t k;            // blocks per graph
    int32_t ng;           // graphs in the context
    int32_t kmask;        // blk_local(p) = p & kmask when non-zero (-1 for one graph, k-1 for k a power of two)
    const int64_t *xadj;
    const int32_t *adj;
    const int32_t *adjw;
    const int32_t *vwgt;
    const int32_t *wI;
    const int64_t *Lb;    // [K] L_max of the graph each block belongs to
    const int32_t *gid;   // [n] graph of each node (null for one graph)
    SparseRows sp;        // sparse gain table when sp.on(), else the dense W[n][k]
    __host__ __device__ int32_t K() const { return ng * k; }
};

__device__ __forceinline__ uint32_t sp_home(int32_t b, uint32_t cap) {
    return (((uint32_t)b * 0x9E3779B1u) >> 8) & (cap - 1);
}
// omega(v, block column b)
__device__ __forceinline__ int32_t sp_get(const SparseRows &t, int64_t v, int32_t b) {
    const int64_t o = t.off[v];
    const uint32_t cap = (uint32_t)(t.off[v + 1] - o);
    uint32_t h = sp_home(b, cap);
    for (uint32_t i = 0; i < cap; i++) {
        const int2 e = t.slot[o + h];
        if (e.x == b) return e.y;
        if (e.x == kEmpty) return 0;
        h = (h + 1) & (cap - 1);
    }
    return 0;
}
// omega(v, b) += w, inserting b at the first free slot of its probe sequence
__device__ __forceinline__ void sp_add(const SparseRows &t, int64_t v, int32_t b, int32_t w) {
    const int64_t o = t.off[v];
    const uint32_t cap = (uint32_t)(t.off[v + 1] - o);
    uint32_t h = sp_home(b, cap);
    for (uint32_t i = 0; i < cap; i++) {
        int *key = &t.slot[o + h].x;
        int kk = *(volatile int *)key;
        if (kk == kEmpty) {
            kk = atomicCAS(key, kEmpty, b);
            if (kk == kEmpty) kk = b;
        }
        if (kk == b) {
            atomicAdd(&t.slot[o + h].y, w);
            return;
        }
        h = (h + 1) & (cap - 1);
    }
    atomicOr(t.overflow, 1);
}
// omega(v, b) -= w for a block b that is in the row
__device__ __forceinline__ void sp_sub(const SparseRows &t, int64_t v, int32_t b, int32_t w) {
    const int64_t o = t.off[v];
    const uint32_t cap = (uint32_t)(t.off[v + 1] - o);
    uint32_t h = sp_home(b, cap);
    for (uint32_t i = 0; i < cap; i++) {
        const int kk = *(volatile int *)&t.slot[o + h].x;
        if (kk == b) {
            atomicSub(&t.slot[o + h].y, w);
            return;
        }
        if (kk == kEmpty) break;
        h = (h + 1) & (cap - 1);
    }
    atomicOr(t.overflow, 2);      // cannot happen: the block of a neighbour is always in the row
}

__device__ __forceinline__ int32_t blk_local(int32_t p, int32_t k, int32_t kmask) {
    return kmask ? (p & kmask) : p % k;
}
__device__ __forceinline__ int32_t blk_local(const GraphDev &g, int32_t p) { return blk_local(p, g.k, g.kmask); }
// first global block of p's graph
__device__ __forceinline__ int32_t blk_base(const GraphDev &g, int32_t p) { return p - blk_local(g, p); }
__device__ __forceinline__ int32_t blk_graph(const GraphDev &g, int32_t p) { return g.ng == 1 ? 0 : p / g.k; }

__device__ __forceinline__ int64_t node_c(const GraphDev &g, int64_t v) { return g.vwgt ? (int64_t)g.vwgt[v] : 1; }
__device__ __forceinline__ int32_t edge_w(const GraphDev &g, int64_t e) { return g.adjw ? g.adjw[e] : 1; }

// What a team launch needs (team.cuh): the grid barrier's arrival counter, the
// error word (set when a bounded wait gives up), per-CTA digit totals
// [size][256], block-weight totals [2][size][256] and scan totals, and the
// number of CTAs (one per binding, since the counter counts by it).
struct Team {
    unsigned long long *bar = nullptr;
    int32_t *err = nullptr;
    int32_t *hist = nullptr;
    unsigned long long *hist64 = nullptr;
    long long *tot = nullptr;
    int size = 1;
};

// team.cu: one grid barrier of the team, which its last `absent` CTAs never
// reach; *passed = the CTAs that went past it.  False: the team has no grid barrier.
bool barrier_probe(const Team &t, int absent, int32_t *passed, cudaStream_t s);

// Grid-stride loop over a device-held count (all threads of the grid).
#define UPR_FOR(i, cnt) \
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (cnt); i += (int64_t)gridDim.x * blockDim.x)

// A grid of 256-thread blocks for up to `max` items, at most 8 blocks per SM.
inline unsigned grid_for(int64_t max) {
    const int64_t b = ceil_div(max > 0 ? max : 1, 256);
    return (unsigned)std::min<int64_t>(b, (int64_t)device_sm_count() * 8);
}

// ---- graph.cu: step (e), step (a), create-time work
struct HubChunk { int32_t v; int32_t pad; int64_t begin, end; };
// C[0..K) = block weights of part.
void block_weights(const GraphDev &g, const int32_t *part, int64_t *C, cudaStream_t s);
// cut[0..ng) = edge cut of each graph.  bad (given: neighbour ids unchecked so
// far): set non-zero when one lies outside [0, n); none is read through.
void edge_cut(const GraphDev &g, const int32_t *part, int64_t *cut, cudaStream_t s, int64_t *bad = nullptr);
void incident_weights(const GraphDev &g, int32_t *wI, int64_t *wmax, cudaStream_t s);
// *cut = the cut of part (one graph) from the gain table W = W(part) (dense or hashed rows) and omega(I(v)).
void cut_from_table(const GraphDev &g, const int32_t *part, const int32_t *W, int64_t *cut, cudaStream_t s);
// A tile of the table build: nodes [v0, v1) and the adjacency entries [e0, e1)
// of its non-hub nodes (a hub, if any, is the tile's last node).  With hashed
// rows its non-hub rows have at most kTileSlots slots.
constexpr int kTileSlots = 4096;
constexpr int kSparseTileNodes = 128;         // rows of a tile with hashed rows
struct TableTile { int64_t e0, e1; int32_t v0, v1; };
// Static schedules from the packed offsets (bind.cu), over segments of
// kSchedSegment nodes.  sched_count: cnt[4 s + 0..3] = exclusive offsets of
// segment s's hub chunks, tiles, hashed-row slots and hubs; tot[0..3] = the
// totals.  sp_mode 0:
// no hashed rows, 1: min(k, 2 deg) + 1 slots rounded up to a power of two,
// 3: min(k, deg) + 1.  sched_write fills the arrays (sp_off with hashed rows).
constexpr int64_t kSchedSegment = 1024;
int64_t sched_segments(int64_t n);
void sched_count(const int64_t *xadj, int64_t n, int64_t m, int tile_nodes, int sp_mode, int32_t k, int64_t *cnt,
                 int64_t *tot, cudaStream_t s);
void sched_write(const int64_t *xadj, int64_t n, int64_t m, int tile_nodes, int sp_mode, int32_t k,
                 const int64_t *off, HubChunk *chunks, TableTile *tiles, int64_t *sp_off, int32_t *hubs,
                 cudaStream_t s);
// *bad = 1 unless xadj[0] = 0, xadj[n] = m and xadj is non-decreasing
void xadj_check(const int64_t *xadj, int64_t n, int64_t m, int32_t *bad, cudaStream_t s);
// A batch's packed offsets from each graph's own (graph i's n_i + 1 offsets at
// raw + noff[i] + i), shifted by the entries before it (eoff), checked as
// xadj_check checks one graph
// One segment of a gather of host arrays: len elements from src (page-locked
// host memory, read by the GPU directly) to the destination + off.
struct HostSeg {
    const void *src;
    int64_t off, len;
};
constexpr int64_t kGatherChunk = 1 << 16;
// d_segs (device memory): the segments; elem: 4 or 8 bytes per element
void gather_host(const HostSeg *d_segs, int64_t nseg, size_t elem, void *dst, cudaStream_t s);
void xadj_pack(const int64_t *raw, const int64_t *noff, const int64_t *eoff, int32_t ng, int64_t n, int64_t *out,
               int32_t *bad, cudaStream_t s);
// W must hold n*k ints.  Rows of hubs (degree > kHubDegree) are completed by the chunk pass.
// By the binding's tiles (every binding with nodes has them).
// With deg_sum: runs only when 4 * (*deg_sum) >= m (the rebuild alternative to table_move).
void gain_table(const GraphDev &g, const int32_t *part, int32_t *W, const HubChunk *hub_chunks, int64_t n_chunks,
                const TableTile *tiles, int64_t n_tiles, int32_t tile_nodes, const int64_t *deg_sum, cudaStream_t s);
// How moved hubs are found for the chunked delta update: through m_pos (moves
// of M: from/to are M_from/M_to) or, when m_pos is null, through r_to/r_at
// (moves of the current rebalancing sub-round: R indices in [*r_base,
// *r_base + *r_count), from/to are R_from/R_to).
struct HubMoves {
    const int32_t *m_pos;
    const int32_t *r_to, *r_at, *r_base, *r_count;
    const int32_t *from, *to;
};
// For each listed node v moving from[i] -> to[i] (i < *d_count, entries start at
// *d_offset when given): W[u][from] -= w, W[u][to] += w for every neighbour u.
// With deg_sum: runs only when 4 * (*deg_sum) < m (otherwise a rebuild is cheaper).
// Hubs are handled chunk by chunk through hub_chunks and hm.
void table_move(const GraphDev &g, int32_t *W, const int32_t *nodes, const int32_t *from, const int32_t *to,
                const int32_t *d_count, const int32_t *d_offset, const int64_t *deg_sum, int64_t max_count,
                const HubChunk *hub_chunks, int64_t n_chunks, HubMoves hm, cudaStream_t s);
// Batches: gid[v] = graph of node v (noff: [ng + 1] first nodes), and each
// graph's neighbour ids (local to the graph on input) shifted by its first
// node; an id that leaves [0, n) becomes -1 for the checks to report.
void pack_batch(const GraphDev &g, const int64_t *noff, int32_t *gid, int32_t *adj, cudaStream_t s);
// W[v][b] = omega(v, V_b) from the sparse table (inspection only).
void sparse_to_dense(const GraphDev &g, int32_t *W, cudaStream_t s);
// Graph checks; writes a bitmask of violations into *d_flags (see engine.cu).
// Checks the CSR on the device (bits of *d_flags, hash sums in d_acc[0..1]):
// ranges, self loops, weights, symmetry by a multiset hash, and bit 128 for a
// row whose ids are not strictly increasing.
void validate_graph(const GraphDev &g, uint64_t *d_acc, int32_t *d_flags, cudaStream_t s);
// Exact duplicate check (bit 32 of *d_flags) for graphs with an unsorted row:
// hubs lists the n_hubs nodes of degree > kHubDegree, noff the batch's node
// offsets (ignored for one graph), max_graph_nodes the largest graph's node
// count, scratch: scratch_ints free ints.
void validate_duplicates(const GraphDev &g, int32_t *d_flags, const int32_t *hubs, int64_t n_hubs,
                         const int64_t *noff, int64_t max_graph_nodes, int32_t *scratch, int64_t scratch_ints,
                         cudaStream_t s);

// ---- select.cu: step (b) and applying M
struct Penalty {
    const int64_t *PW;    // [K][73] inclusive prefix over slots of available node weight
    const int64_t *F;     // [73] floor(tau_r * (3/2)^l * 2^Q)
    const int64_t *C;     // [K] round-start block weights
    const int64_t *Lb;    // [K] L_max of each block's graph
    const int8_t *first;  // [K] smallest slot l with PW[b][l] >= 1, -1 if none (the excess-1 case)
    // > 0 (unit node weights, one graph, gb + pack_bits <= 30): the dense
    // selection kernel scores a column as one integer, ((gain - penalty) <<
    // pack_bits) + (2^pack_bits - 1 - b), pack_bits = the bits of a column index
    int pack_bits = 0;
    int gbits = 0;
};
// A list of nodes (device memory; own: given when they are boundary nodes, all
// nodes' omega(v, V_P(v)) by node) and the selection's results by list index:
// best target (-1: no candidate), score, gain.
struct NodeList { const int32_t *node, *d_n, *own = nullptr; };
struct Candidates { int32_t *tgt, *s0, *gain; };
// Buckets and their prefixes, part = part0 and C = C0, the boundary nodes in
// node order, and with cut_pending the cut of part0 per graph (cut and cut_in).
struct NodePass {
    Team team;
    const int32_t *part0;
    const int64_t *C0;
    int32_t *part;
    int64_t *C;
    int32_t t_num, t_den;
    unsigned long long *BW;
    int64_t *PW;
    int8_t *first;
    int8_t *avail_out;                        // nullable
    int32_t *slot_out;                        // nullable
    int32_t *own;                             // [n] omega(v, V_P(v))
    int32_t *list, *d_list;
    int cut_pending;
    int64_t *cut, *cut_in;                    // [ng]
    // set by node_pass
    int64_t n = 0;
    int32_t k = 0, kmask = 0, K = 0, ng = 0;
    int use_shared = 0;
    const int32_t *W = nullptr, *wI = nullptr, *vwgt = nullptr, *gid = nullptr;
    SparseRows sp{};
};
// room: the dynamic shared memory the kernel that runs the pass can have; a
// histogram beyond it stays in global memory.  (A kernel's static part counts
// against the same 227 KB of a CTA: 38 KB in k_node_pass, 45 KB in the small
// graphs' kernel.)
constexpr size_t kNodePassSmem = 184 * 1024;
size_t node_pass_args(const GraphDev &g, NodePass &a, const int32_t *W, size_t room);
void node_pass(const GraphDev &g, NodePass a, const int32_t *W, cudaStream_t s);
// Lanes per node (G) and 16-byte chunks per lane (CH) of the vectorised
// selection and proposal kernels (k % 4 == 0, k <= 256, 4*G*CH >= k).  A
// schedule only decides how the work is spread over lanes, never the
// result.  G = 0: the default (the fewest chunks per lane).
struct LaneCfg { int32_t G, CH; };
// The schedules worth timing for k (the default first); returns their number (0..3).
int lane_candidates(int32_t k, LaneCfg *out);
void select_moves(const GraphDev &g, NodeList nl, const int32_t *part, const int32_t *W, Penalty pen, Candidates out,
                  LaneCfg cfg, cudaStream_t s);
// Step (b3): the candidates' inflow penalties, M in its order and applied
// (team.cuh).  bufA / bufB: 16 n bytes each.
struct SelOrder {
    Team team;
    NodeList nl;
    Candidates cand;
    Penalty pen;
    const int32_t *part0;
    int32_t *part;                            // [n] part0; becomes part0 with M applied
    int64_t *C;                               // [K] likewise
    int32_t *score;                           // [n] kept score by list index, else 0
    int64_t *c_excl, *seg_base;               // [n], [K] scratch
    void *bufA, *bufB;
    int32_t *M_node, *M_from, *M_to;
    int64_t *M_score;
    int32_t *m_pos;
    int64_t *deg_sum;                         // degree sum of M
    int32_t *d_cand, *d_moves;                // candidates, |M|
    // set by select_order
    int K = 0, kbits = 0;
    const int32_t *vwgt = nullptr;
    const int64_t *xadj = nullptr;
};
// (the *_args functions fill the fields a wrapper sets; they return the dynamic
// shared memory of the launch)
void select_order_args(const GraphDev &g, SelOrder &a);
void select_order(const GraphDev &g, SelOrder a, int gbits, cudaStream_t s);

// ---- rebalance.cu: step (d)
// Device-resident control block of the rebalancing loop.
struct RebalCtl {
    int32_t active;      // the current sub-round runs
    int32_t stopped;     // the loop has finished
    int32_t light;       // one graph: lightest block that may receive moves, or -1
    int32_t subrounds;   // sub-rounds that ran
    int32_t nR;          // rebalancing moves so far (length of R)
    int32_t n1_active;   // length of the node list if this sub-round runs, else 0
    int32_t flag;        // batch controllers: "some block is overloaded" / "the excluded set grew"
    uint32_t ticket;     // batch controllers: CTAs finished (the last one updates the control block)
};
struct RebalState {
    const int64_t *C;     // [K] current block weights
    const int8_t *over;   // [K] overloaded now
    const int8_t *excl;   // [K] not a target: overloaded at the first sub-round, or rejected a move
    const int32_t *light; // [ng] lightest non-excluded block of each graph, or -1
    const int64_t *Lb;    // [K] L_max of each block's graph
    // per listed node i with a proposal, its block and gain by list index, so
    // that later passes over the list read them in order
    int32_t *lsrc = nullptr, *lgain = nullptr;
    // > 0 (unit node weights, one graph, 1 + gb + pack_bits <= 32): the dense
    // proposal kernel scores a column as one integer, (omega << pack_bits) +
    // (2^pack_bits - 1 - b), pack_bits = the bits of a column index
    int pack_bits = 0;
};
// Proposals of the listed nodes in overloaded blocks: prop_tgt/prop_gain by node, flags by list position.
void rebalance_propose_scalar_list(const GraphDev &g, const int32_t *list, const int32_t *d_n1, int64_t n1_max,
                                   const int32_t *part, const int32_t *W, RebalState st, int32_t *prop_tgt,
                                   int32_t *prop_gain, int32_t *flags, cudaStream_t s);
void rebalance_propose_list(const GraphDev &g, const int32_t *list, const int32_t *d_n1, int64_t n1_max,
                            const int32_t *part, const int32_t *W, RebalState st, int32_t *prop_tgt,
                            int32_t *prop_gain, int32_t *flags, LaneCfg cfg, cudaStream_t s);
constexpr int kPrioBins = 256;
// The first list: the nodes of the overloaded blocks, in node order.  One
// graph: also the excluded set, the control block and the first sub-round's
// begin (cond: the condition of a graph-resident loop).
struct RebalStart {
    Team team;
    const int32_t *part;
    const int64_t *C;
    int32_t *list, *d_list;
    int8_t *excl, *over, *reject;
    int32_t max_subrounds;
    RebalCtl *ctl;
    cudaGraphConditionalHandle cond;
    // set by rebalance_start
    int64_t n = 0;
    int K = 0, batch = 0;
    const int64_t *Lb = nullptr;
};
void rebalance_start_args(const GraphDev &g, RebalStart &a);
void rebalance_start(const GraphDev &g, RebalStart a, cudaStream_t s);
// A sub-round after its proposals: the proposers (flags by list index, their
// blocks and gains in lsrc / lgain) become the list, the minimal prefix per
// source and the longest fitting prefix per target in priority order are
// appended to R at ctl->nR (*d_na of them) and applied to part and C.
// Proposal prefilter (exact; hist null: none): a source's proposals in the
// priority bins after the one where its cumulative weight reaches the excess
// can never be in its minimal prefix.  hist (K * kPrioBins, zero) is left zero.
// bufA, bufB: 32 n bytes each.
struct RebalTeam {
    Team team;
    const int32_t *flags;
    int32_t *list;
    const int32_t *lsrc, *lgain, *d_n1;
    int32_t *list2, *lsrc2, *lgain2;         // [n] scratch
    int gbits, cbits, gain_only;             // gain_only: the priority is the gain alone (Sec. 7.2), else Sec. 6.1's
    unsigned long long *hist, *rep;          // prefilter weights; [kPrioBins] a key per bin
    int32_t *cut, *exact;                    // [K] cut bin per source; every bin holds one key value
    const int8_t *over;
    int64_t *C;
    void *bufA, *bufB;
    uint32_t *U;                             // [n] the kept proposals in priority order
    int32_t *at;                             // [n] their targets while selected, then while admitted
    int64_t *c_excl, *seg_base;              // [n], [K] scratch (K > 256)
    int32_t *part;
    const int32_t *prop_tgt;
    int8_t *reject;
    const RebalCtl *ctl;
    int32_t *R_node, *R_from, *R_to, *R_sub, *r_to, *r_at;
    int32_t *d_np, *d_nk, *d_na;             // proposers, kept, admitted
    // set by rebalance_order
    int K = 0, kbits = 0;
    const int32_t *vwgt = nullptr;
    const int64_t *Lb = nullptr;
};
constexpr int kRebRankK = 256;       // blocks up to which a sub-round ranks by per-warp block sums
size_t rebalance_order_args(const GraphDev &g, RebalTeam &a);
void rebalance_order(const GraphDev &g, RebalTeam a, cudaStream_t s);
// Loop control of a batch: the excluded set and the control block; a
// sub-round's begin (light: each graph's lightest non-excluded block).
void rebalance_init_batch(const GraphDev &g, const int64_t *C, int8_t *excl, RebalCtl *ctl, cudaStream_t s);
void rebalance_begin_batch(const GraphDev &g, const int64_t *C, const int8_t *excl, int8_t *over, int8_t *reject,
                           const int32_t *d_n1, int32_t max_subrounds, RebalCtl *ctl, int32_t *light, cudaStream_t s);
// Sets the condition of a graph's while node: another sub-round is due.
void rebalance_continue(const RebalCtl *ctl, int32_t max_subrounds, cudaGraphConditionalHandle handle,
                        cudaStream_t s);
// A sub-round's end; one graph: the next one begins in the same kernel (over,
// d_n1, and cond as rebalance_start's).
void rebalance_end(const GraphDev &g, const int64_t *C, int8_t *excl, int8_t *reject, int8_t *over,
                   const int32_t *d_na, const int32_t *d_n1, int32_t max_subrounds, RebalCtl *ctl, cudaStream_t s,
                   cudaGraphConditionalHandle cond = 0);

// ---- mixed.cu: one context over batches of different k (one batch per k)
struct MixedBatch;
upr_status mixed_create(const upr_graph *graphs, int32_t n_graphs, const int32_t *k, const double *eps,
                        const upr_params *params, MixedBatch **out);
upr_status mixed_rebind(MixedBatch *mb, const upr_graph *graphs, int32_t n_graphs, const int32_t *k,
                        const double *eps);
void mixed_destroy(MixedBatch *mb);
// engine.cu: a context bound to other graphs (its arena reused when large enough)
upr_status ctx_rebind(upr_ctx *c, const upr_graph *g, int32_t k, double eps, const upr_params *params);
// (beside: how many contexts, this one included, refine at the same time)
upr_status ctx_rebind_batch(upr_ctx *c, const upr_graph *gs, int32_t ng, int32_t k, const double *eps,
                            const upr_params *params, int beside = 1);
upr_status ctx_create_batch(const upr_graph *graphs, int32_t n_graphs, int32_t k, const double *eps,
                            const upr_params *params, int beside, upr_ctx **out);
int64_t mixed_nodes(const MixedBatch *mb);
upr_status mixed_refine(MixedBatch *mb, int32_t *part, int32_t rounds, uint64_t seed, upr_status *status,
                        int64_t *cut_in, int64_t *cut_out, upr_stats *stats);
upr_status mixed_cut(MixedBatch *mb, const int32_t *part, int64_t *cut, int64_t *block_weights);
upr_status mixed_info(const MixedBatch *mb, int32_t *n_graphs, int64_t *node_offsets, int64_t *lmax);

// ---- sequence.cu: step (c); every count lives in device memory, `max` bounds it
void fill_i32(int32_t *a, int64_t n, int32_t v, cudaStream_t s);
void reset_nodes(const int32_t *nodes, const int32_t *d_cnt, int64_t max, int32_t *arr, int32_t val, cudaStream_t s);
// out[g] = number of blocks of graph g above L_max
void count_over(const GraphDev &g, const int64_t *C, int32_t *out, cudaStream_t s);
// X = the interleaving of M and R (append: M, then R), merged into I (d_nI
// moves; a batch's also sorted by graph into O_*, graph g's moves in
// [seg_beg[g], seg_end[g])), and every node's packed state for seq_gains.
// bufA, bufB: 24 n bytes each; ex: 24 n bytes; qmax: 12 n bytes.
struct SeqBuild {
    Team team;
    const int32_t *M_node, *M_from, *M_to, *dM;
    const int32_t *R_node, *R_from, *R_to, *dR;
    const int32_t *part0, *m_pos, *r_to;
    const int64_t *C0;
    int32_t append;
    void *bufA, *bufB;
    int64_t *ex;                                             // prefix sums over the sorted entries and events
    uint32_t *qmax;                                          // emitted part of R_b after each event
    int32_t *rbeg, *rend, *ebeg, *eend, *qfin, *left_excl;   // [K]
    int32_t *emit, *pos_m;                                   // [n]
    int32_t *X_node, *X_from, *X_to, *fin;                   // [2n]
    int32_t *I_node, *I_from, *I_to;
    int2 *pk;
    int32_t *diff;                                           // cleared up to d_nI
    int64_t *deg_sum;                                        // degrees of I's nodes, added
    int32_t *dX, *dI;
    int32_t *O_node, *O_from, *O_to, *seg_beg, *seg_end;     // batches
    // set by seq_build
    int64_t n = 0;
    int32_t k = 0, kmask = 0, K = 0, ng = 0;
    int kbits = 0, ngbits = 0;
    const int32_t *vwgt = nullptr, *gid = nullptr;
    const int64_t *xadj = nullptr, *Lb = nullptr;
};
void seq_build_args(const GraphDev &g, SeqBuild &a);
void seq_build(const GraphDev &g, SeqBuild a, cudaStream_t s);
void seq_gains(const GraphDev &g, const int32_t *I_node, const int32_t *I_from, const int32_t *I_to,
               const int32_t *d_nI, int64_t max, const int2 *pk, int64_t *gain, const HubChunk *hub_chunks,
               int64_t n_chunks, cudaStream_t s);
// Prefix gains Gsum and the overloaded blocks after every prefix (diff,
// diff_excl); one graph: the best balanced prefix (best = gain, length; -1:
// none, *d_infeasible set) applied to part0, C0 and *cut, and *undone = the
// degree sum of the moves after it.  reset: m_pos and r_to of M and R go back to -1.
struct SeqBest {
    Team team;
    const int32_t *I_node, *I_from, *I_to, *dI;
    const int64_t *gain;
    int64_t *Gsum;
    void *bufA, *bufB;
    int32_t *diff, *diff_excl;
    int32_t *part0;
    int64_t *C0, *cut;
    long long *best;
    int64_t *undone;
    int32_t *d_over0, *d_infeasible;
    int reset;
    const int32_t *M_node, *dM, *R_node, *dR;
    int32_t *m_pos, *r_to;
    // set by seq_best
    int32_t K = 0;
    int kbits = 0;
    const int32_t *vwgt = nullptr, *gid = nullptr;
    const int64_t *xadj = nullptr, *Lb = nullptr;
};
void seq_best_args(const GraphDev &g, SeqBest &a);
void seq_best(const GraphDev &g, SeqBest a, cudaStream_t s);
// The moves of I undone after the best prefix: positions i >= j* (one graph,
// best[1] = j*, -1 = none kept) or i - seg_beg[g] >= best_j[g] (a batch, gid set).
struct Rollback {
    const int32_t *I_node, *I_from, *I_to;
    const int32_t *d_nI;
    const long long *best;
    const int32_t *gid, *seg_beg;
    const long long *best_j;
};
// The oscillation guard of Sec. 2: locked[v] = 1 exactly for the nodes of the
// applied prefix of I whose move came from rebalancing alone (m_pos < 0,
// r_to >= 0); and no candidate among the locked nodes.
void guard_locks(const struct Rollback &rb, int64_t max, int64_t n, const int32_t *m_pos, const int32_t *r_to,
                 int8_t *locked, cudaStream_t s);
void guard_filter(const int8_t *locked, int64_t n_max, NodeList nl, Candidates cand, cudaStream_t s);
// W(P o I) -> W(P o I^{j*}): delta updates of the undone moves (pk: positions
// in I), or nothing when 4 * (their degree sum *deg_sum; a batch's is summed
// here, onto the 0 that seq_best left) >= m, in which case the caller rebuilds
// with gain_table(..., deg_sum).
void table_rollback(const GraphDev &g, const Rollback &rb, int64_t max, const int2 *pk, int32_t *W,
                    const HubChunk *hub_chunks, int64_t n_chunks, int64_t *deg_sum, cudaStream_t s);
// Per graph: the best eligible prefix j* (ties: shortest; none: infeasible,
// j* = 0), cut[g] -= G_g(j*); tot = (sum j*, sum G(j*), infeasible graphs).
void seq_best_seg(const GraphDev &g, const int32_t *I_node, const int32_t *d_nI, int64_t max, const int32_t *seg_beg,
                  const int64_t *Gsum, const int32_t *diff, const int32_t *diff_excl, const int32_t *over0,
                  long long *best_g, long long *best_j, int64_t *cut, int32_t *infeasible, int64_t *tot,
                  cudaStream_t s);
void seq_apply_prefix_seg(const GraphDev &g, const int32_t *I_node, const int32_t *I_from, const int32_t *I_to,
                          const int32_t *d_nI, int64_t max, const int32_t *seg_beg, const long long *best_j,
                          int32_t *part0, int64_t *C0, cudaStream_t s);

// ---- small.cu, small_form.cuh: all rounds of a call on a small graph in one launch
// The team is one CTA or one cluster (n <= kSmallNodes), the table dense, keys
// within 63 bits and scores and blocks within 32.
constexpr int64_t kSmallNodes = 65536;
struct SmallRefine {
    Team team;
    GraphDev g;
    int32_t *W;
    int build;                               // the table is built first (else it is valid)
    const HubChunk *chunks;
    int64_t n_chunks;
    int32_t rounds;
    const int64_t *F;                        // [rounds][kSlots] penalty factors
    NodePass np;                             // cut_pending: of the first round
    SelOrder so;
    RebalStart rs;
    RebalTeam rt;
    RebalState st;
    int32_t *prop_gain, *flags;
    SeqBuild sq;
    SeqBest sb;
    RebalCtl *ctl;
    // sums over the rounds: candidates, moves, rebalancing moves, sub-rounds,
    // |I|, applied, -, infeasible rounds; [10..13]: ns in the table build,
    // selection, rebalancing, sequence
    long long *d;
};
bool small_refine_ok(const GraphDev &g, int gbits, int cbits);
void small_refine(const SmallRefine &a, cudaStream_t s);
// (unit node weights; sub-rounds that rank by block sums, K <= kRebRankK)
template <bool UNIT, bool RANK>
void small_form(SmallRefine a, cudaStream_t s);

// ---- lp.cu: unconstrained label propagation (Sec. 5)
// active[v] = 1 for the boundary nodes of part (table W of part)
void lp_boundary(const GraphDev &g, const int32_t *part, const int32_t *W, int8_t *active, cudaStream_t s);
// list[0..*d_cnt) = the active nodes (active given, i < n), or the indices of
// the candidates (tgt given, i < *d_n), ascending
struct LpList {
    Team team;
    const int8_t *active;
    const int32_t *tgt, *d_n;
    int64_t n;
    int32_t *list, *d_cnt;
};
void lp_list(const LpList &a, cudaStream_t s);
// the listed candidates (indices into nl, d_cnt of them, ascending) to their
// targets: part (a copy of part0), C, the move list, m_pos markers and the
// movers' degree sum
void lp_apply(const GraphDev &g, const int32_t *movers, const int32_t *d_cnt, NodeList nl, Candidates cand,
              const int32_t *part0, int32_t *part, int64_t *C, int32_t *M_node,
              int32_t *M_from, int32_t *M_to, int64_t *M_score, int32_t *m_pos, int64_t *deg_sum, int64_t max_count,
              cudaStream_t s);
// next[u] = 1 for the unmoved neighbours u of the nodes whose block changed
// from before to after, every such node being in nodes1[0..*d_cnt1) or
// nodes2[0..*d_cnt2) (the hubs' rows by their chunks); *d_count = their number
void lp_next(const GraphDev &g, const int32_t *before, const int32_t *after, const int32_t *nodes1,
             const int32_t *d_cnt1, const int32_t *nodes2, const int32_t *d_cnt2, const HubChunk *hub_chunks,
             int64_t n_chunks, int8_t *next, int32_t *d_count, cudaStream_t s);
// *d_count = the number of non-zero entries of active
void lp_count(const int8_t *active, int64_t n, int32_t *d_count, cudaStream_t s);

}  // namespace upr
